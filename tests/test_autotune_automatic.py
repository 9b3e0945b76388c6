"""tuned_options on the CPU, with a fake timer: the library's automatic choice is among the candidates (for an m
that is no multiple of four it alone uses the tiles), and a cached choice serves the size and the kernels that it
was timed on only."""
import types

from paper_2008_02205_gb300 import autotune


def _timer(times, calls):
    def time_apply(prob, opt, reps, warmup, stream):
        calls.append(opt["apply_kernel"])
        used = opt["apply_kernel"] or 2
        return times.get(opt["apply_kernel"], 90.0), {"apply_kernel": used, "tile_chunk": prob.m, "tile_max_halo": 100}
    return time_apply


def test_the_automatic_choice_is_timed_and_kept(monkeypatch, tmp_path):
    monkeypatch.setenv("MLPG_TUNE_CACHE", str(tmp_path / "tune.json"))
    calls = []
    monkeypatch.setattr(autotune, "time_apply", _timer({0: 14.0, 1: 39.0}, calls))
    prob = types.SimpleNamespace(m=14, dim=2, n=181 * 181)
    assert autotune.tuned_options(prob) == autotune.AUTOMATIC
    assert calls == [0, 1]
    assert autotune.tuned_options(prob) == autotune.AUTOMATIC and calls == [0, 1]   # from the cache
    near = types.SimpleNamespace(m=14, dim=2, n=170 * 170)
    assert autotune.tuned_options(near) == autotune.AUTOMATIC and calls == [0, 1]
    small = types.SimpleNamespace(m=14, dim=2, n=32 * 32)
    autotune.tuned_options(small)
    assert calls == [0, 1, 0, 1]


def test_a_choice_timed_on_other_kernels_is_tuned_again(monkeypatch, tmp_path):
    monkeypatch.setenv("MLPG_TUNE_CACHE", str(tmp_path / "tune.json"))
    calls = []
    monkeypatch.setattr(autotune, "time_apply", _timer({0: 50.0, 2: 40.0}, calls))
    prob = types.SimpleNamespace(m=12, dim=2, n=4096)
    autotune._store([autotune._size_key(2, 12, 4096), "dim2-m12"],
                    {"choice": {"apply_kernel": 1, "tile_rows": 0, "tile_dpt": 0}, "n": 4096, "table": []})
    assert autotune.tuned_options(prob)["apply_kernel"] == 2 and calls
    calls.clear()
    assert autotune.tuned_options(prob)["apply_kernel"] == 2 and not calls
    monkeypatch.setattr(autotune, "kernel_version", lambda: "other")
    autotune.tuned_options(prob)
    assert calls
