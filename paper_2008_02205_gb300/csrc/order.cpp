// Spatial order of the points (host, once per point set): recursive bisection.  A set is cut across its longest extent into
// two halves whose sizes are multiples of the largest power of two up to 64
// that fits twice, down to pairs, so that every aligned run of 2, 4, .. 64
// points is one compact box whatever the lattice.  A Morton order keeps its
// boxes only where the points per side are a power of two: at 75^2 its pairs of
// rows share 0.81 of their columns (the longest pair 101 columns against 67
// here), a 64-row halo has up to 324 points (231 here); at 64^2 the two orders agree.
// The row tiles use it; the preconditioner keeps its Morton blocks, because which
// points share a block decides where a restarted solve converges at all (with these
// blocks the FP64 solve of a 6^3 lognormal problem stagnated).
#include <algorithm>
#include <exception>
#include <thread>
#include <utility>

#include "internal.h"

namespace mlpg {

namespace {
struct OrderPoint {
    double c[3];
    int32_t id;
};

void bisect(OrderPoint *p, int64_t cnt, int dim, int threads) {
    while (cnt > 2) {
        double lo[3], hi[3];
        for (int a = 0; a < dim; ++a) lo[a] = hi[a] = p[0].c[a];
        for (int64_t k = 1; k < cnt; ++k)
            for (int a = 0; a < dim; ++a) {
                lo[a] = std::min(lo[a], p[k].c[a]);
                hi[a] = std::max(hi[a], p[k].c[a]);
            }
        int ax = 0;
        for (int a = 1; a < dim; ++a)
            if (hi[a] - lo[a] > hi[ax] - lo[ax]) ax = a;
        int64_t unit = 64;
        while (2 * unit > cnt) unit /= 2;
        int64_t half = (cnt + unit) / (2 * unit) * unit;
        if (half >= cnt) half = cnt - unit;
        // ties by point number: the two sets, and so the order, do not depend on the library
        std::nth_element(p, p + half, p + cnt, [ax](const OrderPoint &u, const OrderPoint &v) {
            return u.c[ax] < v.c[ax] || (u.c[ax] == v.c[ax] && u.id < v.id);
        });
        if (threads > 1 && cnt > 4096) {
            std::exception_ptr err;
            std::thread t;
            try {
                t = std::thread([&err, p, half, dim, threads] {
                    try {
                        bisect(p, half, dim, threads / 2);
                    } catch (...) {
                        err = std::current_exception();
                    }
                });
            } catch (...) {   // no thread: both halves here
                bisect(p, half, dim, 1);
            }
            bisect(p + half, cnt - half, dim, threads - threads / 2);
            if (t.joinable()) t.join();
            if (err) std::rethrow_exception(err);
            return;
        }
        bisect(p, half, dim, 1);
        p += half;
        cnt -= half;
    }
    if (cnt == 2 && p[1].id < p[0].id) std::swap(p[0], p[1]);
}
}  // namespace

void spatial_order(int64_t n, int dim, const double *x, int32_t *order) {
    std::vector<OrderPoint> p(n);
    for (int64_t i = 0; i < n; ++i) {
        p[i] = OrderPoint{{0.0, 0.0, 0.0}, (int32_t)i};
        for (int a = 0; a < dim; ++a) p[i].c[a] = x[i * dim + a];
    }
    bisect(p.data(), n, dim, (int)std::max(1u, std::thread::hardware_concurrency()));
    for (int64_t i = 0; i < n; ++i) order[i] = p[i].id;
}

}  // namespace mlpg
