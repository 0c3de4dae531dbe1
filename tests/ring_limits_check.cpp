// Host check of the ring decomposition (csrc/rings.h) at its limits.
//   alloc       every allocation of a build fails in turn (steps of argv[2]): std::bad_alloc each time, raised
//               from outside the parallel regions (from inside, the process would end)
//   far <z>     nodes |z| <= z: prints 1 if the build takes them, 0 if it declines
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "../paper_1410_3584_gb300/csrc/rings.h"

static std::atomic<long> g_count{0}, g_fail{-1};

static void *take(std::size_t n) {
    const long k = g_count.fetch_add(1), f = g_fail.load();
    if (f >= 0 && k >= f) throw std::bad_alloc();
    void *p = std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void *operator new(std::size_t n) { return take(n); }
void *operator new[](std::size_t n) { return take(n); }
void *operator new(std::size_t n, const std::nothrow_t &) noexcept { return std::malloc(n ? n : 1); }
void operator delete(void *p) noexcept { std::free(p); }
void operator delete[](void *p) noexcept { std::free(p); }
void operator delete(void *p, std::size_t) noexcept { std::free(p); }
void operator delete[](void *p, std::size_t) noexcept { std::free(p); }

using namespace nlp;

// 1: built, 0: declined
static int build(int dim, double far, int nr, int nth, int nph) {
    auto z = [&](int64_t j, int a) {
        const int c = (int)(j % nph), b = (int)(j / nph) % nth, i = (int)(j / nph / nth);
        const double r = far * (i + .5) / (nr - .5), u = dim == 3 ? (b + .5) / nth : 0.0;
        const double s = r * std::sqrt(1 - u * u), ph = (dim == 3 ? 2 : 1) * M_PI * c / nph;
        return a == 2 ? r * u : s * (a == 0 ? std::cos(ph) : std::sin(ph));
    };
    RingBuild B;
    if (dim == 3) {
        RingParams R{{40, 36, 32}, 7, 1, 768, 128, 1, 2, (int64_t)nr * nth, nph};
        return build_rings(R, z, B);
    }
    std::vector<RingSpan> span;
    RingParams R{{40, 36, 1}, 7, 1, 768, 128, 2, 40, nr, nph};
    return build_rings_2d(R, z, B, span);
}

int main(int argc, char **argv) {
    if (argc != 3) return 2;
    if (!std::strcmp(argv[1], "far")) {
        for (int dim = 3; dim >= 2; --dim) std::printf("%d ", build(dim, atof(argv[2]), 6, dim == 3 ? 4 : 1, 600));
        return 0;
    }
    for (int dim = 3; dim >= 2; --dim) {
        g_fail = -1;
        g_count = 0;
        if (!build(dim, 18, 6, dim == 3 ? 4 : 1, 40)) return 1;
        const long n = g_count.load();
        int caught = 0, tried = 0;
        for (long f = 0; f < n; f += atol(argv[2])) {   // (allocations of a build vary a little with the threads)
            g_fail = f;
            g_count = 0;
            ++tried;
            try {
                build(dim, 18, 6, dim == 3 ? 4 : 1, 40);
            } catch (const std::bad_alloc &) {
                ++caught;
            }
            g_fail = -1;
        }
        if (caught < tried - 2) return 1;
    }
    return 0;
}
