// Host check of ring_reach (csrc/rings.h): builds the rings (or the 2D arcs) of a node set and asserts
// that every footprint cell of every node lies within the reach that its axis is given.
// argv: nf0 nf1 nf2 nr nth nph f0 f1 f2 w pad (f: ball radius over the Nyquist radius; nth = 0: 2D).
// Prints how many nodes' footprints end at the reach along x; exit code 1 if one ends past it.
#include <cstdio>
#include <cstdlib>

#include "../paper_1410_3584_gb300/csrc/rings.h"

using namespace nlp;

int main(int argc, char **argv) {
    if (argc != 12) return 2;
    const int nf[3] = {atoi(argv[1]), atoi(argv[2]), atoi(argv[3])}, nr = atoi(argv[4]), nth = atoi(argv[5]);
    const int nph = atoi(argv[6]), w = atoi(argv[10]), pad = atoi(argv[11]), nu = nth ? nth : 1;
    const double f[3] = {atof(argv[7]), atof(argv[8]), atof(argv[9])};
    const int64_t M = (int64_t)nr * nu * nph;
    std::vector<double> pos(3 * M);
    double m[3] = {0, 0, 0};   // axis 0: x, the strips' rows; 1: across them; 2: the last axis (3D)
    for (int a = 0; a < nr; ++a)
        for (int b = 0; b < nu; ++b)
            for (int c = 0; c < nph; ++c) {
                double *p = &pos[3 * (((int64_t)a * nu + b) * nph + c)];
                const double r = (a + .5) / nr, u = (b + .5) / nu, st = std::sqrt(1 - u * u);
                const double ph = (nth ? 2 : 1) * M_PI * c / nph;
                if (nth) {
                    p[0] = f[0] * nf[0] / 2 * r * st * std::cos(ph);
                    p[1] = f[1] * nf[1] / 2 * r * st * std::sin(ph);
                    p[2] = f[2] * nf[2] / 2 * r * u;
                } else {
                    p[0] = f[2] * nf[2] / 2 * r * std::sin(ph);
                    p[1] = f[1] * nf[1] / 2 * r * std::cos(ph);
                }
                for (int k = 0; k < 3; ++k) m[k] = std::max(m[k], std::fabs(p[k]));
            }
    auto z = [&](int64_t j, int a) { return pos[3 * j + a]; };
    RingBuild B;
    std::vector<RingSpan> span;
    bool ok;
    if (nth) {
        RingParams R{{nf[0], nf[1], nf[2]}, w, pad, 768, 128, 1, 2, (int64_t)nr * nth, nph};
        ok = build_rings(R, z, B);
    } else {
        RingParams R{{nf[2], nf[1], 1}, w, pad, 768, 128, 2, 40, nr, nph};
        ok = build_rings_2d(R, z, B, span);
    }
    if (!ok || (int64_t)B.node.size() != M) return 2;
    const int64_t rx = ring_reach(m[0], w, pad), ry = ring_reach(m[1], w, 0), rz = ring_reach(m[2], w, 0);
    const int W = ring_window(w, pad);
    int64_t at = 0;
    for (int64_t q = 0; q < M; ++q) {
        const int64_t x0 = B.ox[q], x1 = x0 + W - 1, y0 = B.oy[q], y1 = y0 + w - 1;
        const int64_t z0 = nth ? (int64_t)std::ceil(z(B.node[q], 2) - .5 * w) : 0, z1 = nth ? z0 + w - 1 : 0;
        if (x0 < -rx || x1 > rx || y0 < -ry || y1 > ry || z0 < -rz || z1 > rz) {
            std::printf("node %lld: x %lld..%lld of %lld, y %lld..%lld of %lld, z %lld..%lld of %lld\n", (long long)q,
                        (long long)x0, (long long)x1, (long long)rx, (long long)y0, (long long)y1, (long long)ry,
                        (long long)z0, (long long)z1, (long long)rz);
            return 1;
        }
        at += x1 == rx || x0 == -rx;
    }
    std::printf("%lld\n", (long long)at);
    return 0;
}
