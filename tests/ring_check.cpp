// Host check of the ring decomposition (csrc/rings.h): builds it for a spherical node set of the
// given sizes, follows its tables as the kernels do (strips, nodes, patches, items, images) in
// FP64, and compares with the direct sums over every node's w^3 taps on the periodic grid.
// argv: nf0 nf1 nf2 nr nth nph f0 f1 f2 w pad cell_max (f: ball radius over the Nyquist radius).
// nth = 0: a 2D polar set on axes 1 and 2 (half turns, x along the last axis; nf0 and f0 unused).
// Prints the two relative errors; exit code 1 if a table points outside what it may.
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../paper_1410_3584_gb300/csrc/rings.h"

using namespace nlp;
typedef std::complex<double> C;

#define CHECK(x)                                                  \
    do {                                                          \
        if (!(x)) {                                               \
            std::printf("line %d: %s\n", __LINE__, #x);           \
            return 1;                                             \
        }                                                         \
    } while (0)

static int mod(int64_t a, int n) {
    const int64_t r = a % n;
    return (int)(r < 0 ? r + n : r);
}

// 2D: strips read from the half spectrum by their spans, spread values gathered by the patches
static int check_2d(int ny, int nx, int nr, int nph, double fy, double fx, int w, int pad, int cell_max) {
    RingParams R{{nx, ny, 1}, w, pad, cell_max, 128, 2, 2, nr, nph};
    const int64_t M = (int64_t)nr * nph;
    std::vector<double> pos(2 * M);
    for (int a = 0; a < nr; ++a)
        for (int c = 0; c < nph; ++c) {
            const double r = (a + .5) / nr, ph = M_PI * c / nph;
            pos[2 * ((int64_t)a * nph + c)] = fx * nx / 2 * r * std::sin(ph);
            pos[2 * ((int64_t)a * nph + c) + 1] = fy * ny / 2 * r * std::cos(ph);
        }
    auto z = [&](int64_t j, int a) { return pos[2 * j + a]; };
    RingBuild B;
    std::vector<RingSpan> span;
    CHECK(build_rings_2d(R, z, B, span));
    auto phi = [&](double t) {
        const double x = 2 * t / w, s = 1 - x * x;
        return s > 0 ? std::exp(2.3 * w * (std::sqrt(s) - 1)) : 0.0;
    };
    const int W = ring_window(w, pad), nh = nx / 2 + 1, PY = (ny + kPatchY - 1) / kPatchY;
    std::mt19937 g(1);
    std::normal_distribution<double> nd;
    std::vector<C> F((size_t)nx * ny);   // a random Hermitian spectrum [y][x]
    auto at = [&](int64_t y, int64_t x) -> C & { return F[(size_t)mod(y, ny) * nx + mod(x, nx)]; };
    for (C &v : F) v = C(nd(g), nd(g));
    for (int y = 0; y < ny; ++y)
        for (int x = 0; x < nx; ++x) {
            const C m = .5 * (at(y, x) + std::conj(at(-y, -x)));
            at(y, x) = m;
            at(-y, -x) = std::conj(m);
        }
    std::vector<C> A(B.cells + 2, C(NAN, NAN)), S(B.cells + 2, C(0, 0)), cj(M), G((size_t)ny * nh), H(G.size());
    double e1 = 0, n1 = 0, e2 = 0, n2 = 0;
    int64_t seen = 0;
    auto wgt = [&](int64_t q, int x, int y) { return phi(x - z(q, 0)) * phi(y - z(q, 1)); };
    for (const RingArc &a : B.arcs) {
        for (int r = 0; r < a.nrow; ++r) {
            const RingSpan &p = span[a.row0 + r];
            CHECK(p.n >= 0 && (p.n == 0 || p.cell >= a.cell0) && p.cell + p.n <= a.cell0 + a.ncell && a.cell0 + a.ncell <= B.cells);
            for (int c = 0; c < p.n; ++c) A[p.cell + c] = at(p.y, p.x + c);
        }
        for (int j = a.j0; j < a.j1; ++j, ++seen) {
            const int64_t q = B.node[j];
            const int x0 = (int)std::ceil(z(q, 0) - .5 * w), y0 = (int)std::ceil(z(q, 1) - .5 * w);
            C v = 0, ref = 0;
            cj[q] = C(nd(g), nd(g));
            for (int r = 0; r < w; ++r)
                for (int b = 0; b < W; ++b) {
                    const int c = a.cell0 + B.rows[a.row0 + B.ny[j] + r] + B.nx[j] + b;
                    CHECK(B.ny[j] + r < a.nrow && c >= a.cell0 && c < a.cell0 + a.ncell && !std::isnan(A[c].real()));
                    v += wgt(q, B.ox[j] + b, B.oy[j] + r) * A[c];
                    S[c] += wgt(q, B.ox[j] + b, B.oy[j] + r) * cj[q];
                }
            for (int r = 0; r < w; ++r)
                for (int b = 0; b < w; ++b) {
                    ref += wgt(q, x0 + b, y0 + r) * at(y0 + r, x0 + b);
                    const C t = cj[q] * wgt(q, x0 + b, y0 + r);
                    int k = mod(x0 + b, nx);
                    if (k < nh) H[(size_t)mod(y0 + r, ny) * nh + k] += t;
                    k = mod(-(x0 + b), nx);
                    if (k < nh) H[(size_t)mod(-(y0 + r), ny) * nh + k] += std::conj(t);
                }
            e1 = std::max(e1, std::abs(v - ref));
            n1 = std::max(n1, std::abs(ref));
        }
    }
    CHECK(seen == M);
    for (size_t p = 0; p < B.pat.size(); p += 3)
        for (int e = B.pat[p + 1]; e < B.pat[p + 2]; ++e) {
            const RingEnt &E = B.ents[e];
            for (int l = 0; l < 32; ++l) {
                if (!(E.mask >> l & 1)) continue;
                const int x = B.pat[p] / PY * kPatchX + l % 8, y = B.pat[p] % PY * kPatchY + l / 8;
                const bool m = E.psi & kEntMirror;
                const int c = m ? E.off[l / 8] - l % 8 : E.off[l / 8] + l % 8;
                CHECK(x < nh && y < ny && c >= 0 && c < B.cells);
                G[(size_t)y * nh + x] += m ? std::conj(S[c]) : S[c];
            }
        }
    for (size_t i = 0; i < G.size(); ++i) {
        e2 = std::max(e2, std::abs(G[i] - H[i]));
        n2 = std::max(n2, std::abs(H[i]));
    }
    std::printf("%.3e %.3e\n", e1 / n1, e2 / n2);
    return 0;
}

int main(int argc, char **argv) {
    CHECK(argc == 13);
    const int nx = atoi(argv[1]), ny = atoi(argv[2]), nz = atoi(argv[3]), nr = atoi(argv[4]), nth = atoi(argv[5]);
    const int nph = atoi(argv[6]), w = atoi(argv[10]), pad = atoi(argv[11]);
    const double f[3] = {atof(argv[7]), atof(argv[8]), atof(argv[9])};
    if (nth == 0) return check_2d(ny, nz, nr, nph, f[1], f[2], w, pad, atoi(argv[12]));
    RingParams R{{nx, ny, nz}, w, pad, atoi(argv[12]), 128, 1, 2, (int64_t)nr * nth, nph};
    const int64_t M = R.nring * nph;
    std::vector<double> pos(3 * M);
    for (int a = 0; a < nr; ++a)
        for (int b = 0; b < nth; ++b)
            for (int c = 0; c < nph; ++c) {
                const double r = (a + .5) / nr, u = (b + .5) / nth, st = std::sqrt(1 - u * u), ph = 2 * M_PI * c / nph;
                double *p = &pos[3 * (((int64_t)a * nth + b) * nph + c)];
                p[0] = f[0] * nx / 2 * r * st * std::cos(ph);
                p[1] = f[1] * ny / 2 * r * st * std::sin(ph);
                p[2] = f[2] * nz / 2 * r * u;
            }
    auto z = [&](int64_t j, int a) { return pos[3 * j + a]; };
    RingBuild B;
    CHECK(build_rings(R, z, B));
    auto phi = [&](double t) {
        const double x = 2 * t / w, s = 1 - x * x;
        return s > 0 ? std::exp(2.3 * w * (std::sqrt(s) - 1)) : 0.0;
    };
    const int W = ring_window(w, pad), nh = nz / 2 + 1, PY = (ny + kPatchY - 1) / kPatchY;
    int64_t seen = 0;
    for (size_t i = 0; i < B.arcs.size(); ++i) {
        const RingArc &a = B.arcs[i];
        int c = 0;
        while ((int)i >= B.cls[c].end) ++c;
        CHECK(a.ncell <= B.cls[c].cells && a.nrow <= B.cls[c].rows && a.j1 - a.j0 <= B.cls[c].nodes);
        CHECK(a.cell0 % 2 == 0 && a.cell0 + a.ncell <= B.cells && (!pad || a.ncell % 2 == 0));
        seen += a.j1 - a.j0;
        for (int j = a.j0; j < a.j1; ++j)
            for (int r = 0; r < w; ++r) {
                CHECK(B.ny[j] + r < a.nrow);
                const int o = B.rows[a.row0 + B.ny[j] + r] + B.nx[j];
                CHECK(o >= 0 && o + W <= a.ncell && (!pad || o % 2 == 0));
            }
    }
    CHECK(seen == M);
    // a random Hermitian spectrum
    std::mt19937 g(1);
    std::normal_distribution<double> nd;
    std::vector<C> F((size_t)nx * ny * nz);
    auto at = [&](int64_t x, int64_t y, int64_t q) -> C & { return F[((size_t)mod(x, nx) * ny + mod(y, ny)) * nz + mod(q, nz)]; };
    for (C &v : F) v = C(nd(g), nd(g));
    for (int x = 0; x < nx; ++x)
        for (int y = 0; y < ny; ++y)
            for (int q = 0; q < nz; ++q) {
                const C m = .5 * (at(x, y, q) + std::conj(at(-x, -y, -q)));
                at(x, y, q) = m;
                at(-x, -y, -q) = std::conj(m);
            }
    auto psi = [&](int row, int i) {
        const double zc = z(B.psi_ring[row] * nph, 2);
        return phi(std::ceil(zc - .5 * w) + (B.psi_sign[row] > 0 ? i : w - 1 - i) - zc);
    };
    for (size_t p = 0; p < B.pat.size(); p += 3)
        for (int i = B.pat[p + 1]; i < B.pat[p + 2]; ++i) {
            const RingItem &I = B.item[i];
            CHECK(I.patch == B.pat[p] && I.e1 > I.e0 && I.z0 >= 0 && I.z1 >= I.z0 && I.z1 <= std::max(I.z0, B.zlen));
            CHECK(I.plane0 + I.z1 - I.z0 <= B.planes);
            if (i > B.pat[p + 1])
                CHECK(B.item[i - 1].e1 == I.e0 && B.item[i - 1].z0 <= I.z0 && B.item[i - 1].z1 <= I.z1);
        }
    // columns -> strips
    std::vector<C> A(B.cells + 2, C(NAN, NAN)), S(B.cells + 2, C(0, 0));
    for (const RingItem &I : B.item) {
        int before = INT32_MIN;
        for (int e = I.e0; e < I.e1; ++e) {
            const RingEnt &E = B.ents[e];
            const int row = (int)(E.psi & kEntRow), s = B.psi_s[row];
            CHECK(s >= before);
            before = s;
            if (E.psi & kEntSpread) continue;
            for (int l = 0; l < 32; ++l) {
                if (!(E.mask >> l & 1)) continue;
                const int x = I.patch / PY * kPatchX + l % 8, y = I.patch % PY * kPatchY + l / 8, c = E.off[l / 8] + l % 8;
                CHECK(x < nx && y < ny && c >= 0 && c < B.cells);
                C t = 0;
                for (int i = 0; i < w; ++i) t += psi(row, i) * at(x, y, s + i);
                A[c] = t;
            }
        }
    }
    // nodes: interpolation against the direct sum, then random values spread over the strips
    std::vector<C> cj(M);
    double e1 = 0, n1 = 0, e2 = 0, n2 = 0;
    auto wgt = [&](int64_t q, int x, int y) { return phi(x - z(q, 0)) * phi(y - z(q, 1)); };
    for (const RingArc &a : B.arcs)
        for (int j = a.j0; j < a.j1; ++j) {
            const int64_t q = B.node[j];
            const int t[3] = {(int)std::ceil(z(q, 0) - .5 * w), (int)std::ceil(z(q, 1) - .5 * w), (int)std::ceil(z(q, 2) - .5 * w)};
            C v = 0, ref = 0;
            cj[q] = C(nd(g), nd(g));
            for (int r = 0; r < w; ++r)
                for (int b = 0; b < W; ++b) {
                    const int c = a.cell0 + B.rows[a.row0 + B.ny[j] + r] + B.nx[j] + b;
                    CHECK(!std::isnan(A[c].real()));   // every cell of a footprint was written
                    v += wgt(q, B.ox[j] + b, B.oy[j] + r) * A[c];
                    S[c] += wgt(q, B.ox[j] + b, B.oy[j] + r) * cj[q];
                }
            for (int r = 0; r < w; ++r)
                for (int b = 0; b < w; ++b)
                    for (int i = 0; i < w; ++i)
                        ref += wgt(q, t[0] + b, t[1] + r) * phi(t[2] + i - z(q, 2)) * at(t[0] + b, t[1] + r, t[2] + i);
            e1 = std::max(e1, std::abs(v - ref));
            n1 = std::max(n1, std::abs(ref));
        }
    // strips -> columns (with the images), against the direct spreading of values and conjugates
    std::vector<C> G((size_t)nx * ny * nh), H(G.size());
    for (const RingItem &I : B.item)
        for (int e = I.e0; e < I.e1; ++e) {
            const RingEnt &E = B.ents[e];
            const int row = (int)(E.psi & kEntRow);
            const bool m = E.psi & kEntMirror;
            for (int l = 0; l < 32; ++l) {
                if (!(E.mask >> l & 1)) continue;
                const int x = I.patch / PY * kPatchX + l % 8, y = I.patch % PY * kPatchY + l / 8;
                const int c = m ? E.off[l / 8] - l % 8 : E.off[l / 8] + l % 8;
                CHECK(c >= 0 && c < B.cells);
                for (int i = 0; i < w; ++i) {
                    const int q = B.psi_s[row] + i;
                    if (q < I.z0 || q >= I.z1) {
                        CHECK(q < 0 || q >= B.zlen);   // planes an item drops are not stored
                        continue;
                    }
                    G[((size_t)x * ny + y) * nh + q] += psi(row, i) * (m ? std::conj(S[c]) : S[c]);
                }
            }
        }
    for (int64_t q = 0; q < M; ++q) {
        const int t[3] = {(int)std::ceil(z(q, 0) - .5 * w), (int)std::ceil(z(q, 1) - .5 * w), (int)std::ceil(z(q, 2) - .5 * w)};
        for (int r = 0; r < w; ++r)
            for (int b = 0; b < w; ++b)
                for (int i = 0; i < w; ++i) {
                    const C v = cj[q] * wgt(q, t[0] + b, t[1] + r) * phi(t[2] + i - z(q, 2));
                    int k = mod(t[2] + i, nz);
                    if (k < nh) H[((size_t)mod(t[0] + b, nx) * ny + mod(t[1] + r, ny)) * nh + k] += v;
                    k = mod(-(t[2] + i), nz);
                    if (k < nh) H[((size_t)mod(-(t[0] + b), nx) * ny + mod(-(t[1] + r), ny)) * nh + k] += std::conj(v);
                }
    }
    for (size_t i = 0; i < G.size(); ++i) {
        e2 = std::max(e2, std::abs(G[i] - H[i]));
        n2 = std::max(n2, std::abs(H[i]));
    }
    std::printf("%.3e %.3e\n", e1 / n1, e2 / n2);
    return 0;
}
