// Host construction of the ring decomposition of the 3D node set (see ring_dev.cuh).
//
// The spherical quadrature is a tensor product, so the n_phi nodes of one (r, theta) pair form
// a ring at one k_z: they share the w kernel values of the last axis.  A ring is cut into arcs
// (runs of consecutive nodes), and every arc owns a strip: for each fine-grid row y that its
// nodes reach, the interval of x that they reach.  The type-2 interpolation contracts the
// last axis once per strip cell (instead of once per node and column) and then takes w^2 taps
// per node; the type-1 spreading is the transpose.  The strips are exchanged with the fine
// grid by patches of 8 x 4 columns, each holding the list of the arcs that reach it, sorted by
// their first tap along the last axis.
#pragma once
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <numeric>
#include <vector>

#include "ring_types.h"

namespace nlp {

constexpr int kArcNodes = 128;            // most nodes of an arc
constexpr int kArcRows = 1024;            // most rows of a strip
constexpr double kRingFar = 1 << 28;      // node coordinates stay below it (32-bit tables)

struct RingParams {
    int nf[3];
    int w;
    int pad;         // footprint of a node along x: 0 = its w taps, 1 = the even-aligned window around them
    int cell_max;    // most cells of a strip
    int item_len;    // most entries of an item
    int turn;        // 1: the rings are whole turns (3D), 2: half turns (2D)
    int lane_cost;   // cost of a node's lane against a strip cell's
    int64_t nring;
    int nph;
    int arc_nodes = kArcNodes;   // most nodes of an arc of this plan
};

struct RingBuild {
    std::vector<RingArc> arcs;         // largest strips first
    std::vector<int> rows;             // per arc row: cell of x = xbase, relative to cell0
    std::vector<int64_t> node;         // source node of every stored node
    std::vector<int> nx, ny;           // per stored node: footprint origin, relative to its arc
    std::vector<int> ox, oy;           // per stored node: footprint origin on the unwrapped fine grid
    std::vector<RingEnt> ents;
    std::vector<int> pat;              // active patches, most entries first: id, first item, end
    std::vector<RingItem> item;        // runs of the patches' entries
    int64_t planes = 0;                // scratch planes of all items
    std::vector<int64_t> psi_ring;     // per kernel-value row: ring, sign (+1 / -1) and first tap
    std::vector<int> psi_sign, psi_s;
    int64_t cells = 0;
    int zlen = 0;                      // planes [0, zlen) of the half spectrum that windows reach
    RingClass cls[kArcClasses] = {};
};

// cells of a node's footprint along x (along y: its w taps)
inline int ring_window(int w, int pad) { return pad ? 2 * ((w + 2) / 2) : w; }

// Farthest position from 0 that the footprint of a node at |z| <= m reaches along an axis.  Its taps end
// within w/2 of it; a padded footprint (along x) starts at most one position below the first tap and so
// ends up to ring_window - w positions past the last, two for even w.  Those cells have zero weights, but
// they are read: the spectrum has to be written there as well.
inline int64_t ring_reach(double m, int w, int pad) {
    return (int64_t)std::min(1e9, std::floor(m + 0.5 * w)) + (ring_window(w, pad) - w);
}

inline int64_t ring_floordiv(int64_t a, int64_t b) { return a >= 0 ? a / b : -((-a + b - 1) / b); }

// Runs parts of a parallel region: an exception may not leave the region (the process would end), so the
// first one stops the rest, and rethrow() raises it as std::bad_alloc, which is all they can be, after it.
class RegionGuard {
    std::atomic<bool> failed_{false};

public:
    template <class Fn> void run(const Fn &fn) {
        if (failed_.load(std::memory_order_relaxed)) return;
        try {
            fn();
        } catch (...) {
            failed_.store(true);
        }
    }
    void rethrow() const {
        if (failed_.load()) throw std::bad_alloc();
    }
};

struct ArcTmp { RingArc a; int64_t ring; int c0, y0, xb; };
// The arcs with their rows' intervals [lo, hi) of x, in ring order.
struct RingArcs {
    std::vector<ArcTmp> arcs;
    std::vector<std::vector<int>> lo, hi;
};

// z(j, a): strip coordinate of node j, a = 0 along the rows (x), 1 across them (y); the nodes of
// ring r are r nph .. r nph + nph - 1, their angles spanning 2 pi / R.turn.  Fills the arcs, rows and
// nodes of B.  False if the sizes or coordinates do not fit the 32-bit tables.
template <class Coord> bool build_arcs(const RingParams &R, const Coord &z, RingBuild &B, RingArcs &out) {
    const int w = R.w, W = ring_window(w, R.pad), nph = R.nph;
    const int64_t nring = R.nring, M = nring * nph;
    std::vector<int> fx(M), fy(M);   // footprint origins
    std::atomic<bool> fits(true);
    RegionGuard guard;
#pragma omp parallel for schedule(static)
    for (int64_t j = 0; j < M; ++j) {
        if (!(std::fabs(z(j, 0)) < kRingFar && std::fabs(z(j, 1)) < kRingFar)) {
            fits.store(false);
            continue;
        }
        const int64_t x0 = (int64_t)std::ceil(z(j, 0) - 0.5 * w), y0 = (int64_t)std::ceil(z(j, 1) - 0.5 * w);
        fx[j] = (int)(R.pad ? 2 * ring_floordiv(x0, 2) : x0);
        fy[j] = (int)y0;
    }
    if (!fits.load()) return false;
    // ---- arcs: each ring in K equal runs, K the candidate of least cost: powers of two (a whole
    // small ring keeps its hole; halves split where x changes sign have one interval per row)
    // and the counts that fill a warp with 32, 64, 96 or 128 nodes a run, subject to the limits on
    // cells, rows and nodes.  Cost in cells: the strips' cells and rows, the lanes that the nodes
    // occupy (32 at a time) and a launch share per arc.
    auto arc_range = [&](int K, int a, int &c0, int &c1) {
        const int sh = K == 1 || R.turn > 1 ? 0 : (int)((3 * (int64_t)nph) / 4);   // halves where x changes sign
        c0 = sh + (int)((int64_t)a * nph / K);
        c1 = sh + (int)((int64_t)(a + 1) * nph / K);
    };
    struct Scratch { std::vector<int> lo, hi; };
    auto strip = [&](int64_t ring, int c0, int c1, Scratch &S, int &ymin) -> int {   // cells of nodes [c0, c1) mod nph
        const int64_t b = ring * nph;
        int ylo = INT32_MAX, yhi = INT32_MIN;
        for (int c = c0; c < c1; ++c) {
            const int64_t j = b + (c >= nph ? c - nph : c);
            ylo = std::min(ylo, fy[j]);
            yhi = std::max(yhi, fy[j]);
        }
        const int nr = yhi - ylo + w;
        if (nr > kArcRows) return INT32_MAX;   // past its limits
        S.lo.assign(nr, INT32_MAX);
        S.hi.assign(nr, INT32_MIN);
        for (int c = c0; c < c1; ++c) {
            const int64_t j = b + (c >= nph ? c - nph : c);
            const int x = fx[j], r0 = fy[j] - ylo;
            for (int r = r0; r < r0 + w; ++r) {
                S.lo[r] = std::min(S.lo[r], x);
                S.hi[r] = std::max(S.hi[r], x + W);
            }
        }
        int64_t n = 0;
        for (int r = 0; r < nr; ++r)
            if (S.hi[r] > S.lo[r]) n += S.hi[r] - S.lo[r];
        ymin = ylo;
        return (int)std::min<int64_t>(n, INT32_MAX);
    };
    std::vector<int> Ks(nring);
#pragma omp parallel
    {
        Scratch S;
#pragma omp for schedule(dynamic, 8)
        for (int64_t g = 0; g < nring; ++g) guard.run([&] {
            int64_t best = INT64_MAX;
            int bestK = nph, worse = 0;
            auto attempt = [&](int K) {   // false: past its limits
                int64_t cost = 0;
                for (int a = 0; a < K; ++a) {
                    int c0, c1, y;
                    arc_range(K, a, c0, c1);
                    if (c1 - c0 > R.arc_nodes) return false;
                    const int n = strip(g, c0, c1, S, y);
                    if (n > R.cell_max) return false;
                    cost += 48 + n + (int)S.lo.size() + (int64_t)R.lane_cost * ((c1 - c0 + 31) / 32 * 32);
                }
                if (cost < best) {
                    best = cost;
                    bestK = K;
                    worse = 0;
                } else {
                    ++worse;
                }
                return true;
            };
            for (int K = 1;; K = std::min(2 * K, nph)) {
                attempt(K);
                if (K >= nph || worse >= 1) break;
            }
            for (int m = std::min(32, R.arc_nodes); m <= R.arc_nodes; m += 32) {
                const int K = (nph + m - 1) / m;
                if (K & (K - 1)) attempt(K);
            }
            Ks[g] = bestK;
        });
    }
    guard.rethrow();
    std::vector<int64_t> first(nring + 1, 0);
    for (int64_t g = 0; g < nring; ++g) first[g + 1] = first[g] + Ks[g];
    const int64_t na = first[nring];
    if (na > (1 << 28)) return false;
    std::vector<ArcTmp> &arcs = out.arcs;
    std::vector<std::vector<int>> &lo = out.lo, &hi = out.hi;
    arcs.resize(na);
    lo.resize(na);
    hi.resize(na);
#pragma omp parallel
    {
        Scratch S;
#pragma omp for schedule(dynamic, 8)
        for (int64_t g = 0; g < nring; ++g) guard.run([&] {
            for (int a = 0; a < Ks[g]; ++a) {
                ArcTmp &A = arcs[first[g] + a];
                int c0, c1;
                arc_range(Ks[g], a, c0, c1);
                A.ring = g;
                A.c0 = c0;
                A.a.j0 = 0;
                A.a.j1 = c1 - c0;
                A.a.ncell = strip(g, c0, c1, S, A.y0);
                A.a.nrow = (int)S.lo.size();
                int xb = INT32_MAX;
                for (size_t r = 0; r < S.lo.size(); ++r) xb = std::min(xb, S.lo[r]);
                A.xb = xb;
                lo[first[g] + a] = S.lo;
                hi[first[g] + a] = S.hi;
            }
        });
    }
    guard.rethrow();
    // strip storage and nodes in ring order; the arcs themselves largest strip first
    int64_t cells = 0, rows = 0, nodes = 0;
    for (int64_t i = 0; i < na; ++i) {
        RingArc &a = arcs[i].a;
        if (a.ncell > R.cell_max) return false;
        a.cell0 = (int)cells;
        a.row0 = (int)rows;
        const int n = a.j1;
        a.j0 = (int)nodes;
        a.j1 = (int)(nodes + n);
        cells += (a.ncell + 1) & ~1;
        rows += a.nrow;
        nodes += n;
        if (cells > INT32_MAX - 4096 || rows > INT32_MAX - 4096) return false;
    }
    B.cells = cells;
    B.rows.resize(rows);
    B.node.resize(M);
    B.nx.resize(M);
    B.ny.resize(M);
    B.ox.resize(M);
    B.oy.resize(M);
#pragma omp parallel for schedule(dynamic, 8)
    for (int64_t i = 0; i < na; ++i) {
        const ArcTmp &A = arcs[i];
        int o = 0;
        for (int r = 0; r < A.a.nrow; ++r) {   // xs = lo: cell(x) = o + x - lo = (o - (lo - xb)) + (x - xb)
            const int n = hi[i][r] > lo[i][r] ? hi[i][r] - lo[i][r] : 0;
            B.rows[A.a.row0 + r] = n > 0 ? o - (lo[i][r] - A.xb) : 0;
            o += n;
        }
        for (int u = 0; u < A.a.j1 - A.a.j0; ++u) {
            const int c = A.c0 + u;
            const int64_t j = A.ring * nph + (c >= nph ? c - nph : c), q = A.a.j0 + u;
            B.node[q] = j;
            B.nx[q] = fx[j] - A.xb;
            B.ny[q] = fy[j] - A.y0;
            if (B.nx[q] > 32767 || B.ny[q] > 32767) fits.store(false);
            B.ox[q] = fx[j];
            B.oy[q] = fy[j];
        }
    }
    if (!fits.load()) return false;   // origins are packed as 16-bit offsets
    // ---- arcs by size, in classes of strip sizes (each a launch with its own shared memory)
    std::vector<int> order(na);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return arcs[a].a.ncell > arcs[b].a.ncell; });
    B.arcs.resize(na);
    for (int64_t i = 0; i < na; ++i) B.arcs[i] = arcs[order[i]].a;
    int c = 0;
    for (int64_t i = 0; i < na;) {
        // class c: strips of more than cell_max / 2^(c+1) cells, the last class all that are left
        if (c + 1 < kArcClasses && B.arcs[i].ncell <= (R.cell_max >> (c + 1))) {
            B.cls[c++].end = (int)i;
            continue;
        }
        RingClass &C = B.cls[c];
        C.cells = std::max(C.cells, (B.arcs[i].ncell + 1) & ~1);
        C.rows = std::max(C.rows, B.arcs[i].nrow);
        C.nodes = std::max(C.nodes, (B.arcs[i].j1 - B.arcs[i].j0 + 1) & ~1);
        ++i;
    }
    for (; c < kArcClasses; ++c) B.cls[c].end = (int)na;
    return true;
}

// Entries of a strip's cells on the patches, cells numbered by the strip coordinates modulo
// (NX, NY): the arc itself (sgn +1) or its mirror image at -l (sgn -1); columns x past xmax are
// left out.  emit(patch, entry) for every patch the arc reaches; cell: scratch.
template <class Emit>
void arc_entries(const ArcTmp &A, const std::vector<int> &lo, const std::vector<int> &hi, const std::vector<int> &rows,
                 int NX, int NY, int xmax, int sgn, std::vector<RingEnt> &cell, const Emit &emit) {
    const int PX = (NX + kPatchX - 1) / kPatchX, PY = (NY + kPatchY - 1) / kPatchY;
    // virtual patches: period index times patches per period plus patch
    auto vx = [&](int64_t x) { const int64_t q = ring_floordiv(x, NX); return q * PX + (x - q * NX) / kPatchX; };
    auto vy = [&](int64_t y) { const int64_t q = ring_floordiv(y, NY); return q * PY + (y - q * NY) / kPatchY; };
    int64_t x0 = INT64_MAX, x1 = INT64_MIN;
    for (int r = 0; r < A.a.nrow; ++r) {
        if (hi[r] <= lo[r]) continue;
        x0 = std::min<int64_t>(x0, sgn > 0 ? lo[r] : -(hi[r] - 1));
        x1 = std::max<int64_t>(x1, sgn > 0 ? hi[r] - 1 : -lo[r]);
    }
    const int64_t ya = sgn > 0 ? A.y0 : -(A.y0 + A.a.nrow - 1), yb = ya + A.a.nrow - 1;
    const int64_t vx0 = vx(x0), vy0 = vy(ya);
    const int64_t mx = vx(x1) - vx0 + 1, my = vy(yb) - vy0 + 1;
    cell.assign((size_t)(mx * my), RingEnt{});
    for (int64_t y = ya; y <= yb; ++y) {
        const int r = (int)(sgn > 0 ? y - A.y0 : -y - A.y0);
        if (hi[r] <= lo[r]) continue;
        const int64_t xs = sgn > 0 ? lo[r] : -(int64_t)(hi[r] - 1);
        const int64_t xe = sgn > 0 ? hi[r] : -(int64_t)lo[r] + 1;
        const int64_t base = (int64_t)A.a.cell0 + rows[A.a.row0 + r] - A.xb;   // cell of x = base + x
        const int64_t qy = ring_floordiv(y, NY), yw = y - qy * NY;
        const int ry = (int)(yw % kPatchY);
        int64_t q0 = ring_floordiv(xs, NX) * NX, org = q0 + (xs - q0) / kPatchX * kPatchX;   // of the period, of the patch
        RingEnt *e = &cell[(size_t)((qy * PY + yw / kPatchY - vy0) * mx + (vx(xs) - vx0))];
        for (int64_t x = xs; x < xe; ++e) {
            const int64_t end = std::min(xe, std::min(org + kPatchX, q0 + NX));
            const int64_t len = std::min(end, q0 + xmax + 1) - x;   // columns past xmax are left out
            if (len > 0) e->mask |= ((1u << len) - 1) << (ry * kPatchX + (int)(x - org));
            e->off[ry] = (int)(sgn > 0 ? base + org : base - org);
            x = end;
            if (end == q0 + NX) q0 += NX;
            org = end;
        }
    }
    for (int64_t v = 0; v < mx * my; ++v) {
        if (!cell[v].mask) continue;
        const int64_t X = vx0 + v % mx, Y = vy0 + v / mx;
        emit((int)((X - ring_floordiv(X, PX) * PX) * PY + (Y - ring_floordiv(Y, PY) * PY)), cell[v]);
    }
}

// The slices' entries by patch, each patch's in slice order: out[off[p]] .. out[off[p + 1] - 1] are those of
// patch p, as get(entry).  (A counting sort: the patches are known, and a comparison sort of all entries
// was a third of the time to create a 2D plan.)  The slices are emptied.
template <class Tmp, class Out, class Get>
void entries_by_patch(std::vector<std::vector<Tmp>> &part, int np, std::vector<int> &off, std::vector<Out> &out,
                      const Get &get) {
    off.assign(np + 1, 0);
    size_t n = 0;
    for (auto &p : part) {
        n += p.size();
        for (const Tmp &T : p) off[T.patch + 1]++;
    }
    for (int p = 0; p < np; ++p) off[p + 1] += off[p];
    std::vector<int> pos(off.begin(), off.end() - 1);
    out.resize(n);
    for (auto &p : part) {
        for (const Tmp &T : p) out[pos[T.patch]++] = get(T);
        std::vector<Tmp>().swap(p);
    }
}

// The ring decomposition of 3D nodes: arcs on the first two axes, kernel-value rows along the last.
template <class Coord> bool build_rings(const RingParams &R, const Coord &z, RingBuild &B) {
    RingArcs S;
    if (!build_arcs(R, z, B, S)) return false;
    const std::vector<ArcTmp> &arcs = S.arcs;
    const int w = R.w, nph = R.nph;
    const int64_t nring = R.nring, na = (int64_t)arcs.size();
    // ---- kernel-value rows: the ring itself (first tap s), and the images of it (the conjugate
    // at -l and the periods along the last axis) that reach the stored planes [0, nf/2]
    const int N2 = R.nf[2], zhi = N2 / 2;
    struct Img { int row, sign; };
    std::vector<std::vector<Img>> img(nring);
    std::vector<int> ring_s(nring);
    for (int64_t g = 0; g < nring; ++g) {
        if (!(std::fabs(z(g * nph, 2)) < kRingFar)) return false;
        const int s = (int)std::ceil(z(g * nph, 2) - 0.5 * w);
        ring_s[g] = s;
        auto add = [&](int sign, int s0) {
            img[g].push_back({(int)B.psi_ring.size(), sign});
            B.psi_ring.push_back(g);
            B.psi_sign.push_back(sign);
            B.psi_s.push_back(s0);
            if (s0 <= zhi && s0 + w > 0) B.zlen = std::max(B.zlen, std::min(s0 + w, zhi + 1));
        };
        add(+1, s);   // row 0 of the ring: always there (the interpolation uses it)
        for (int sign = 1; sign >= -1; sign -= 2) {
            const int b = sign > 0 ? s : -(s + w - 1);   // first tap of the image
            for (int64_t k = ring_floordiv(-(int64_t)b - w, N2); k <= ring_floordiv(zhi - (int64_t)b, N2) + 1; ++k) {
                const int64_t t = b + k * N2;
                if (t > zhi || t + w <= 0 || (sign > 0 && k == 0)) continue;
                add(sign, (int)t);
            }
        }
    }
    if (B.psi_ring.size() >= (size_t)kEntRow) return false;
    // ---- entries: every (arc, image) on every patch it reaches
    const int NX = R.nf[0], NY = R.nf[1];
    const int PX = (NX + kPatchX - 1) / kPatchX, PY = (NY + kPatchY - 1) / kPatchY;
    struct Tmp { int patch, s; RingEnt e; };
    const int nt = 64;   // fixed slices of the arcs: the entry order does not depend on the threads
    std::vector<std::vector<Tmp>> part(nt);
    RegionGuard guard;
#pragma omp parallel for schedule(dynamic, 1)
    for (int t = 0; t < nt; ++t) guard.run([&] {
        std::vector<Tmp> &out = part[t];
        std::vector<RingEnt> cell;
        for (int64_t i = na * t / nt; i < na * (t + 1) / nt; ++i) {
            const ArcTmp &A = arcs[i];
            for (int sgn = 1; sgn >= -1; sgn -= 2) {
                bool any = false;
                for (const Img &m : img[A.ring]) any |= m.sign == sgn;
                if (!any) continue;
                arc_entries(A, S.lo[i], S.hi[i], B.rows, NX, NY, NX, sgn, cell, [&](int patch, const RingEnt &e) {
                    for (size_t k = 0; k < img[A.ring].size(); ++k) {
                        const Img &m = img[A.ring][k];
                        if (m.sign != sgn) continue;
                        Tmp T;
                        T.patch = patch;
                        T.s = B.psi_s[m.row];
                        T.e = e;
                        T.e.psi = (uint32_t)m.row | (sgn < 0 ? kEntMirror : 0u) | (k > 0 ? kEntSpread : 0u);
                        out.push_back(T);
                    }
                });
            }
        }
    });
    guard.rethrow();
    int64_t ne = 0;
    for (auto &p : part) ne += (int64_t)p.size();
    if (ne > INT32_MAX / 8) return false;
    const int np = PX * PY;
    std::vector<int> poff;
    std::vector<Tmp> all;
    entries_by_patch(part, np, poff, all, [](const Tmp &T) { return T; });
    B.ents.resize(ne);
#pragma omp parallel for schedule(dynamic, 16)
    for (int p = 0; p < np; ++p) {
        std::stable_sort(all.begin() + poff[p], all.begin() + poff[p + 1],
                         [](const Tmp &a, const Tmp &b) { return a.s < b.s; });
        for (int e = poff[p]; e < poff[p + 1]; ++e) B.ents[e] = all[e].e;
    }
    std::vector<int> act;
    for (int p = 0; p < np; ++p)
        if (poff[p + 1] > poff[p]) act.push_back(p);
    std::stable_sort(act.begin(), act.end(),
                     [&](int a, int b) { return poff[a + 1] - poff[a] > poff[b + 1] - poff[b]; });
    // items: runs of the patches' entries, long enough to amortise their first window of columns,
    // short enough for several warps per scheduler
    const int64_t len = std::max<int64_t>(32, std::min<int64_t>(R.item_len, ne / (152 * 48) + 1));
    for (int p : act) {
        B.pat.push_back(p);
        B.pat.push_back((int)B.item.size());
        const int64_t n = poff[p + 1] - poff[p], k = (n + len - 1) / len;
        for (int64_t u = 0; u < k; ++u) {
            RingItem I;
            I.patch = p;
            I.e0 = (int)(poff[p] + n * u / k);
            I.e1 = (int)(poff[p] + n * (u + 1) / k);
            // planes of G its entries reach: [z0, z1), in the scratch from plane0
            I.z0 = std::max(0, all[I.e0].s);
            I.z1 = std::max(I.z0, std::min(all[I.e1 - 1].s + w, B.zlen));
            I.plane0 = (int)B.planes;
            B.planes += I.z1 - I.z0;
            B.item.push_back(I);
        }
        B.pat.push_back((int)B.item.size());
        if (B.planes > INT32_MAX / 64) return false;
    }
    return true;
}

// The arcs of 2D nodes (x: the last axis, whose half spectrum 0 .. nf/2 is stored; y: axis 1) and,
// per patch, the arcs and mirror images that reach it: ents, and pat = {id, first entry, end}, the
// patches with most entries first.  Strips are read from the spectrum itself: span holds, per row,
// its first cell, x and y there, and its cells.
template <class Coord> bool build_rings_2d(const RingParams &R, const Coord &z, RingBuild &B, std::vector<RingSpan> &span) {
    RingArcs S;
    if (!build_arcs(R, z, B, S)) return false;
    const int64_t na = (int64_t)S.arcs.size();
    span.resize(B.rows.size());
#pragma omp parallel for schedule(static)
    for (int64_t i = 0; i < na; ++i) {
        const ArcTmp &A = S.arcs[i];
        for (int r = 0; r < A.a.nrow; ++r) {
            const int x = S.lo[i][r], n = S.hi[i][r] > x ? S.hi[i][r] - x : 0;
            span[A.a.row0 + r] = n ? RingSpan{A.a.cell0 + B.rows[A.a.row0 + r] + x - A.xb, x, A.y0 + r, n} : RingSpan{0, 0, 0, 0};
        }
    }
    const int NX = R.nf[0], NY = R.nf[1];
    const int np = ((NX + kPatchX - 1) / kPatchX) * ((NY + kPatchY - 1) / kPatchY);
    struct Tmp { int patch; RingEnt e; };
    const int nt = 64;   // fixed slices of the arcs: the entry order does not depend on the threads
    std::vector<std::vector<Tmp>> part(nt);
    RegionGuard guard;
#pragma omp parallel for schedule(dynamic, 1)
    for (int t = 0; t < nt; ++t) guard.run([&] {
        std::vector<RingEnt> cell;
        for (int64_t i = na * t / nt; i < na * (t + 1) / nt; ++i)
            for (int sgn = 1; sgn >= -1; sgn -= 2)
                arc_entries(S.arcs[i], S.lo[i], S.hi[i], B.rows, NX, NY, NX / 2, sgn, cell, [&](int patch, const RingEnt &e) {
                    part[t].push_back({patch, e});
                    part[t].back().e.psi = sgn < 0 ? kEntMirror : 0u;
                });
    });
    guard.rethrow();
    int64_t ne = 0;
    for (auto &p : part) ne += (int64_t)p.size();
    if (ne > INT32_MAX / 8) return false;
    std::vector<int> poff, act;
    entries_by_patch(part, np, poff, B.ents, [](const Tmp &T) { return T.e; });
    for (int p = 0; p < np; ++p)
        if (poff[p + 1] > poff[p]) act.push_back(p);
    std::stable_sort(act.begin(), act.end(), [&](int a, int b) { return poff[a + 1] - poff[a] > poff[b + 1] - poff[b]; });
    for (int p : act) {
        B.pat.push_back(p);
        B.pat.push_back(poff[p]);
        B.pat.push_back(poff[p + 1]);
    }
    return true;
}

}  // namespace nlp
