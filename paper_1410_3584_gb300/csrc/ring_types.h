// Tables of the ring decomposition shared by its host construction (rings.h) and its kernels
// (ring_dev.cuh).
#pragma once
#include <cstddef>
#include <cstdint>

namespace nlp {

constexpr int kPatchX = 8, kPatchY = 4;   // columns of a patch (one warp)
constexpr int kArcClasses = 1;            // launches of the node kernel by strip size: all arcs in one

struct RingArc {
    int j0, j1;     // node range
    int cell0;      // first strip cell
    int ncell;
    int row0, nrow; // row table entries: strip cell of (x, row) = cell0 + row table + x
};

// One arc on one patch: lane l (x = l mod 8, y = l / 8) of `mask` has strip cell off[y] + x
// (mirror image: off[y] - x).
struct RingEnt {
    uint32_t mask;
    uint32_t psi;   // row of the last-axis kernel values, and the flags below
    int off[kPatchY];
};
constexpr uint32_t kEntMirror = 0x80000000u;   // conjugate image at -l (spreading only)
constexpr uint32_t kEntSpread = 0x40000000u;   // any image but the arc itself: spreading only
constexpr uint32_t kEntRow = 0x3fffffffu;

// A run of one patch's entries, and the planes of the scratch its columns go to (spreading).
struct RingItem {
    int patch, e0, e1;
    int z0, z1, plane0;
};

// 2D: the cells of one strip row: first cell, position (x, y) of it on the fine grid, count.
struct RingSpan {
    int cell, x, y, n;
};

// Arcs [previous class's end, end) and what their shared memory must hold.
struct RingClass {
    int end, cells, rows, nodes;
};

}  // namespace nlp
