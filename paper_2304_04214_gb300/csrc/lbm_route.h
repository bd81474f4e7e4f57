// lbm_route.h -- which kernels run a time step, by the chosen variant, storage
// and grid: host arithmetic only (no CUDA header), so that a C++ compiler alone
// can build and check it.
#pragma once
#include "lbm.h"

#ifndef LBM_STEP_THREADS
#define LBM_STEP_THREADS 128   // threads per block of the step kernels (BX x BY)
#endif

namespace lbmk {

constexpr int BY = 2;  // rows per block: (0,1) and (ny-2,ny-1) share a block
constexpr int STEP_THREADS = LBM_STEP_THREADS;

struct StepRoute {
    int kind;      // the kernel of the interior rows: LBM_KERNEL_CELL, PAIR, QUAD or STAGED
    bool one;      // wall blocks and interior blocks in one launch (CELL, PAIR), or the
                   // wall rows on the side stream beside the interior kernel
    bool split;    // 16-bit CELL: the two cells of a thread are a block's width apart
    bool even;     // QUAD on rows that start on a pair of cells only (nx = 4m + 2)
    int bx, nbx;   // threads of a block along x, blocks along x
};

// The variant that `kind` stands for: AUTO is QUAD for the 16-bit storages where
// nx is a multiple of four, else PAIR (nx even), else CELL.
inline int resolve_kind(int kind, int elem, int nx) {
    if (kind != LBM_KERNEL_AUTO) return kind;
    if (elem == 2 && nx % 4 == 0) return LBM_KERNEL_QUAD;
    return nx % 2 == 0 ? LBM_KERNEL_PAIR : LBM_KERNEL_CELL;
}

// Up to about 100,000 cells all blocks of the one launch are resident at once and
// it saves the fork and join (64x32x32: FP32 5.1 -> 4.4 us per step in a graph, FP16
// 5.4 -> 4.8); beyond that the wall blocks, whose chain is the longer one, hold
// up the interior ones that wait for their place (96x32x48: FP32 6.0 -> 6.5 us;
// 400x40x32: 11.6 -> 12.6).
constexpr long long ONE_LAUNCH_CELLS = 100000;

// kind: the variant chosen (LBM_KERNEL_AUTO or a name); objective: the step sums
// an adjoint window's objective, which the CELL and PAIR kernels can; elem: bytes of
// a stored population.  A variant chosen by name runs as that kernel on every
// lattice it accepts.  AUTO takes what is fastest and gives the same bits: PAIR's
// kernel for a step in one launch, QUAD's for larger 16-bit lattices of even nx.
inline StepRoute step_route(int kind, bool objective, int elem, int nx, int ny, int nz) {
    StepRoute r;
    const bool named_quad = kind == LBM_KERNEL_QUAD && !objective;
    r.kind = resolve_kind(kind, elem, nx);
    if (objective && r.kind != LBM_KERNEL_CELL) r.kind = LBM_KERNEL_PAIR;
    r.split = r.kind == LBM_KERNEL_CELL && elem == 2;
    r.one = (long long)nx * ny * nz <= ONE_LAUNCH_CELLS && r.kind != LBM_KERNEL_STAGED && !named_quad;
    if (r.one && r.kind == LBM_KERNEL_QUAD) r.kind = LBM_KERNEL_PAIR;
    r.even = false;
    if (!r.one && kind == LBM_KERNEL_AUTO && r.kind == LBM_KERNEL_PAIR && elem == 2) {
        // 16-bit words are worth four cells a thread also where rows start on a pair
        r.kind = LBM_KERNEL_QUAD;
        r.even = true;
    }
    if (r.kind == LBM_KERNEL_CELL && elem == 4) {
        r.bx = r.one || nx < 64 ? 32 : 64;
        r.nbx = (nx + r.bx - 1) / r.bx;
    } else if (r.kind == LBM_KERNEL_QUAD) {
        r.bx = 32;
        r.nbx = (nx + 4 * r.bx - 1) / (4 * r.bx);
    } else {
        // two cells a thread: 2 bx columns of two rows; bx = 32 where it covers
        // the row with fewer empty columns (400 columns: 448 instead of 512, 11.4 ->
        // 10.8 us per 400x40x32 FP32 step)
        const int n32 = (nx + 63) / 64, wide = STEP_THREADS / BY;
        r.bx = n32 % (wide / 32) ? 32 : wide;
        r.nbx = (nx + 2 * r.bx - 1) / (2 * r.bx);
    }
    return r;
}

}  // namespace lbmk
