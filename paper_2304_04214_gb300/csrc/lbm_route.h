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

// Bytes of a stored population.
inline int elem_bytes(int precision) { return precision == LBM_FP32 ? 4 : 2; }

// The variant that `kind` stands for: AUTO is QUAD for the 16-bit storages where
// nx is a multiple of four, else PAIR (nx even), else CELL.
inline int resolve_kind(int kind, int precision, int nx) {
    if (kind != LBM_KERNEL_AUTO) return kind;
    if (elem_bytes(precision) == 2 && nx % 4 == 0) return LBM_KERNEL_QUAD;
    return nx % 2 == 0 ? LBM_KERNEL_PAIR : LBM_KERNEL_CELL;
}

// A step in one launch saves the fork and join of the side stream (64x32x32 in a
// graph: FP32 5.4 -> 4.5 us, FP16 5.5 -> 4.7) as long as all its blocks are resident
// at once: the wall blocks, whose chain is the longer one, come first, and blocks
// that wait for their place hold up the step (us, one launch / two: 66x32x47 FP16
// 6.8 / 5.9, 8x110x110 FP32 16.9 / 15.7, 33x40x70 FP32 7.7 / 6.4; all resident: 48x48x42
// 5.66 / 5.70, 130x24x32 5.8 / 6.1).  The kernels' launch bounds keep this many
// threads resident on an SM; larger lattices fill the chip without it.
constexpr long long ONE_LAUNCH_CELLS = 100000;
constexpr int ONE_BLOCKS_PER_SM = 4;

// kind: the variant chosen (LBM_KERNEL_AUTO or a name); objective: the step sums
// an adjoint window's objective, which the CELL and PAIR kernels can; precision: the
// storage; sms: SMs of the device.  A variant chosen by name runs as that kernel on
// every lattice it accepts.  AUTO takes what is fastest and gives the same bits:
// PAIR's kernel for a step in one launch, QUAD's also on some larger lattices of
// nx = 4m + 2.
inline StepRoute step_route(int kind, bool objective, int precision, int nx, int ny, int nz, int sms) {
    StepRoute r;
    const int elem = elem_bytes(precision);
    const bool named_quad = kind == LBM_KERNEL_QUAD && !objective;
    r.kind = resolve_kind(kind, precision, nx);
    if (objective && r.kind != LBM_KERNEL_CELL) r.kind = LBM_KERNEL_PAIR;
    r.split = r.kind == LBM_KERNEL_CELL && elem == 2;
    r.even = false;
    const bool cell32 = r.kind == LBM_KERNEL_CELL && elem == 4;
    auto blocks = [&](int bx, int cells) { r.bx = bx; r.nbx = (nx + bx * cells - 1) / (bx * cells); };
    // two cells a thread: 2 bx columns of two rows; bx = 32 where it covers the row
    // with fewer empty columns (400 columns: 448 instead of 512, 11.4 -> 10.8 us per
    // 400x40x32 FP32 step)
    const int n32 = (nx + 63) / 64, wide = STEP_THREADS / BY, pair_bx = n32 % (wide / 32) ? 32 : wide;
    auto resident = [&] {
        return (long long)r.nbx * r.bx * ny * nz <= (long long)sms * ONE_BLOCKS_PER_SM * STEP_THREADS;
    };
    if (cell32) blocks(32, 1);
    else blocks(pair_bx, 2);
    // narrow odd rows: 32 columns to a block instead of 64 (21x100x100 FP16 15.2 -> 9.9 us;
    // one cell a thread 13.2), unless the wider blocks are all resident as it is
    // (21x16x30: 4.4 with 64, 4.9 with 32)
    if (r.split && nx <= 32 && !resident()) blocks(16, 2);
    // without interior rows there is nothing for wall rows to run beside (999x4x24 FP32
    // 5.7 / 6.9), and QUAD's warps of 128 columns are mostly empty on rows of up to 64
    // (16x60x100 FP16 10.0 / 11.4, 36x50x55 7.0 / 7.0, BF16 7.2 / 7.6)
    r.one = (long long)nx * ny * nz <= ONE_LAUNCH_CELLS && r.kind != LBM_KERNEL_STAGED && !named_quad &&
            (resident() || ny == 2 * BY || (r.kind == LBM_KERNEL_QUAD && nx <= 64));
    if (r.one) {
        if (r.kind == LBM_KERNEL_QUAD) r.kind = LBM_KERNEL_PAIR;
        return r;
    }
    if (cell32) blocks(nx < 64 ? 32 : 64, 1);
    const bool rowbase = precision == LBM_BF16_DEV || precision == LBM_FP16_ROW;
    if (kind == LBM_KERNEL_AUTO && r.kind == LBM_KERNEL_PAIR && rowbase && n32 % 2 == 0) {
        // Four cells a thread also where rows start on a pair of them, for the
        // storages whose row bases a thread then loads half as often, and if the warps
        // of 128 columns leave no more of them empty than two cells a thread do (us,
        // four / two cells: 602x60x48 BF16 28.0 / 28.7, 66x60x60 9.3 / 9.7, 222x60x60 FP16 row
        // 15.1 / 15.5; FP16 602x60x48 27.2 / 26.6; 34x60x60 BF16 9.2 / 7.3, 386x96x96 64.4 / 61.8)
        r.kind = LBM_KERNEL_QUAD;
        r.even = true;
    }
    if (r.kind == LBM_KERNEL_QUAD) blocks(32, 4);
    return r;
}

}  // namespace lbmk
