// tri_layout.cuh -- the shared-memory layout of the tridiagonal solves (lo.cu) and the shared
// memory a solve of n cells needs: for the kernels, their launchers and the batch, which sizes
// one launch for slabs of different n.  Host compilers can read it too.
#pragma once
#include <algorithm>
#include <cuda_runtime.h>
#include "../../include/trt.h"

namespace trt {

// The layout of a system's rows in shared memory: P chunks, chunk l the rows l n / P ..
// (l + 1) n / P - 1, its row k in slot k LP + l; face i shares the slot of row i, face n has
// the slot after all others.  LP is odd in units of 8 so that the staging's stores (threads
// along the rows) spread over the banks.  S is not monotone in n: an even n <= 256 has two
// rows in every chunk, an odd one three in one of them.
struct TriLayout {
    int P, LP, S;   // chunks, slots per row-in-chunk, slots
};
__host__ __device__ inline TriLayout tri_layout(int n)
{
    TriLayout t;
    t.P = n / 2 < 128 ? n / 2 : 128;
    if (t.P < 1) t.P = 1;
    t.LP = (t.P + 31) / 32 * 32 + 8;
    t.S = t.LP * ((n + t.P - 1) / t.P) + 1;
    return t;
}

// TriLayout's slots of the rows and faces 0 .. nx (Problem::lo_slot)
inline void lo_slots(int nx, int *slot)
{
    const TriLayout y = tri_layout(nx);
    for (int l = 0; l < y.P; ++l)
        for (int i = (l * nx) / y.P, k = 0; i < ((l + 1) * nx) / y.P; ++i, ++k) slot[i] = k * y.LP + l;
    slot[nx] = y.S - 1;
}

// shared memory of one LO solve: the rows, the pair form's 7th array (the face factors of
// Fold, free again when the solver wants its 3 P values), or the refined FP32 form's two
// copies of the rows
inline size_t lo_smem(int precision, int nx)
{
    const TriLayout y = tri_layout(nx);
    const size_t S = y.S, rb = 3 * (size_t)y.P;
    if (precision & TRT_LO_FP32) return 6 * S * (sizeof(double) + sizeof(float)) + rb * sizeof(float);
    if (precision & TRT_LO_PAIR) return (6 * S + std::max(S, rb)) * sizeof(double);
    return (6 * S + rb) * sizeof(double);
}

// doubles of the grey kernel's block maxima (32 per value)
constexpr int kGreyNV = 7;
constexpr int kGreyRed = 32 * kGreyNV;

// shared memory of one grey solve: Newton terms, block maxima, the solver's rows
inline size_t grey_smem(int nx)
{
    const TriLayout y = tri_layout(nx);
    return sizeof(double) * (3 * (size_t)nx + kGreyRed + 6 * (size_t)y.S + 3 * (size_t)y.P);
}

// The shared memory of launches that cover several slabs, and their largest n: each slab's
// CTA lays out its own n, so the most that any slab needs, not the need of the largest slab
// (60 cells need 4608 bytes of an FP64 solve, 59 cells 6504).
struct BatchSmem {
    int max_nx = 1;
    size_t lo = 0, grey = 0;
    void add(int precision, int nx)
    {
        max_nx = std::max(max_nx, nx);
        lo = std::max(lo, lo_smem(precision, nx));
        grey = std::max(grey, grey_smem(nx));
    }
};

}  // namespace trt
