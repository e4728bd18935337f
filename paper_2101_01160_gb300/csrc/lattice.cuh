// Device helpers of the MDLG lattice mapping (Sec. 2).  The integer results
// (lattice cell, displacement class) depend on FP64 arithmetic, so each
// operation is an explicitly rounded intrinsic: no contraction into FMA, the
// same rounding as a plain IEEE evaluation of x = cx*h + off and
// floor(x / dxl) on the host.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace mdlg {

// Position encoded as (cell coordinate, offset): x = c*h + off.
__device__ __forceinline__ double cell_position(int c, double h, double off) {
    return __dadd_rn(__dmul_rn((double)c, h), off);
}

// Lattice cell of coordinate x: floor(x / dxl) reduced modulo lx (a point on
// a cell boundary belongs to the upper cell).
__device__ __forceinline__ long long lattice_cell(double x, double dxl, int lx) {
    long long l = (long long)floor(__ddiv_rn(x, dxl));
    l %= lx;
    if (l < 0) l += lx;
    return l;
}

// The lattice cell of the position encoded as (cell coordinate c, offset
// off), floor(RN(RN(c*h + off) / dxl)) mod lx as lattice_cell computes it,
// decided in FP32 wherever FP32 provably gives the same cell.  With a =
// RN32(c * hf), hf = RN32(h), invf = RN32(1/dxl):
//     q = RN32(RN32(a + off) * invf),   S = RN32(RN32(|a| + |off|) * invf),
// the distance of q from the exact quotient (c*h + off)/dxl is below
// S 2^-21 (a: two roundings of c*h, the sum one, the offset one if it is
// FP64, the product two -- each at most 2^-24 relative to |a| + |off|), and
// the FP64 reference lies within a few 2^-53 relative of the same quotient.
// So when q is more than S 2^-20 from the nearest integer, floor(q) is the
// cell; otherwise (points on or within about S 1e-6 of a lattice line) the
// FP64 evaluation of lattice_cell decides.  Bit-identical to lattice_cell
// for every finite encoded position; in the common case a few FP32 and
// 32-bit integer operations replace the FP64 ones and the 64-bit modulo
// (GB300's FP64 rate is a small fraction of its FP32 rate).  lx < 2^22.
// The FP64 evaluation, out of line: it runs only near lattice lines, and
// keeping it out of the unrolled callers keeps their code small.
static __device__ __noinline__ int lattice_cell_slow(int c, double off, double h, double dxl, int lx) {
    return (int)lattice_cell(cell_position(c, h, off), dxl, lx);
}

// (float)c for 0 <= c < 2^23, from the float bits of 2^23 + c: two ordinary
// operations in place of a conversion (conversions, like rint and floor, run
// on the special-function pipe at a quarter of the rate).
__device__ __forceinline__ float small_int_to_float(int c) {
    return __fsub_rn(__int_as_float(0x4b000000 | c), 8388608.0f);
}

// The decision of lattice_cell_f32 without the reduction modulo lx: the
// quotient's floor where FP32 decides it, else the FP64 cell (already
// reduced; callers reduce either).  0 <= c < 2^23.  Adding 1.5 * 2^23 rounds
// |q| < 2^22 to the nearest integer in its low bits.
template <typename T>
__device__ __forceinline__ int lattice_floor_f32(int c, T off, double h, float hf, double dxl, float invf,
                                                 int lx) {
    const float a = __fmul_rn(small_int_to_float(c), hf);
    const float o = (float)off;
    const float q = __fmul_rn(__fadd_rn(a, o), invf);
    const float S = __fmul_rn(__fadd_rn(fabsf(a), fabsf(o)), invf);
    const float big = __fadd_rn(q, 12582912.0f);
    const float d = __fsub_rn(q, __fsub_rn(big, 12582912.0f));   // q - rint(q), exact
    if (S < 0x1p22f && fabsf(d) > __fmul_rn(S, 0x1p-20f))
        return __float_as_int(big) - 0x4b400000 - (d < 0.0f ? 1 : 0);
    return lattice_cell_slow(c, (double)off, h, dxl, lx);
}

// l modulo lx: positions within a box edge of the box need one wrap; others
// the general reduction.
__device__ __forceinline__ int lattice_wrap(int l, int lx) {
    if (l < 0) l += lx;
    else if (l >= lx) l -= lx;
    if (l < 0 || l >= lx) {
        l %= lx;
        if (l < 0) l += lx;
    }
    return l;
}

template <typename T>
__device__ __forceinline__ int lattice_cell_f32(int c, T off, double h, float hf, double dxl, float invf,
                                                int lx) {
    return lattice_wrap(lattice_floor_f32<T>(c, off, h, hf, dxl, invf, lx), lx);
}

// Division of 0 <= c < 2^31 by an invariant ncell >= 1 as one high product
// and a shift (Granlund and Montgomery 1994): with s = ceil(log2 ncell) and
// m = floor(2^(31+s) / ncell) + 1 < 2^32 + 1, c m / 2^(31+s) exceeds c /
// ncell by less than c / 2^(31+s) < 1 / ncell, so the floors agree.
struct CellDiv {
    uint32_t mul;
    int32_t shift;     // of the high 32 bits of c * mul; -1: ncell = 1
};
inline CellDiv cell_div(int ncell) {
    int s = 0;
    while ((1ll << s) < ncell) ++s;
    if (s == 0) return CellDiv{0u, -1};
    return CellDiv{(uint32_t)((1ull << (31 + s)) / (uint64_t)ncell + 1ull), s - 1};
}

// Splits a linear cell index c = cy * ncell + cx, 0 <= c < 2^31.
__device__ __forceinline__ void split_cell(int c, int ncell, CellDiv D, int &cx, int &cy) {
    const int y = D.shift < 0 ? c : (int)(__umulhi((uint32_t)c, D.mul) >> D.shift);
    cx = c - y * ncell;
    cy = y;
}

// Nearest periodic image of a lattice displacement d in (-lx, lx) (two
// cells of [0, lx)), in (-lx/2, lx/2]: lattice_shift without the modulo.
__device__ __forceinline__ int lattice_shift_near(int d, int lx) {
    if (d < 0) d += lx;
    if (d > lx / 2) d -= lx;
    return d;
}

// Lattice displacement reduced to the nearest periodic image, in
// (-lx/2, lx/2].
static __device__ __noinline__ int lattice_shift(int d, int lx) {
    d %= lx;
    if (d < 0) d += lx;
    if (d > lx / 2) d -= lx;
    return d;
}

// Nearest image of the difference d of two lattice_floor_f32 values: one wrap
// for positions within a box edge of the box, the general reduction else.
__device__ __forceinline__ int lattice_shift_floors(int d, int lx) {
    const int half = lx / 2, low = half + 1 - lx;   // (-lx/2, lx/2] as integers
    if (d > half) d -= lx;
    if (d < low) d += lx;
    return d > half || d < low ? lattice_shift(d, lx) : d;
}

__device__ __forceinline__ double nearest_image(double d, double L) {
    return __dsub_rn(d, __dmul_rn(L, rint(__ddiv_rn(d, L))));
}

// Adds one count to sh[bin] for every lane with bin >= 0; lanes holding the
// same bin are merged into one shared-memory atomic.  All 32 lanes of the
// warp must call it.
__device__ __forceinline__ void warp_hist_add(int *sh, int bin, int lane) {
    const unsigned m = __match_any_sync(0xffffffffu, bin);
    if (bin >= 0 && lane == __ffs(m) - 1) atomicAdd(&sh[bin], __popc(m));
}

// Sum of two doubles over the CTA; the result is valid in thread 0.
// Fixed reduction tree (warp shuffles, then warp 0), so the result is the
// same on every run.
__device__ __forceinline__ void block_sum2(double &a, double &b) {
    __shared__ double s_a[32], s_b[32];
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();
    if (lane == 0) {
        s_a[w] = a;
        s_b[w] = b;
    }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = lane < nw ? s_a[lane] : 0.0;
        b = lane < nw ? s_b[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
        }
    }
}

}  // namespace mdlg
