// MDLG binning of two position snapshots (Sec. 2, Eq. n_i summed over the
// lattice sites): standalone entry point mdlg_bin.  The fused variant that
// runs inside the MD step lives in md.cu; both share the device helpers of
// lattice.cuh.
//
// Design: the work is 24 bytes (FP32 offsets) per particle, so the target is
// the memory rate, and GB300's FP64 rate (1/60 of FP32) sets the rule: one
// FP64 operation per particle and axis costs as much as reading the particle.
//   * lattice cells are decided in FP32 where that provably gives the FP64
//     cell (lattice_floor_f32);
//   * the displacement is taken in the cell frame, wrap(c1 - c0) h + (o1 -
//     o0), and its powers are formed as pairs of FP32 values (h split in three
//     parts, error terms by fused multiply-adds): a square is off by at most
//     3 2^-48 of itself, a fourth power by 9 2^-48.  They are summed in three
//     FP32 values by Knuth's two-sum, which catches what every addition rounds
//     off, however many particles a thread takes; each thread's sums become
//     FP64 once at its end.  (With the low part of the fourth moments added
//     plainly an addition's error did not average out: 1e-12 after 220 equal
//     displacements.  Catching it costs 4 us of 96.)  FP64 offsets, displacements within 1 % of half the
//     box (where the nearest image is a choice), below 2^-20 of the cell
//     edge (whose fourth power would leave FP32's range) or not finite go
//     through FP64;
//   * the (2W+1)^2 histogram is privatised per CTA in shared memory, one
//     atomic per particle (the hardware merges equal addresses of a warp);
//   * up to BIN_CLUSTER_MAX particles a single launch of one thread-block
//     cluster does everything and its first CTA adds the others' results
//     through distributed shared memory: no memsets, no scratch, no second
//     kernel.  Above it, a one-wave grid with per-CTA moment partials that a
//     one-block kernel sums with fixed strides and a fixed tree, so results do
//     not depend on scheduling.
// What bounds it now is the instruction rate: more than 317 warp instructions
// per 32 particles (counted before the moments' third terms), issue slots 73 %
// busy, DRAM at a quarter of its rate.
// Measured (6.4M FP32 particles, W = 4): 1016 us per call with FP64 positions,
// 64-bit remainders and an FP64 division per axis, 96 us now, the moments'
// error against 64 bits at most 1.2e-16 on four inputs; 2047 FP64 particles alone 257 ->
// 80 us with the host's part (memsets, allocation and a second kernel gone).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <mutex>

#include "common.cuh"
#include "lattice.cuh"

namespace mdlg {

namespace cg = cooperative_groups;

struct SnapDev {
    const int32_t *cell;
    const void *ox;
    const void *oy;
};

struct BinParams {
    int n, ncell, lx, W;
    CellDiv div;                   // split of the linear cell index
    float hf, invf;                // FP32 lattice cells (lattice_floor_f32)
    float scale;                   // power of two that brings h into [1, 2)
    float h0, h1, h2;              // scale * h in three parts
    float dmin, dmax;              // scaled |displacement| range of the FP32 pairs
    double h, L, dxl;
    double unscale2, unscale4;     // scale^-2, scale^-4
};

// a + b = s + e exactly (Knuth)
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// The moment sums of one thread: pairs (a, b) of FP32 in scaled units, what
// the pairs drop with a sign of its own in c2 / c4, and FP64 sums of the
// displacements that do not go through the pairs.
struct BinSums {
    float a2 = 0.f, b2 = 0.f, c2 = 0.f, a4 = 0.f, b4 = 0.f, c4 = 0.f;
    double d2 = 0.0, d4 = 0.0;
    __device__ __forceinline__ void add64(double e) {
        const double q = e * e;
        d2 += q;
        d4 += q * q;
    }
    __device__ __forceinline__ double m2(const BinParams &P) const {
        return d2 + ((double)a2 + ((double)b2 + (double)c2)) * P.unscale2;
    }
    __device__ __forceinline__ double m4(const BinParams &P) const {
        return d4 + ((double)a4 + ((double)b4 + (double)c4)) * P.unscale4;
    }
};

// The displacement as the difference of FP64 positions, nearest image.
static __device__ __noinline__ double bin_disp64(int c1, double o1, int c0, double o0, double h, double L) {
    return nearest_image(cell_position(c1, h, o1) - cell_position(c0, h, o0), L);
}

// Adds one displacement component, cells c0 -> c1, offsets o0 -> o1.
__device__ __forceinline__ void bin_moments(const BinParams &P, int c0, float o0, int c1, float o1, BinSums &S) {
    int dc = c1 - c0;
    if (dc > P.ncell / 2) dc -= P.ncell;
    if (dc < -(P.ncell / 2)) dc += P.ncell;
    const float c = __fsub_rn(__int_as_float(0x4b400000 + dc), 12582912.0f);   // |dc| < 2^22
    // dc h = p + pe + t + te: exact products of the parts of h; what the pair
    // (x, y) drops is a function of dc alone for most particles, so it does
    // not average out over them and is kept in eps
    const float p = __fmul_rn(c, P.h0), pe = __fmaf_rn(c, P.h0, -p);
    const float t = __fmul_rn(c, P.h1), te = __fmaf_rn(c, P.h2, __fmaf_rn(c, P.h1, -t));
    float d, de, s, se, lo, l1, l2, w;
    two_sum(__fmul_rn(o1, P.scale), -__fmul_rn(o0, P.scale), d, de);
    two_sum(p, d, s, se);
    two_sum(pe, t, w, l1);
    two_sum(__fadd_rn(se, de), w, lo, l2);
    const float eps = __fadd_rn(te, __fadd_rn(l1, l2));
    const float x = __fadd_rn(s, lo), y = __fsub_rn(lo, __fsub_rn(x, s));   // |lo| << |s| or s = 0
    const float ax = fabsf(x);
    if (ax > P.dmin && ax < P.dmax) {
        // (x + y)^2 = q + r + y^2, the square of q + r = u + v + r^2.  The
        // last terms are below the pairs' last bits and positive, so adding
        // them there would drop them every time; they go to c2 and c4.  The
        // low bits of r are those of a square (1 modulo 8 in units of the
        // last place), so what its additions round off has a sign too.
        const float q = __fmul_rn(x, x), x2 = __fadd_rn(x, x);
        const float r = __fmaf_rn(x2, y, __fmaf_rn(x, x, -q));
        const float u = __fmul_rn(q, q), q2 = __fadd_rn(q, q);
        const float v = __fmaf_rn(q2, r, __fmaf_rn(q, q, -u));
        float e, f, k;
        two_sum(S.a2, q, S.a2, e);
        two_sum(e, r, e, f);
        two_sum(S.b2, e, S.b2, k);
        const float z = __fmaf_rn(x2, eps, __fmul_rn(y, y));   // what q + r lacks
        S.c2 = __fadd_rn(S.c2, __fadd_rn(z, __fadd_rn(f, k)));
        two_sum(S.a4, u, S.a4, e);
        two_sum(e, v, e, f);
        two_sum(S.b4, e, S.b4, k);
        S.c4 = __fadd_rn(S.c4, __fadd_rn(__fmaf_rn(q2, z, __fmul_rn(r, r)), __fadd_rn(f, k)));
    } else if (!(x == 0.f && y == 0.f && eps == 0.f)) {
        S.add64(bin_disp64(c1, (double)o1, c0, (double)o0, P.h, P.L));
    }
}

__device__ __forceinline__ void bin_moments(const BinParams &P, int c0, double o0, int c1, double o1, BinSums &S) {
    int dc = c1 - c0;
    if (dc > P.ncell / 2) dc -= P.ncell;
    if (dc < -(P.ncell / 2)) dc += P.ncell;
    double e = __fma_rn((double)dc, P.h, __dsub_rn(o1, o0));
    if (!(fabs(e) < 0.49 * P.L)) e = bin_disp64(c1, o1, c0, o0, P.h, P.L);
    S.add64(e);
}

// Counts one particle and adds its displacement's powers.
template <typename T>
__device__ __forceinline__ void bin_particle(const BinParams &P, int k0, T x0, T y0, int k1, T x1, T y1, int *hist,
                                             unsigned &ovf, BinSums &S) {
    int cx0, cy0, cx1, cy1;
    split_cell(k0, P.ncell, P.div, cx0, cy0);
    split_cell(k1, P.ncell, P.div, cx1, cy1);
    const auto cell = [&](int c, T o) { return lattice_floor_f32<T>(c, o, P.h, P.hf, P.dxl, P.invf, P.lx); };
    const int vx = lattice_shift_floors(cell(cx1, x1) - cell(cx0, x0), P.lx);
    const int vy = lattice_shift_floors(cell(cy1, y1) - cell(cy0, y0), P.lx);
    if (vx >= -P.W && vx <= P.W && vy >= -P.W && vy <= P.W)
        atomicAdd(&hist[(vy + P.W) * (2 * P.W + 1) + vx + P.W], 1);
    else
        ++ovf;
    bin_moments(P, cx0, x0, cx1, x1, S);
    bin_moments(P, cy0, y0, cy1, y1, S);
}

template <typename T> struct BinVec4;
template <> struct BinVec4<float> {
    static __device__ __forceinline__ void load(const float *p, float (&v)[4]) {
        const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    }
};
template <> struct BinVec4<double> {
    static __device__ __forceinline__ void load(const double *p, double (&v)[4]) {
        const double2 q0 = __ldg(reinterpret_cast<const double2 *>(p));
        const double2 q1 = __ldg(reinterpret_cast<const double2 *>(p) + 1);
        v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    }
};

// Grid-stride over groups of four particles (VEC: 16-byte aligned arrays,
// vector loads, all loads of a group before any arithmetic), then the rest
// one per thread.
template <typename T, bool VEC>
__device__ __forceinline__ void bin_loop(const SnapDev &a, const SnapDev &b, const BinParams &P, int *hist,
                                         unsigned &ovf, BinSums &S) {
    const T *ax = static_cast<const T *>(a.ox), *ay = static_cast<const T *>(a.oy);
    const T *bx = static_cast<const T *>(b.ox), *by = static_cast<const T *>(b.oy);
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long ngroup = VEC ? P.n / 4 : 0;
    for (long long g = tid; g < ngroup; g += stride) {
        const int4 q0 = __ldg(reinterpret_cast<const int4 *>(a.cell) + g);
        const int4 q1 = __ldg(reinterpret_cast<const int4 *>(b.cell) + g);
        const int c0[4] = {q0.x, q0.y, q0.z, q0.w}, c1[4] = {q1.x, q1.y, q1.z, q1.w};
        T x0[4], y0[4], x1[4], y1[4];
        BinVec4<T>::load(ax + 4 * g, x0);
        BinVec4<T>::load(ay + 4 * g, y0);
        BinVec4<T>::load(bx + 4 * g, x1);
        BinVec4<T>::load(by + 4 * g, y1);
#pragma unroll
        for (int u = 0; u < 4; ++u) bin_particle<T>(P, c0[u], x0[u], y0[u], c1[u], x1[u], y1[u], hist, ovf, S);
    }
    for (long long j = 4 * ngroup + tid; j < P.n; j += stride)
        bin_particle<T>(P, a.cell[j], ax[j], ay[j], b.cell[j], bx[j], by[j], hist, ovf, S);
}

constexpr int BIN_THREADS = 256;

template <typename T, bool VEC>
__global__ void __launch_bounds__(BIN_THREADS) k_bin_snapshots(SnapDev a, SnapDev b, BinParams P, int *hist,
                                                               unsigned long long *ovf, double *part) {
    extern __shared__ int sh[];
    const int nb = (2 * P.W + 1) * (2 * P.W + 1);
    for (int i = threadIdx.x; i < nb; i += BIN_THREADS) sh[i] = 0;
    __syncthreads();
    BinSums S;
    unsigned my_ovf = 0;
    bin_loop<T, VEC>(a, b, P, sh, my_ovf, S);
    my_ovf = __reduce_add_sync(0xffffffffu, my_ovf);
    if ((threadIdx.x & 31) == 0 && my_ovf) atomicAdd(ovf, (unsigned long long)my_ovf);
    double m2 = S.m2(P), m4 = S.m4(P);
    block_sum2(m2, m4);
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += BIN_THREADS)
        if (sh[i]) atomicAdd(&hist[i], sh[i]);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = m2;
        part[2 * blockIdx.x + 1] = m4;
    }
}

// Small snapshots: one cluster, one launch, up to eight particles per thread
// (a cluster of 2047 FP64 particles takes 7.9 us; the grid path's two small
// kernels alone take 5.4 us before the launches' gaps).
constexpr int BIN_CLUSTER_THREADS = 512;
constexpr int BIN_CLUSTER_CTAS = 8;                    // largest portable cluster
constexpr int BIN_CLUSTER_MAX = 8 * BIN_CLUSTER_CTAS * BIN_CLUSTER_THREADS;

template <typename T>
__global__ void __launch_bounds__(BIN_CLUSTER_THREADS) k_bin_cluster(SnapDev a, SnapDev b, BinParams P, int *hist,
                                                                     long long *ovf, double *mom) {
    extern __shared__ int sh[];
    __shared__ unsigned s_ovf;
    __shared__ double s_m[2];
    const int nb = (2 * P.W + 1) * (2 * P.W + 1);
    for (int i = threadIdx.x; i < nb; i += BIN_CLUSTER_THREADS) sh[i] = 0;
    if (threadIdx.x == 0) s_ovf = 0;
    __syncthreads();
    BinSums S;
    unsigned my_ovf = 0;
    bin_loop<T, false>(a, b, P, sh, my_ovf, S);
    my_ovf = __reduce_add_sync(0xffffffffu, my_ovf);
    if ((threadIdx.x & 31) == 0 && my_ovf) atomicAdd(&s_ovf, my_ovf);
    double m2 = S.m2(P), m4 = S.m4(P);
    block_sum2(m2, m4);
    if (threadIdx.x == 0) {
        s_m[0] = m2;
        s_m[1] = m4;
    }
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();
    if (cl.block_rank() == 0) {
        const int nc = (int)cl.num_blocks();
        for (int i = threadIdx.x; i < nb; i += BIN_CLUSTER_THREADS) {
            int t = 0;
            for (int c = 0; c < nc; ++c) t += *cl.map_shared_rank(&sh[i], c);
            hist[i] = t;
        }
        if (threadIdx.x < 2) {
            double t = 0.0;
            for (int c = 0; c < nc; ++c) t += *cl.map_shared_rank(&s_m[threadIdx.x], c);
            mom[threadIdx.x] = t;
        } else if (threadIdx.x == 32) {
            long long t = 0;
            for (int c = 0; c < nc; ++c) t += *cl.map_shared_rank(&s_ovf, c);
            *ovf = t;
        }
    }
    cl.sync();   // no CTA leaves while the first one reads its shared memory
}

__global__ void k_bin_clear(int *hist, int nb, unsigned long long *ovf) {
    for (int i = threadIdx.x; i < nb; i += blockDim.x) hist[i] = 0;
    if (threadIdx.x == 0) *ovf = 0ull;
}

// Sums the per-CTA moment partials (one CTA, fixed strides and tree).
__global__ void __launch_bounds__(BIN_THREADS) k_sum_partials(const double *part, int nparts, double *mom) {
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nparts; i += BIN_THREADS) {
        a += part[2 * i];
        b += part[2 * i + 1];
    }
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        mom[0] = a;
        mom[1] = b;
    }
}

int bin_check_args(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t lx, int32_t W,
                   const void *hist_out, const void *overflow_out, const void *mom_out) {
    if (!t0 || !t1 || !hist_out || !overflow_out || !mom_out)
        return fail(MD_E_ARG, "mdlg_bin: NULL argument");
    if (n < 0 || n >= (int64_t)1 << 31) return fail(MD_E_ARG, "mdlg_bin: n out of [0, 2^31)");
    if (n > 0 && (!t0->cell || !t0->off_x || !t0->off_y || !t1->cell || !t1->off_x || !t1->off_y))
        return fail(MD_E_ARG, "mdlg_bin: NULL snapshot array");
    if (t0->ncell != t1->ncell || t0->h != t1->h || t0->off_is_f64 != t1->off_is_f64)
        return fail(MD_E_ARG, "mdlg_bin: snapshots differ in ncell, h or offset type");
    if (t0->ncell < 1 || !(t0->h > 0.0)) return fail(MD_E_ARG, "mdlg_bin: bad ncell or h");
    if ((int64_t)t0->ncell * t0->ncell >= (int64_t)1 << 31)
        return fail(MD_E_ARG, "mdlg_bin: ncell^2 must fit in int32");
    if (lx < 1) return fail(MD_E_ARG, "mdlg_bin: lx must be >= 1");
    if (W < 0 || W > MD_MAX_W) return fail(MD_E_ARG, "mdlg_bin: W out of [0,%d]", MD_MAX_W);
    return MD_OK;
}

template <typename T>
const void *bin_kernel(bool vec) {
    return vec ? (const void *)k_bin_snapshots<T, true> : (const void *)k_bin_snapshots<T, false>;
}

BinParams bin_params(const md_snapshot *t0, int64_t n, int32_t lx, int32_t W) {
    BinParams P;
    P.n = (int)n;
    P.ncell = t0->ncell;
    P.lx = lx;
    P.W = W;
    P.h = t0->h;
    P.L = (double)t0->ncell * t0->h;
    P.dxl = P.L / (double)lx;
    P.div = cell_div(t0->ncell);
    P.hf = (float)t0->h;
    // lattices so fine that a difference of floors could leave 32 bits: the
    // reduced FP64 cells throughout
    P.invf = lx < 1 << 30 ? (float)(1.0 / P.dxl) : NAN;
    int e = 0;
    std::frexp(t0->h, &e);
    P.scale = std::ldexp(1.0f, 1 - e);
    const double hs = std::ldexp(t0->h, 1 - e);
    P.h0 = (float)hs;
    P.h1 = (float)(hs - (double)P.h0);
    P.h2 = (float)(hs - (double)P.h0 - (double)P.h1);
    P.dmin = 0x1p-20f;
    P.dmax = (float)(0.49 * (double)t0->ncell * hs);
    // a cell edge so far from 1 that scaling an offset could leave FP32's
    // range: a NaN scale sends every displacement through FP64
    if (e < -60 || e > 60) P.scale = NAN;
    P.unscale2 = std::ldexp(1.0, 2 * (e - 1));
    P.unscale4 = std::ldexp(1.0, 4 * (e - 1));
    return P;
}

bool bin_vec(const md_snapshot *t0, const md_snapshot *t1) {
    const void *v[6] = {t0->cell, t0->off_x, t0->off_y, t1->cell, t1->off_x, t1->off_y};
    for (const void *p : v)
        if ((uintptr_t)p & 15u) return false;
    return true;
}

// Enqueues the binning kernels of the grid path with the moment partials in
// `part` (>= 2*grid doubles of device memory).
int bin_launch(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t lx, int32_t W,
               int32_t *hist_out, int64_t *overflow_out, double *mom_out, double *part, int grid,
               cudaStream_t st) {
    const int nb = (2 * W + 1) * (2 * W + 1);
    SnapDev a{t0->cell, t0->off_x, t0->off_y};
    SnapDev b{t1->cell, t1->off_x, t1->off_y};
    BinParams P = bin_params(t0, n, lx, W);
    k_bin_clear<<<1, 512, 0, st>>>(hist_out, nb, (unsigned long long *)overflow_out);
    MD_CUDA_TRY(cudaGetLastError());
    const bool vec = bin_vec(t0, t1);
    void *args[] = {&a, &b, &P, &hist_out, &overflow_out, &part};
    MD_CUDA_TRY(cudaLaunchKernel(t0->off_is_f64 ? bin_kernel<double>(vec) : bin_kernel<float>(vec), dim3(grid),
                                 dim3(BIN_THREADS), args, nb * sizeof(int), st));
    k_sum_partials<<<1, BIN_THREADS, 0, st>>>(part, grid, mom_out);
    MD_CUDA_TRY(cudaGetLastError());
    return MD_OK;
}

// The cluster path: as many CTAs (1, 2, 4 or 8) as give each thread one
// particle, at most eight CTAs.
int bin_launch_cluster(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t lx, int32_t W,
                       int32_t *hist_out, int64_t *overflow_out, double *mom_out, cudaStream_t st) {
    SnapDev a{t0->cell, t0->off_x, t0->off_y};
    SnapDev b{t1->cell, t1->off_x, t1->off_y};
    const BinParams P = bin_params(t0, n, lx, W);
    int ctas = 1;
    while (ctas < BIN_CLUSTER_CTAS && (int64_t)ctas * BIN_CLUSTER_THREADS < n) ctas *= 2;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(BIN_CLUSTER_THREADS);
    cfg.dynamicSmemBytes = (2 * W + 1) * (2 * W + 1) * sizeof(int);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MD_CUDA_TRY(cudaLaunchKernelEx(&cfg, t0->off_is_f64 ? k_bin_cluster<double> : k_bin_cluster<float>, a, b, P,
                                   (int *)hist_out, (long long *)overflow_out, mom_out));
    return MD_OK;
}

// Moment partials of mdlg_bin_noalloc, for callers that cannot allocate
// device memory while they run (their memory belongs to a framework's
// caching allocator or a fixed budget, or their loop must not stall on
// allocator calls): a fixed device array instead of a per-call allocation
// (2 doubles per CTA, room for BIN_SCRATCH_CTAS CTAs, 32 KiB, held by every
// GPU that loads the library until the process exits).  Every CTA of a
// launch overwrites its own two entries and the reduction reads only the
// first `grid`, so it never needs clearing.  Host code must not pass the
// array's name to a kernel (on the host it only stands in for the symbol);
// it passes the device address that cudaGetSymbolAddress returns.
constexpr int BIN_SCRATCH_CTAS = 2048;
static __device__ __align__(256) double g_bin_scratch[2 * BIN_SCRATCH_CTAS];

// CTAs of one binning launch: one wave of resident CTAs of the instantiation
// (at most 8 per SM), fewer when there is less work (SM count and occupancy
// of the current device: a process may bin on GPUs of different sizes).
int bin_grid(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t W) {
    const bool vec = bin_vec(t0, t1);
    int dev = 0, nsm = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm <= 0)
        nsm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm,
                                                      t0->off_is_f64 ? bin_kernel<double>(vec) : bin_kernel<float>(vec),
                                                      BIN_THREADS, (2 * W + 1) * (2 * W + 1) * sizeof(int)) !=
            cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int64_t work = vec ? (n + 3) / 4 : n;
    int64_t want = (work + BIN_THREADS - 1) / BIN_THREADS;
    const int64_t cap = (int64_t)nsm * std::min(per_sm, 8);
    if (want > cap) want = cap;
    if (want < 1) want = 1;
    return (int)want;
}

// Device address of g_bin_scratch on the current device.  Looked up with
// that device current on the first call made on it, and looked up again
// when the device's context has changed since (after a cudaDeviceReset the
// module is loaded afresh and the array may live elsewhere).  The table is
// guarded by a mutex, so host threads may call concurrently.
using CtxGetCurrentFn = int (*)(void **);
constexpr int BIN_MAX_DEV = 64;
struct ScratchSlot {
    const void *ctx = nullptr;
    double *ptr = nullptr;
};
std::mutex g_scratch_mu;
ScratchSlot g_scratch[BIN_MAX_DEV];

CtxGetCurrentFn ctx_get_current() {
    static CtxGetCurrentFn fn = [] {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<CtxGetCurrentFn>(p);
    }();
    return fn;
}

int scratch_address(double **out) {
    int dev = 0;
    MD_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= BIN_MAX_DEV)
        return fail(MD_E_LIMIT, "mdlg_bin_noalloc: device %d >= %d", dev, BIN_MAX_DEV);
    const CtxGetCurrentFn get = ctx_get_current();
    auto current = [get]() {
        void *c = nullptr;
        if (!get || get(&c) != 0) c = nullptr;
        return c;
    };
    // no current context yet on this thread (or no way to ask): look up,
    // which also makes the device's primary context current
    const void *ctx = current();
    std::lock_guard<std::mutex> lk(g_scratch_mu);
    ScratchSlot &sl = g_scratch[dev];
    if (!sl.ptr || !ctx || sl.ctx != ctx) {
        double *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress((void **)&p, g_bin_scratch);
        if (e != cudaSuccess)
            return fail(MD_E_CUDA, "mdlg_bin_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
        sl.ptr = p;
        sl.ctx = current();
    }
    *out = sl.ptr;
    return MD_OK;
}

}  // namespace mdlg

using namespace mdlg;

extern "C" int mdlg_bin(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t lx,
                        int32_t W, int32_t *hist_out, int64_t *overflow_out, double *mom_out,
                        void *stream) {
    mdlg::Range range_("mdlg_bin");
    int rc = bin_check_args(t0, t1, n, lx, W, hist_out, overflow_out, mom_out);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    if (n <= BIN_CLUSTER_MAX) return bin_launch_cluster(t0, t1, n, lx, W, hist_out, overflow_out, mom_out, st);
    const int grid = bin_grid(t0, t1, n, W);
    double *part = nullptr;
    MD_CUDA_TRY(scratch_alloc((void **)&part, 2 * sizeof(double) * grid, st));
    rc = bin_launch(t0, t1, n, lx, W, hist_out, overflow_out, mom_out, part, grid, st);
    cudaError_t e = scratch_free(part, st);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(MD_E_CUDA, "mdlg_bin: cudaFreeAsync: %s", cudaGetErrorString(e));
    return MD_OK;
}

// Same computation as mdlg_bin with the partials in g_bin_scratch.  The
// array's device address is looked up on the first call on each device
// (with that device current), and again after a cudaDeviceReset, so that
// first call should come before any stream capture; nothing is allocated.
// Calls that overlap on the GPU share the array and race.
extern "C" int mdlg_bin_noalloc(const md_snapshot *t0, const md_snapshot *t1, int64_t n, int32_t lx,
                                int32_t W, int32_t *hist_out, int64_t *overflow_out, double *mom_out,
                                void *stream) {
    mdlg::Range range_("mdlg_bin_noalloc");
    int rc = bin_check_args(t0, t1, n, lx, W, hist_out, overflow_out, mom_out);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const int grid = bin_grid(t0, t1, n, W);
    if (grid > BIN_SCRATCH_CTAS)
        return fail(MD_E_LIMIT, "mdlg_bin_noalloc: %d CTAs exceed the scratch capacity of %d", grid,
                    BIN_SCRATCH_CTAS);
    double *scratch = nullptr;
    rc = scratch_address(&scratch);
    if (rc) return rc;
    if (n <= BIN_CLUSTER_MAX) return bin_launch_cluster(t0, t1, n, lx, W, hist_out, overflow_out, mom_out, st);
    return bin_launch(t0, t1, n, lx, W, hist_out, overflow_out, mom_out, scratch, grid, st);
}
