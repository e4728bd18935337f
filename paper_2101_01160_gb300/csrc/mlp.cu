// The f_eq surrogate (a project addition, not in the paper): an MLP mapping
// the state point (phi, T, Delta t_LG, Delta x) to the probabilities of the
// (2W+1)^2 = 81 displacement classes, trained on histograms measured by the
// MD of this library.  Hidden layers are BF16 GEMMs on the tensor cores
// (tcgen05.mma, FP32 accumulation in TMEM).  A training step is three
// launches: the forward and backward chain of each 128-row tile on one
// thread-block cluster (k_train_chain), the weight gradients' partial sums
// (k_train_grads), and their sum with the Adam update (k_train_update).
//
// Model: x_f = (x - shift)/scale; h_1 = silu(W_1 x_f + b_1) (CUDA cores);
// h_l = silu(W_l h_{l-1} + b_l), l = 2..L-1 (tensor cores); logits =
// W_L h_{L-1} + b_L (tensor cores, classes padded to 128 with zero rows);
// p = softmax(logits[0..81)); loss = mean D_KL(t || p).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "umma.cuh"

namespace mdlg {

using bf16 = __nv_bfloat16;

constexpr int GBM = 128;   // GEMM tile rows (TMEM lanes)
constexpr int GBK = 64;    // K per pipeline stage
constexpr int GRAD_MAX_SPLIT = 64;   // splits of a weight gradient over the batch
constexpr int GRAD_ROWS = 128;       // rows of one partial bias or first-layer gradient
constexpr uint64_t GEMM_WAIT_NS = 2000000000ull;

struct GemmArgs {
    const bf16 *A;      // [M][K] row-major (K contiguous)
    const bf16 *B;      // [N][K] row-major
    int lda, ldb, M, N, K;
    float *C;           // [M][ldc] FP32
    int ldc;
    int *status;
    uint64_t wait_ns;   // limit of every mbarrier wait (0: GEMM_WAIT_NS)
    int dbg_skip_commit;   // bf16_gemm_selftest: CTA 0 does not signal stage dbg_skip_commit - 1 (0: never)
};

__device__ __forceinline__ float silu(float z) { return z / (1.0f + __expf(-z)); }
__device__ __forceinline__ float silu_grad(float z) {
    const float s = 1.0f / (1.0f + __expf(-z));
    return s * (1.0f + z * (1.0f - s));
}

__device__ __forceinline__ void cpa16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(umma::saddr(dst)), "l"(src) : "memory");
}

// Byte offset of element (row r, k) of a K-major tile of GBK columns in the
// no-swizzle core-matrix layout: 8x8 blocks of 128 bytes, blocks along K
// adjacent (LBO = 128 B), 8-row groups GBK/8 blocks apart (SBO = 1024 B).
__device__ __forceinline__ int tile_off(int r, int k8) { return (r >> 3) * 1024 + k8 * 128 + (r & 7) * 16; }

// C = A * B^T on the tensor cores; one CTA computes a 128 x N tile (N <= 256,
// a multiple of 16) with the accumulator in N TMEM columns.  K is consumed
// in stages of 64: the loads of stage k+1 overlap the MMAs of stage k.
__global__ void __launch_bounds__(128) k_gemm(GemmArgs g) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = g.N;
    const int a_bytes = GBM * GBK * 2, b_bytes = N * GBK * 2;
    unsigned char *st0 = sm, *st1 = sm + a_bytes + b_bytes;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sm + 2 * (a_bytes + b_bytes));
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(mbar + 3);   // mbar[2]: drain after a failed wait
    __shared__ int s_ok;
    const uint32_t ncols = N <= 32 ? 32u : (N <= 64 ? 64u : (N <= 128 ? 128u : 256u));
    const uint64_t wait_ns = g.wait_ns ? g.wait_ns : GEMM_WAIT_NS;
    if (warp == 0) umma::tmem_alloc(s_tmem, ncols);
    if (tid == 0) {
        umma::mbar_init(&mbar[0], 1);
        umma::mbar_init(&mbar[1], 1);
        umma::mbar_init(&mbar[2], 1);
        umma::mbar_fence_init();
        s_ok = 1;
    }
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    const uint32_t tmem = *s_tmem;
    const int m0 = blockIdx.x * GBM;
    const int nk = g.K / GBK;
    const int n0 = (int)blockIdx.y * N;    // first output column of this CTA (N split)
    const uint32_t idesc = umma::idesc_bf16(GBM, N);
    for (int kt = 0; kt < nk; ++kt) {
        const int s = kt & 1;
        unsigned char *sa = s ? st1 : st0;
        unsigned char *sb = sa + a_bytes;
        if (kt >= 2 && !umma::mbar_wait(&mbar[s], ((kt - 2) >> 1) & 1, wait_ns)) s_ok = 0;
        __syncthreads();
        if (!s_ok) break;
        for (int c = tid; c < GBM * 8; c += 128) {
            const int r = c >> 3, k8 = c & 7;
            cpa16(sa + tile_off(r, k8), g.A + (size_t)(m0 + r) * g.lda + kt * GBK + k8 * 8);
        }
        for (int c = tid; c < N * 8; c += 128) {
            const int r = c >> 3, k8 = c & 7;
            cpa16(sb + tile_off(r, k8), g.B + (size_t)(n0 + r) * g.ldb + kt * GBK + k8 * 8);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        umma::fence_proxy_smem();
        __syncthreads();
        if (tid == 0) {
            umma::fence_after();
            const uint32_t a0 = umma::saddr(sa), b0 = umma::saddr(sb);
#pragma unroll
            for (int k4 = 0; k4 < GBK / 16; ++k4)
                umma::mma(tmem, umma::desc(a0 + k4 * 256, 128, 1024), umma::desc(b0 + k4 * 256, 128, 1024),
                          idesc, (kt | k4) ? 1u : 0u);
            // the self-test withholds one signal so that a later wait runs out
            if (!(g.dbg_skip_commit == kt + 1 && blockIdx.x == 0)) umma::commit(&mbar[s]);
        }
    }
    if (s_ok) {
        const int last = nk - 1;
        if (!umma::mbar_wait(&mbar[last & 1], (last >> 1) & 1, wait_ns)) s_ok = 0;
    }
    if (!s_ok && tid == 0) {
        // a wait gave up: the MMAs this CTA issued may still run; wait (with a
        // limit) until they are done before their TMEM is freed
        umma::commit(&mbar[2]);
        umma::mbar_wait(&mbar[2], 0, wait_ns);
    }
    __syncthreads();
    umma::fence_after();
    if (s_ok) {
        const int row = m0 + warp * 32 + lane;
        for (int cl = 0; cl < N; cl += 16) {
            float v[16];
            umma::ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cl, v);
            float4 *dst = reinterpret_cast<float4 *>(g.C + (size_t)row * g.ldc + n0 + cl);
#pragma unroll
            for (int q = 0; q < 4; ++q) dst[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    } else if (tid == 0) {
        atomicOr(g.status, 1);
    }
    umma::fence_before();
    __syncthreads();
    if (warp == 0) umma::tmem_free(tmem, ncols);
}

size_t gemm_smem(int N) { return 2 * (size_t)(GBM * GBK * 2 + N * GBK * 2) + 32; }

// A GEMM with fewer 128-row tiles than the device has SMs is split over N
// into two column blocks of N/2 (grid.y), each CTA with its own accumulator;
// the arithmetic of every output is the same.
int gemm_launch(const GemmArgs &g, cudaStream_t st) {
    if (g.M % GBM || g.K % GBK || g.N % 16 || g.N < 16 || g.N > 256 || g.lda % 8 || g.ldb % 8)
        return fail(MD_E_ARG, "gemm: M %% 128, K %% 64, N %% 16 in [16,256], lda/ldb %% 8 required");
    int dev = 0, nsm = 0;
    MD_CUDA_TRY(cudaGetDevice(&dev));
    MD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const int nsplit = (g.N % 32 == 0 && g.M / GBM < nsm) ? 2 : 1;
    GemmArgs gg = g;
    gg.N = g.N / nsplit;
    const size_t smem = gemm_smem(gg.N);
    MD_CUDA_TRY(cudaFuncSetAttribute(k_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_gemm<<<dim3(g.M / GBM, nsplit), 128, smem, st>>>(gg);
    MD_CUDA_TRY(cudaGetLastError());
    return MD_OK;
}

// ---------------------------------------------------------------- fused inference
// Whole forward pass in one persistent, warp-specialised kernel over 128-row
// tiles, two tiles in flight per CTA ("slots") so that the CUDA-core
// epilogue of one slot overlaps the tensor-core MMAs of the other.
//   warp 0 lane 0  producer: streams weight chunks, pre-packed in global
//                  memory in the exact shared-memory layout, with one bulk
//                  copy (TMA) each into a ring of F_STAGES buffers;
//   warp 1         MMA issuer: per (tile pair, layer, slot) waits for the
//                  slot's activations, issues tcgen05.mma into the slot's
//                  128 x 256 FP32 accumulator in TMEM, commits;
//   warps 2..17    epilogue, 8 warps per slot: stage the inputs, then per
//                  layer TMEM -> bias + SiLU -> BF16 activations written
//                  back over the slot's tile, or after the last layer a
//                  softmax staged in shared memory and stored coalesced.
// Layer 1 (4 inputs) is one K = 16 MMA on split operands: with
// x = x_hi + x_lo, W = W_hi + W_lo and b = b_hi + b_lo (BF16 parts), the A
// row holds (x_hi, x_lo, x_hi, 1, 1, 0, 0) and the B row (W_hi, W_hi, W_lo,
// b_hi, b_lo, 0, 0), so the FP32 accumulator receives
// x_hi W_hi + x_lo W_hi + x_hi W_lo + b, the affine map up to the x_lo W_lo
// term (relative ~2^-16).  The other layers add their bias the same way: a
// first K = 16 MMA of a row of ones (one 8 x 16 block read with a zero
// row-group stride) with (b_hi, b_lo, 0, ...) initialises the accumulator,
// so the epilogue reads finished pre-activations from TMEM.
// A warp may read only the TMEM lanes 32 (warp mod 4) .. +31, so epilogue
// warp w serves rows 32 (w mod 4) + lane and one half of the columns.
// What bounds it: each slot alternates between its MMAs (about 2,500 clocks
// per hidden layer) and its epilogue (2,350: the SFU), so two slots keep either
// unit a little over half busy.  Time per 1,048,576 queries (81 classes): 397
// us.  It was 490 while one lane of a divergent branch issued the MMAs: 650
// clocks passed between a layer's first two chunks and the issuer, not the
// tensor core, was the bound (with 3/4 of the MMAs left out it still took 437
// us).  The issuing warp now runs in uniform control flow and elects the lane.
// Ring stages of 6 x 16 KB: 430 us; 4 x 24 KB as 3 x 32 KB; a CTA pair per 256
// rows (cta_group::2, half the weight traffic) needs an exchange between the
// CTAs per chunk and layer and took 748 us with the old issuer.
// Every wait is bounded; a wait that gives up sets the status flag and the
// roles wind down (uniformly within a slot) instead of hanging.
constexpr int FK = 64;                     // features per weight chunk (training)
constexpr int F_STAGES = 3;
constexpr int F_SBO_A = 256 / 8 * 128;     // 8-row groups of the 256-wide activation tile
constexpr int F_SBO_B = FK / 8 * 128;      // 8-row groups of a weight chunk (training)
constexpr int F_SBO_IN = 16 / 8 * 128;     // 8-row groups of the staged K = 16 input rows
constexpr int F_CHUNK_BYTES = 32768;
constexpr int F_SLICES = 1 + 256 / 16;     // of a layer's operand: the bias, then the weights
constexpr int F_MAXL = 15;
constexpr int F_EPI_WARPS = 8;             // per slot
constexpr int F_THREADS = (2 + 2 * F_EPI_WARPS) * 32;
constexpr int F_ACT_BYTES = 128 * 256 * 2;
constexpr int F_RED_OFF = 60 * 1024;       // softmax partials inside a slot's tile
constexpr int F_IN_OFF = 56 * 1024;        // the next tile's inputs inside a slot's tile
constexpr int MLP_MAX_CLASSES = 112;       // FP32 stage rows must end below them

struct FusedArgs {
    const float *X;
    long long M;
    float *P;
    int ncls;
    float4 shift, scale;
    const bf16 *Wp[F_MAXL + 1];    // packed operand of every layer (layer 0: split K = 16 with bias)
    int nt;                        // layers; the last one is the output
    int p_aligned;                 // P 16-byte aligned: output tiles by bulk copy
    int *status;
};

__device__ __forceinline__ int act_off(int r, int k) {
    return (r >> 3) * F_SBO_A + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

// silu(z) = z sigmoid(z) = h + h tanh(h), h = z / 2: one special-function
// operation (tanh.approx, relative error about 2^-11, below the BF16 rounding
// of the stored activation) and one FMA.  The hidden layers' packed weights
// and biases are scaled by 1/2 (exact: a power of two), so the accumulator
// already holds h, bit for bit the half of the unscaled pre-activation.
__device__ __forceinline__ float silu_of_half(float h) {
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(h));
    return fmaf(h, t, h);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

// A layer's packed operand is a run of K = 16 slices of N x 16 (layer 0: one;
// the others: the bias, then 16 of the weights), each [K / 8][N][8]: core
// matrices of 8 rows follow one another along N, so that any run of slices is
// contiguous.  A ring chunk is as many slices as fit a stage.
__device__ __forceinline__ int layer_slices(int l) { return l == 0 ? 1 : F_SLICES; }
__device__ __forceinline__ int chunk_slices(int N) { return F_CHUNK_BYTES / (N * 32); }
__device__ __forceinline__ int slice_off(int n, int k, int N) { return ((k >> 3) * N + n) * 8 + (k & 7); }

__global__ void __launch_bounds__(F_THREADS, 1) k_mlp_fused(FusedArgs a) {
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *ring = sm + 2 * F_ACT_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(ring + F_STAGES * F_CHUNK_BYTES);
    uint64_t *empty = full + F_STAGES;
    uint64_t *accf = empty + F_STAGES;     // per slot: accumulator complete
    uint64_t *actr = accf + 2;             // per slot: activations written, TMEM read
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(actr + 2);
    unsigned char *ones = reinterpret_cast<unsigned char *>(s_tmem + 4);   // 8 x 16 BF16 block
    // (warp index by a shuffle: known to be uniform, so is the issuer's control flow)
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    if (warp == 1) umma::tmem_alloc(s_tmem, 512);
    if (tid < 128) {
        // BF16 element e of the block is (r, k) = ((e % 64) / 8, 8 (e / 64) + e % 8)
        const int k = (tid >> 6) * 8 + (tid & 7);
        reinterpret_cast<bf16 *>(ones)[tid] = __float2bfloat16_rn(k < 2 ? 1.f : 0.f);
    }
    umma::fence_proxy_smem();
    if (tid == 0) {
        for (int i = 0; i < F_STAGES; ++i) {
            umma::mbar_init(&full[i], 1);
            umma::mbar_init(&empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            umma::mbar_init(&accf[i], 1);
            umma::mbar_init(&actr[i], 32 * F_EPI_WARPS);
        }
        umma::mbar_fence_init();
    }
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    const uint32_t tmem = *s_tmem;
    const long long ntiles = (a.M + 127) / 128;
    const long long my_tiles = ntiles > blockIdx.x ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
    const long long npairs = (my_tiles + 1) / 2;
    const int nt = a.nt;
    bool bad = false;

    if (warp == 0) {
        // ------------------------------------------------ producer
        if (lane == 0) {
            int st = 0;
            uint32_t ph = 0;          // phase of the ring pass that stage st is in
            long long c = 0;          // chunks issued
            for (long long p = 0; p < npairs && !bad; ++p)
                for (int l = 0; l < nt && !bad; ++l)
                    for (int s = 0; s < 2 && !bad; ++s) {
                        if (2 * p + s >= my_tiles) continue;
                        const int N = l == nt - 1 ? 128 : 256, ns = layer_slices(l), cs = chunk_slices(N);
                        for (int j = 0; j < ns; j += cs, ++c) {
                            const uint32_t bytes = (uint32_t)(N * 32 * min(cs, ns - j));
                            const bf16 *srcp = a.Wp[l] + (size_t)j * N * 16;
                            // from the second pass on, wait until the MMAs of
                            // the previous pass have released the stage
                            if (c >= F_STAGES && !umma::mbar_wait(&empty[st], ph ^ 1u, GEMM_WAIT_NS)) {
                                bad = true;
                                break;
                            }
                            umma::mbar_expect_tx(&full[st], bytes);
                            umma::bulk_g2s(ring + st * F_CHUNK_BYTES, srcp, bytes, &full[st]);
                            if (++st == F_STAGES) {
                                st = 0;
                                ph ^= 1u;
                            }
                        }
                    }
            // every copy issued must have landed before the CTA exits: the
            // last min(c, F_STAGES) chunks, walking the ring backwards
            for (long long i = 0; i < c && i < F_STAGES; ++i) {
                if (--st < 0) {
                    st = F_STAGES - 1;
                    ph ^= 1u;
                }
                if (!umma::mbar_wait(&full[st], ph, GEMM_WAIT_NS)) bad = true;
            }
            if (bad) atomicOr(a.status, 1);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        // the whole warp runs the loop, one elected lane issues
        int st = 0;
        uint32_t ph = 0;
        long long c = 0;          // chunks consumed
        int last_st = 0;
        uint32_t last_ph = 0;
        const uint64_t ones_desc = umma::desc(umma::saddr(ones), 128, 0);   // every row group: the same 8 rows
        uint32_t kpar[2] = {0u, 0u};   // per slot: parity of the next actr phase
        const auto layer = [&](auto n_, auto ns_, int s, uint64_t first) {   // operand rows, slices; A of slice 0
            constexpr int N = decltype(n_)::value, NS = decltype(ns_)::value, CS = F_CHUNK_BYTES / (N * 32);
            const uint32_t idesc = umma::idesc_bf16(128, N);
            const uint64_t act_desc = umma::desc(umma::saddr(sm + s * F_ACT_BYTES), 128, F_SBO_A);
            const uint64_t ring_desc = umma::desc(umma::saddr(ring), N * 16, 128);
            const uint32_t d = tmem + (uint32_t)(s * 256);
            for (int j = 0; j < NS; j += CS, ++c) {
                if (__any_sync(0xffffffffu, !umma::mbar_wait(&full[st], ph, GEMM_WAIT_NS))) return false;
                umma::fence_after();
                const uint64_t bdesc = ring_desc + (uint64_t)((st * F_CHUNK_BYTES) >> 4);
                const uint64_t adesc = act_desc + (uint64_t)(j * 16);
                if (umma::elect_one()) {
#pragma unroll
                    for (int q = 0; q < CS; ++q)
                        if (j + q < NS)
                            umma::mma(d, q || j ? adesc + (uint64_t)(q * 16) - 16 : first, bdesc + (uint64_t)(q * N * 2),
                                      idesc, q || j ? 1u : 0u);
                    umma::commit(&empty[st]);
                }
                __syncwarp();
                last_st = st;
                last_ph = ph;
                if (++st == F_STAGES) {
                    st = 0;
                    ph ^= 1u;
                }
            }
            if (umma::elect_one()) umma::commit(&accf[s]);
            __syncwarp();
            return true;
        };
        for (long long p = 0; p < npairs && !bad; ++p)
            for (int l = 0; l < nt && !bad; ++l)
                for (int s = 0; s < 2 && !bad; ++s) {
                    if (2 * p + s >= my_tiles) continue;
                    if (__any_sync(0xffffffffu, !umma::mbar_wait(&actr[s], kpar[s], GEMM_WAIT_NS))) {
                        bad = true;
                        break;
                    }
                    kpar[s] ^= 1u;
                    umma::fence_after();
                    using C1 = std::integral_constant<int, 1>;
                    using CF = std::integral_constant<int, F_SLICES>;
                    using N128 = std::integral_constant<int, 128>;
                    using N256 = std::integral_constant<int, 256>;
                    bool ok;
                    if (l == 0)
                        ok = layer(N256{}, C1{}, s, umma::desc(umma::saddr(sm + s * F_ACT_BYTES + F_IN_OFF), 128, F_SBO_IN));
                    else if (l < nt - 1) ok = layer(N256{}, CF{}, s, ones_desc);
                    else ok = layer(N128{}, CF{}, s, ones_desc);
                    bad = !ok;
                }
        // the last MMAs must be complete before TMEM is released
        if (c > 0 && __any_sync(0xffffffffu, !umma::mbar_wait(&empty[last_st], last_ph, GEMM_WAIT_NS))) bad = true;
        if (bad && lane == 0) atomicOr(a.status, 1);
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue slots
        const int e = warp - 2, s = e / F_EPI_WARPS, half = (e / 4) & 1, quad = warp & 3;
        const int r = quad * 32 + lane, bar_id = 1 + s, nthr = 32 * F_EPI_WARPS;
        const int ew = e % F_EPI_WARPS, ts = ew * 32 + lane;   // warp / thread index within the slot
        unsigned char *act = sm + s * F_ACT_BYTES;
        float *stage = reinterpret_cast<float *>(act);
        float *red = reinterpret_cast<float *>(act + F_RED_OFF);   // [max, sum][2 halves][128 rows]
        const uint32_t trow = tmem + (uint32_t)(s * 256) + ((uint32_t)(quad * 32) << 16);
        const int ncls = a.ncls;
        const int hs = (ncls + 31) / 32 * 16;                   // softmax columns per half
        const int cbeg = half * hs, cend = min(cbeg + hs, ncls);
        uint32_t kpar = 0u;                                     // parity of the next accf phase
        const auto input = [&](long long m) {
            return half == 0 && m + r < a.M ? __ldg(reinterpret_cast<const float4 *>(a.X) + m + r)
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
        };
        float4 x = input((blockIdx.x + (long long)s * gridDim.x) * 128);
        for (long long p = 0; p < npairs; ++p) {
            const long long j = 2 * p + s;
            if (j >= my_tiles) break;
            const long long m0 = (blockIdx.x + j * gridDim.x) * 128;
            // ---- inputs: split (x_hi, x_lo, x_hi, 0) rows of the K = 16 operand
            if (half == 0) {
                uint4 u0 = make_uint4(0, 0, 0, 0), u1 = u0;
                if (m0 + r < a.M) {
                    const float f0 = (x.x - a.shift.x) / a.scale.x, f1 = (x.y - a.shift.y) / a.scale.y;
                    const float f2 = (x.z - a.shift.z) / a.scale.z, f3 = (x.w - a.shift.w) / a.scale.w;
                    const __nv_bfloat162 h01 = __floats2bfloat162_rn(f0, f1), h23 = __floats2bfloat162_rn(f2, f3);
                    const float2 g01 = __bfloat1622float2(h01), g23 = __bfloat1622float2(h23);
                    u0.x = *reinterpret_cast<const uint32_t *>(&h01);
                    u0.y = *reinterpret_cast<const uint32_t *>(&h23);
                    u0.z = pack_bf16(f0 - g01.x, f1 - g01.y);
                    u0.w = pack_bf16(f2 - g23.x, f3 - g23.y);
                    u1.x = u0.x;
                    u1.y = u0.y;
                    u1.z = pack_bf16(1.f, 1.f);     // k = 12, 13: the bias columns
                }
                unsigned char *in = act + F_IN_OFF + (r >> 3) * F_SBO_IN + (r & 7) * 16;
                *reinterpret_cast<uint4 *>(in) = u0;
                *reinterpret_cast<uint4 *>(in + 128) = u1;
                umma::fence_proxy_smem();
            }
            umma::mbar_arrive(&actr[s]);
            // ---- layers
            for (int l = 0; l < nt && !bad; ++l) {
                const bool ok = umma::mbar_wait(&accf[s], kpar, GEMM_WAIT_NS);
                kpar ^= 1u;
                // the last tile's rows have left the stage that the activations overwrite
                if (l == 0 && ts == 0) umma::bulk_wait_read();
                if (!umma::bar_and(bar_id, nthr, ok)) {
                    bad = true;
                    break;
                }
                umma::fence_after();
                if (l < nt - 1) {
                    // 8 groups of 16 columns; the TMEM load of group g + 1 is
                    // in flight while group g is computed
                    const int cb = half * 128;
                    uint32_t v[2][16];
                    umma::ld16_async(trow + (uint32_t)cb, v[0]);
                    umma::wait_ld(v[0]);
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        const int cur = g & 1, nxt = cur ^ 1;
                        if (g < 7) umma::ld16_async(trow + (uint32_t)(cb + 16 * (g + 1)), v[nxt]);
                        uint32_t hv[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            hv[i] = pack_bf16(silu_of_half(__uint_as_float(v[cur][2 * i])),
                                              silu_of_half(__uint_as_float(v[cur][2 * i + 1])));
                        *reinterpret_cast<uint4 *>(act + act_off(r, cb + 16 * g)) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
                        *reinterpret_cast<uint4 *>(act + act_off(r, cb + 16 * g + 8)) = make_uint4(hv[4], hv[5], hv[6], hv[7]);
                        if (g < 7) umma::wait_ld(v[nxt]);
                    }
                    umma::fence_before();
                    umma::fence_proxy_smem();
                    umma::mbar_arrive(&actr[s]);
                } else {
                    // softmax: each half takes columns [cbeg, cend); row
                    // maxima and sums are combined through shared memory; the
                    // normalised rows are staged densely (stride ncls) over
                    // the slot's tile, which is then one contiguous block of
                    // P, written by a single bulk copy (TMA)
                    x = input(m0 + 2ll * gridDim.x * 128);   // of the slot's next tile
                    float mx = -INFINITY;
                    for (int c0 = cbeg; c0 < cend; c0 += 16) {
                        uint32_t v[16];
                        umma::ld16_async(trow + (uint32_t)c0, v);
                        umma::wait_ld(v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < cend) mx = fmaxf(mx, __uint_as_float(v[i]));
                    }
                    red[half * 128 + r] = mx;
                    umma::bar_sync(bar_id, nthr);
                    mx = fmaxf(red[r], red[128 + r]);
                    float sum = 0.f;
                    float *row = stage + r * ncls;
                    for (int c0 = cbeg; c0 < cend; c0 += 16) {
                        uint32_t v[16];
                        umma::ld16_async(trow + (uint32_t)c0, v);
                        umma::wait_ld(v);
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (c0 + i < cend) {
                                const float ez = __expf(__uint_as_float(v[i]) - mx);
                                sum += ez;
                                row[c0 + i] = ez;
                            }
                    }
                    umma::fence_before();
                    red[256 + half * 128 + r] = sum;
                    umma::bar_sync(bar_id, nthr);
                    const float inv = 1.0f / (red[256 + r] + red[384 + r]);
                    for (int c = cbeg; c < cend; c += 8) {   // eight loads in flight
                        float q[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) q[i] = row[min(c + i, cend - 1)] * inv;
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            if (c + i < cend) row[c + i] = q[i];
                    }
                    umma::fence_proxy_smem();
                    umma::bar_sync(bar_id, nthr);
                    if (ts == 0) {
                        const long long rows = a.M - m0 < 128 ? a.M - m0 : 128;
                        const uint32_t n = (uint32_t)rows * (uint32_t)ncls, n4 = n & ~3u;
                        float *dst = a.P + (size_t)m0 * ncls;
                        if (a.p_aligned) {
                            if (n4) umma::bulk_s2g(dst, stage, n4 * 4);
                            umma::bulk_commit();
                            for (uint32_t i = n4; i < n; ++i) dst[i] = stage[i];
                        } else {
                            for (uint32_t i = 0; i < n; ++i) dst[i] = stage[i];
                        }
                    }
                }
            }
            if (bad) break;
        }
        if (ts == 0) {
            umma::bulk_wait();              // the output rows have reached global memory
            if (bad) atomicOr(a.status, 1);
        }
    }
    umma::fence_before();
    __syncthreads();
    if (warp == 1) umma::tmem_free(tmem, 512);
}

constexpr size_t FUSED_SMEM = 2 * F_ACT_BYTES + F_STAGES * F_CHUNK_BYTES + (2 * F_STAGES + 4) * 8 + 16 + 256;
static_assert(FUSED_SMEM <= 232448, "fused MLP shared memory above 227 KB");
static_assert(128 * MLP_MAX_CLASSES * 4 <= F_IN_OFF && F_IN_OFF + 128 * 32 <= F_RED_OFF &&
                  F_RED_OFF + 4 * 128 * 4 <= F_ACT_BYTES,
              "softmax stage, inputs and partials overlap");

// Splits v into BF16 parts: part 0 = bf16(v), part 1 = bf16(v - part 0).
__device__ __forceinline__ float split_part(float v, int part) {
    const float hi = __bfloat162float(__float2bfloat16_rn(v));
    return part == 0 ? hi : v - hi;
}

// The packing kernels below multiply a hidden layer's operands by sc = 1/2
// (the output layer's by 1), which is exact for BF16 values: the fused
// kernel's accumulator then holds half the pre-activation (silu_of_half).

// Packs layer 1, W [256][4] and b [256] FP32, into the split K = 16 operand
// (W_hi, W_hi, W_lo, b_hi, b_lo, 0, 0) in the shared-memory layout.
__global__ void k_pack0(const float *W, const float *b, float sc, bf16 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 256 * 16) return;
    const int n = i / 16, k = i % 16;
    float v = 0.f;
    if (k < 12) v = split_part(W[n * 4 + (k & 3)], k < 8 ? 0 : 1);
    else if (k < 14) v = split_part(b[n], k - 12);
    out[slice_off(n, k, 256)] = __float2bfloat16_rn(sc * v);
}

// Packs the bias b [rows] into the K = 16 operand (b_hi, b_lo, 0, ...) of N
// rows, those from `rows` on zero.
__global__ void k_packb(const float *b, int rows, int N, float sc, bf16 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * 16) return;
    const int n = i / 16, k = i % 16;
    const float v = k < 2 && n < rows ? split_part(b[n], k) : 0.f;
    out[slice_off(n, k, N)] = __float2bfloat16_rn(sc * v);
}

// Element of a weight operand of N rows packed in 64-feature chunks, each
// laid out exactly as a shared-memory weight buffer (rows n0 .. n0 + 8 j of a
// chunk are contiguous): the training chain's.
__device__ __forceinline__ int pack_off(int n, int k, int N) {
    const int kk = k % FK;
    return k / FK * N * FK + (n >> 3) * (F_SBO_B / 2) + (kk >> 3) * 64 + (n & 7) * 8 + (kk & 7);
}

// Packs W [rows][256] (FP32, rows <= N, the others zero) as BF16, times sc, in
// slices or in chunks.
template <bool SLICES> __global__ void k_pack(const float *W, int rows, int N, float sc, bf16 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * 256) return;
    const int n = i / 256, k = i % 256;
    const float v = n < rows ? __bfloat162float(__float2bfloat16_rn(W[i])) : 0.f;
    out[SLICES ? slice_off(n, k, N) : pack_off(n, k, N)] = __float2bfloat16_rn(sc * v);
}

// Packs W^T [256][N] (FP32 W [rows][256]) as BF16: the operand of a layer's
// input gradient.
__global__ void k_pack_t(const float *W, int rows, int N, bf16 *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * 256) return;
    const int n = i / 256, k = i % 256;
    out[pack_off(k, n, 256)] = __float2bfloat16_rn(n < rows ? W[i] : 0.f);
}


// ---------------------------------------------------------------- training
// A training step on a batch of B rows was some 50 small launches (per layer
// a GEMM, two transposes, column sums, sums of partials, two Adam kernels),
// 466 us at B = 512 for 0.7 GFLOP: launches, and epilogues that read and
// wrote one row per lane.  It is three launches now; of 5 layers at B = 512:
// k_train_chain 38 us, k_train_grads 7.1 us, k_train_update 4.1 us.
//
// k_train_chain: one thread-block cluster of CS CTAs per 128-row tile runs the
// whole forward pass, the softmax and loss, and the backward pass down to the
// first layer.  CTA `rank` computes columns rank * 256/CS .. of every layer:
// its slice of the weights arrives by bulk copies while the previous layer is
// computed, the accumulator is a 128 x 256/CS tile in TMEM, and the finished
// BF16 activations (or gradients) go into the CTA's own next A operand and
// from there, as contiguous 64-column slabs, to the other CTAs' by bulk copies
// through distributed shared memory that signal the receiver's mbarrier: no
// cluster barrier per layer.  (Storing every 16 bytes into all CTAs and
// meeting at a cluster barrier took 44 us per step when this took 41.)  What it leaves in global memory is transposed, [column][batch], so
// that a warp's 32 rows are contiguous and the weight gradients' operands are
// K-major.  The tile is one row block of 128 (the M of the instruction); the
// columns are what is split, because a batch of 512 has only four row blocks.
// It is bound by the latency of its 2 (layers) dependent steps: of about 7,000
// clocks each, the exchange takes 2,700, the product 1,400, the epilogue 2,800
// (16 columns of a row per thread).
// Every value is that of the layer-by-layer formulation: the K order of the
// products, the FP32 epilogues and the BF16 roundings are the same.

// Where the parameters of a layer lie in the packed vector W_1, b_1, ...
struct ParamMap {
    int nl, ncls;
    __host__ __device__ int out(int l) const { return l == nl - 1 ? ncls : 256; }
    __host__ __device__ int outp(int l) const { return l == nl - 1 ? 128 : 256; }
    __host__ __device__ int in(int l) const { return l == 0 ? 4 : 256; }
    __host__ __device__ int W(int l) const { return l == 0 ? 0 : 1280 + (l - 1) * (65536 + 256); }
    __host__ __device__ int b(int l) const { return W(l) + out(l) * in(l); }
    __host__ __device__ int count() const { return b(nl - 1) + ncls; }
};

struct TrainArgs {
    const float *X, *T;
    int B;
    ParamMap pm;
    float4 shift, scale;
    const float *w;                // packed FP32 parameters
    const bf16 *Wf[F_MAXL + 1];    // packed operands of layers >= 1 (pack_off): W and W^T
    const bf16 *Wb[F_MAXL + 1];
    float *xf;                     // [B][4] features
    float *Z;                      // [hidden layer][256][B] pre-activations
    bf16 *H;                       // [hidden layer][256][B] activations
    bf16 *dZ;                      // [layer][256][B] loss gradients of the pre-activations (last layer: 128 rows)
    float *rowloss;                // [B]
    float inv_batch;
    int *status;
    int dbg_skip;                  // mlp_train_selftest: CTA 0 does not signal product dbg_skip - 1
    uint64_t dbg_wait_ns;          // and waits no longer than this; the others' limit stays, so they find its columns
};

constexpr int T_THREADS = 512;
constexpr int T_GROUPS = T_THREADS / 128;   // column groups of a CTA's epilogue
// A operand: slabs of 128 rows x 64 columns, each contiguous (8-row groups of
// 1024 bytes, as the weights' chunks)
constexpr int T_SLAB = 128 * FK * 2;
__device__ __forceinline__ int tact_off(int r, int k) {
    return (k >> 6) * T_SLAB + (r >> 3) * F_SBO_B + ((k >> 3) & 7) * 128 + (r & 7) * 16 + (k & 7) * 2;
}
constexpr int T_LOGIT_LD = 113;    // odd, > MLP_MAX_CLASSES: rows of the staged logits fall in different banks
constexpr int T_DLOG_LD = 136;

template <int CS> struct TrainShape {
    static constexpr int NS = 256 / CS;            // hidden columns of a CTA
    static constexpr int NO = 128 / CS;            // output columns of a CTA
    static constexpr int NBUF = CS == 2 ? 1 : 2;   // weight buffers (a whole layer's slice each)
    static constexpr int RP = 128 / CS;            // rows of a CTA's softmax
    static constexpr int WBYTES = NS * 256 * 2;
    static constexpr size_t smem = 2 * (size_t)F_ACT_BYTES + NBUF * WBYTES + 64;
    static_assert(CS == 2 || CS == 4, "a CTA's columns are whole 64-column slabs");
};
static_assert(TrainShape<2>::smem <= 232448, "training chain: shared memory above 227 KB");
static_assert(64 * T_LOGIT_LD * 4 + 64 * T_DLOG_LD * 2 <= F_ACT_BYTES, "training chain: softmax stage");

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Address of this CTA's shared-memory location `addr` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, int rank) {
    uint32_t d;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(addr), "r"(rank));
    return d;
}
// Bulk copy of `bytes` of this CTA's shared memory to `dst` in another CTA of
// the cluster, counted on that CTA's mbarrier `bar` (cluster addresses).
__device__ __forceinline__ void bulk_s2cluster(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "r"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
    asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// All CTAs of the cluster: generic writes to any of their shared memory are
// visible, also to the tensor cores, after it.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("fence.proxy.async;" ::: "memory");
    umma::fence_before();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    umma::fence_after();
    asm volatile("fence.proxy.async;" ::: "memory");
}

// TEST: the kernel of mlp_train_selftest; the other has none of its checks.
template <int CS, bool TEST>
__global__ void __launch_bounds__(T_THREADS, 1) k_train_chain(const __grid_constant__ TrainArgs a) {
    using S = TrainShape<CS>;
    extern __shared__ __align__(1024) unsigned char sm[];
    unsigned char *wbuf = sm + 2 * F_ACT_BYTES;
    uint64_t *full = reinterpret_cast<uint64_t *>(wbuf + S::NBUF * S::WBYTES);   // [NBUF]
    uint64_t *done = full + S::NBUF;                                            // accumulator complete
    uint64_t *arr = done + 1;                                                   // [2] the other CTAs' columns of an A operand are here
    uint64_t *drain = arr + 2;                                                  // after a failed wait: what was issued is complete
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(drain + 1);
    uint32_t *s_bad = s_tmem + 1;                                               // a wait of some CTA gave up
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)cluster_rank(), m0 = (int)(blockIdx.x / CS) * 128;
    const ParamMap pm = a.pm;
    const int nl = pm.nl, B = a.B, nops = 2 * (nl - 1);
    // a warp may read only the TMEM lanes 32 (warp mod 4) .. +31: four warps
    // take the 128 rows of one group of the CTA's columns
    const int quad = warp & 3, grp = warp >> 2, r = quad * 32 + lane;
    constexpr uint32_t ncols = S::NS < 32 ? 32 : S::NS;
    if (warp == 0) umma::tmem_alloc(s_tmem, ncols);
    if (tid == 0) {
        for (int i = 0; i < S::NBUF; ++i) umma::mbar_init(&full[i], 1);
        umma::mbar_init(done, 1);
        umma::mbar_init(&arr[0], 1);
        umma::mbar_init(&arr[1], 1);
        umma::mbar_init(drain, 1);
        umma::mbar_fence_init();
        *s_bad = 0;
    }
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    const uint32_t tmem = *s_tmem, trow = tmem + ((uint32_t)(quad * 32) << 16);
    const uint32_t act0 = umma::saddr(sm);
    bool bad = false;
    int loads = nops;       // weight slices that are requested (fewer after a failure)
    uint32_t got = 0;       // warp 0: phases of arr[0] (low half) and arr[1] that have completed
    const bool test = TEST && blockIdx.x == 0;
    const auto wait = [&](uint64_t *bar, uint32_t parity) {
        return umma::mbar_wait(bar, parity, test ? a.dbg_wait_ns : GEMM_WAIT_NS);
    };
    // operation g reads operand g & 1 up to the output layer; the backward
    // pass starts over from the output layer's
    const auto a_buf = [&](int g) { return g < nl - 1 ? g & 1 : (g - 1) & 1; };
    // operation g < nl - 1: layer g + 1 forward; then layers nl - 1 .. 1 backward
    const auto op_layer = [&](int g) { return g < nl - 1 ? g + 1 : 2 * (nl - 1) - g; };
    const auto load = [&](int g) {   // thread 0: this CTA's slice of the operation's weights
        if (g >= nops) return;
        const int l = op_layer(g);
        const bool fwd = g < nl - 1;
        const int N = fwd ? pm.outp(l) : 256, K = fwd ? 256 : pm.outp(l), ns = N / CS;
        const bf16 *src = (fwd ? a.Wf[l] : a.Wb[l]) + rank * ns * FK;
        unsigned char *dst = wbuf + (g % S::NBUF) * S::WBYTES;
        uint64_t *bar = &full[g % S::NBUF];
        umma::mbar_expect_tx(bar, (uint32_t)(ns * K * 2));
        for (int kc = 0; kc < K / FK; ++kc)
            umma::bulk_g2s(dst + kc * ns * FK * 2, src + (size_t)kc * N * FK, (uint32_t)(ns * FK * 2), bar);
    };
    // warp 0: issues the operation's MMAs, one elected lane of uniform control
    // flow (from a divergent branch a product took 0.35 us more); operand
    // g & 1
    const auto product = [&](int g) {
        const int l = op_layer(g);
        const bool fwd = g < nl - 1;
        const int ns = (fwd ? pm.outp(l) : 256) / CS, K = fwd ? 256 : pm.outp(l), cur = a_buf(g);
        // waited for also after a failure: the copies always come, and no
        // CTA may leave before those into it have landed
        const bool here = __all_sync(0xffffffffu, wait(&arr[cur], got >> (16 * cur) & 1u));
        got += here ? 1u << (16 * cur) : 0u;
        bad = __any_sync(0xffffffffu, bad || !here);
        if (bad) return;
        bad = __any_sync(0xffffffffu, !wait(&full[g % S::NBUF], (g / S::NBUF) & 1));
        if (bad) return;
        umma::fence_after();
        const uint32_t idesc = umma::idesc_bf16(128, ns);
        const uint64_t ad = umma::desc(act0 + cur * F_ACT_BYTES, 128, F_SBO_B);
        const uint64_t bd = umma::desc(umma::saddr(wbuf + (g % S::NBUF) * S::WBYTES), 128, F_SBO_B);
        if (umma::elect_one()) {
            for (int kc = 0; kc < K / FK; ++kc)
#pragma unroll
                for (int k4 = 0; k4 < FK / 16; ++k4)
                    umma::mma(tmem, ad + (uint64_t)((kc * T_SLAB) >> 4) + (uint64_t)(k4 * 16),
                              bd + (uint64_t)((kc * ns * FK * 2) >> 4) + (uint64_t)(k4 * 16), idesc,
                              (kc | k4) ? 1u : 0u);
            if (!(test && a.dbg_skip == g + 1)) umma::commit(done);   // the self-test withholds one signal
        }
        __syncwarp();
    };
    // every thread: the operation's accumulator is complete; its weight buffer is free again
    const auto finish = [&](int g) {
        if (!bad && !wait(done, g & 1)) bad = true;
        umma::fence_after();
        if (tid == 0) {
            if (!bad) load(g + S::NBUF);
            else loads = min(loads, g + S::NBUF);
        }
    };
    // 16 BF16 values of row r, columns c .. c + 15 of the layer, into this CTA's operand `buf`
    const auto put = [&](int buf, int c, const uint32_t (&h)[8]) {
        unsigned char *o = sm + buf * F_ACT_BYTES;
        *reinterpret_cast<uint4 *>(o + tact_off(r, c)) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4 *>(o + tact_off(r, c + 8)) = make_uint4(h[4], h[5], h[6], h[7]);
    };
    // All threads, after their puts: sends `n` pieces of `bytes` of operand
    // `buf`, `stride` apart from `off` on, to the other CTAs.  Their operand
    // is free: a CTA computes this layer only with this CTA's columns of the
    // last one, sent after the product that read the operand had finished.
    const auto send = [&](int buf, int off, int n, int stride, uint32_t bytes) {
        umma::fence_proxy_smem();
        umma::fence_before();
        __syncthreads();
        umma::fence_after();
        if (tid == 0) {
            umma::mbar_expect_tx(&arr[buf], (uint32_t)(CS - 1) * n * bytes);
            const uint32_t src = act0 + buf * F_ACT_BYTES + off, bar = umma::saddr(&arr[buf]);
            for (int q = 1; q < CS; ++q) {
                const int to = (rank + q) % CS;
                for (int i = 0; i < n; ++i)
                    bulk_s2cluster(cluster_addr(src + i * stride, to), src + i * stride, bytes, cluster_addr(bar, to));
            }
        }
    };
    const int my_slab = rank * (S::NS / FK) * T_SLAB;
    constexpr uint32_t SLABS = S::NS / FK * T_SLAB;
    const auto put_t = [&](bf16 *dst, int c, const uint32_t (&h)[8]) {   // the same, transposed in global memory
#pragma unroll
        for (int i = 0; i < 16; ++i)
            reinterpret_cast<uint16_t *>(dst)[(size_t)(c + i) * B + m0 + r] =
                (uint16_t)(i & 1 ? h[i / 2] >> 16 : h[i / 2] & 0xffffu);
    };
    constexpr int CH = S::NS / T_GROUPS < 16 ? 16 : S::NS / T_GROUPS;   // columns of a group
    constexpr int CO = S::NO / T_GROUPS < 16 ? 16 : S::NO / T_GROUPS;
    if (tid == 0)
        for (int g = 0; g < S::NBUF; ++g) load(g);
    cluster_sync();   // every CTA of the cluster runs: its shared memory may be written
    // ---- first layer (4 inputs) on the CUDA cores
    {
        const float4 x = make_float4(a.X[4 * (size_t)(m0 + r)], a.X[4 * (size_t)(m0 + r) + 1],
                                     a.X[4 * (size_t)(m0 + r) + 2], a.X[4 * (size_t)(m0 + r) + 3]);
        const float f0 = (x.x - a.shift.x) / a.scale.x, f1 = (x.y - a.shift.y) / a.scale.y;
        const float f2 = (x.z - a.shift.z) / a.scale.z, f3 = (x.w - a.shift.w) / a.scale.w;
        if (rank == 0 && grp == 0) reinterpret_cast<float4 *>(a.xf)[m0 + r] = make_float4(f0, f1, f2, f3);
        const float4 *W = reinterpret_cast<const float4 *>(a.w);
        const float *b = a.w + pm.b(0);
        for (int c0 = grp * CH; c0 < min(S::NS, grp * CH + CH); c0 += 16) {
            const int c = rank * S::NS + c0;
            uint32_t h[8];
            float hv[2], zz[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float4 w = __ldg(W + c + i);
                zz[i] = __ldg(b + c + i) + w.x * f0 + w.y * f1 + w.z * f2 + w.w * f3;
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int o = c + i;
                const float z = zz[i];
                a.Z[(size_t)o * B + m0 + r] = z;
                hv[i & 1] = silu(z);
                if (i & 1) h[i / 2] = pack_bf16(hv[0], hv[1]);
            }
            put_t(a.H, c, h);
            put(0, c, h);
        }
    }
    send(0, my_slab, 1, 0, SLABS);
    // ---- hidden layers
    for (int g = 0; g < nl - 2; ++g) {
        if (warp == 0) product(g);
        const float *b = a.w + pm.b(g + 1) + rank * S::NS + grp * CH;
        float *Z = a.Z + (size_t)(g + 1) * 256 * B;
        bf16 *H = a.H + (size_t)(g + 1) * 256 * B;
        float bias[CH];   // requested while the product runs
#pragma unroll
        for (int i = 0; i < CH; ++i) bias[i] = grp * CH < S::NS ? __ldg(b + i) : 0.f;
        finish(g);
#pragma unroll
        for (int c1 = 0; c1 < CH; c1 += 16) {
            const int c0 = grp * CH + c1, c = rank * S::NS + c0;
            if (c0 >= S::NS) break;
            float v[16];
            umma::ld16(trow + (uint32_t)c0, v);
            uint32_t h[8];
            float hv[2];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const float z = v[i] + bias[c1 + i];
                Z[(size_t)(c + i) * B + m0 + r] = z;
                hv[i & 1] = silu(z);
                if (i & 1) h[i / 2] = pack_bf16(hv[0], hv[1]);
            }
            put_t(H, c, h);
            put(a_buf(g + 1), c, h);
        }
        send(a_buf(g + 1), my_slab, 1, 0, SLABS);
    }
    // targets of this warp's softmax rows, requested while the output layer runs
    constexpr int SR = (S::RP + T_THREADS / 32 - 1) / (T_THREADS / 32);   // rows per warp
    float tgt[SR][4];
#pragma unroll
    for (int u = 0; u < SR; ++u) {
        const int q = warp + u * (T_THREADS / 32);
        const float *T = a.T + (size_t)(m0 + rank * S::RP + q) * pm.ncls;
#pragma unroll
        for (int k = 0; k < 4; ++k) tgt[u][k] = q < S::RP && lane + 32 * k < pm.ncls ? __ldg(T + lane + 32 * k) : 0.f;
    }
    // ---- output layer: logits of row r to the CTA that owns the row, staged
    // in its unused A operand
    const int cur = a_buf(nl - 2);
    float *logits = reinterpret_cast<float *>(sm + (cur ^ 1) * F_ACT_BYTES);          // [RP][T_LOGIT_LD]
    bf16 *dl = reinterpret_cast<bf16 *>(logits + S::RP * T_LOGIT_LD);                 // [RP][T_DLOG_LD]
    {
        const int g = nl - 2;
        if (warp == 0) product(g);
        const float *b = a.w + pm.b(nl - 1);
        float bias[CO];
#pragma unroll
        for (int i = 0; i < CO; ++i) {
            const int c = rank * S::NO + grp * CO + i;
            bias[i] = grp * CO < S::NO && c < pm.ncls ? __ldg(b + c) : 0.f;
        }
        finish(g);
        const uint32_t row = cluster_addr(umma::saddr(logits + (r % S::RP) * T_LOGIT_LD), r / S::RP);
#pragma unroll
        for (int c1 = 0; c1 < CO; c1 += 16) {
            const int c0 = grp * CO + c1, c = rank * S::NO + c0;
            if (c0 >= S::NO) break;
            float v[16];
            umma::ld16(trow + (uint32_t)c0, v);
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (c + i < pm.ncls) st_cluster(row + 4u * (c + i), v[i] + bias[c1 + i]);
        }
        cluster_sync();
    }
    // ---- softmax, the row's share of the mean KL loss, and d loss / d logits
    // = (p sum(t) - t) / B as BF16 (zero in the padding columns); one warp per row
#pragma unroll
    for (int u = 0; u < SR; ++u) {
        const int q = warp + u * (T_THREADS / 32);
        if (q >= S::RP) break;
        const int ncls = pm.ncls, m = m0 + rank * S::RP + q;
        const float *l = logits + q * T_LOGIT_LD;
        const float(&t)[4] = tgt[u];
        float x[4], mx = -INFINITY;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[k] = lane + 32 * k < ncls ? l[lane + 32 * k] : -INFINITY;
            mx = fmaxf(mx, x[k]);
        }
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            x[k] = __expf(x[k] - mx);
            if (lane + 32 * k < ncls) s += x[k];
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        const float inv = 1.0f / s;
        float ts = 0.f, loss = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (lane + 32 * k < ncls) ts += t[k];
        for (int o = 16; o > 0; o >>= 1) ts += __shfl_xor_sync(0xffffffffu, ts, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int c = lane + 32 * k;
            float d = 0.f;
            if (c < ncls) {
                const float p = x[k] * inv;
                if (t[k] > 0.f) loss += t[k] * (__logf(t[k]) - __logf(p));
                d = (p * ts - t[k]) * a.inv_batch;
            }
            dl[q * T_DLOG_LD + c] = __float2bfloat16_rn(d);
        }
        for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
        if (lane == 0) a.rowloss[m] = loss * a.inv_batch;
    }
    __syncthreads();
    for (int e = tid; e < S::RP * 16; e += T_THREADS) {
        const int q = e / 16, k = e % 16 * 8;
        *reinterpret_cast<uint4 *>(sm + cur * F_ACT_BYTES + tact_off(rank * S::RP + q, k)) =
            *reinterpret_cast<const uint4 *>(&dl[q * T_DLOG_LD + k]);
    }
    bf16 *dZ = a.dZ + (size_t)(nl - 1) * 256 * B;
    for (int e = tid; e < S::RP * 128; e += T_THREADS)
        dZ[(size_t)(e / S::RP) * B + m0 + rank * S::RP + e % S::RP] = dl[e % S::RP * T_DLOG_LD + e / S::RP];
    // (every CTA's product of the output layer is complete: the cluster met;
    // after this no thread reads the stage, which the next layer overwrites)
    send(cur, rank * S::RP / 8 * F_SBO_B, 2, T_SLAB, S::RP / 8 * F_SBO_B);
    // ---- backward: dZ_{l-1} = (dZ_l W_l) silu'(Z_{l-1})
    for (int l = nl - 1; l >= 1; --l) {
        const int g = 2 * (nl - 1) - l;
        if (warp == 0) product(g);
        const float *Z = a.Z + (size_t)(l - 1) * 256 * B;
        dZ = a.dZ + (size_t)(l - 1) * 256 * B;
        float z[CH];   // requested while the product runs
#pragma unroll
        for (int i = 0; i < CH; ++i)
            z[i] = grp * CH < S::NS ? Z[(size_t)(rank * S::NS + grp * CH + i) * B + m0 + r] : 0.f;
        finish(g);
#pragma unroll
        for (int c1 = 0; c1 < CH; c1 += 16) {
            const int c0 = grp * CH + c1, c = rank * S::NS + c0;
            if (c0 >= S::NS) break;
            float v[16];
            umma::ld16(trow + (uint32_t)c0, v);
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 16; i += 2)
                h[i / 2] = pack_bf16(v[i] * silu_grad(z[c1 + i]), v[i + 1] * silu_grad(z[c1 + i + 1]));
            put_t(dZ, c, h);
            if (l > 1) put(a_buf(g + 1), c, h);
        }
        if (l > 1) send(a_buf(g + 1), my_slab, 1, 0, SLABS);
    }
    if (warp == 0) bad = __any_sync(0xffffffffu, bad);
    if (bad)
        for (int q = 0; q < CS; ++q) st_cluster(cluster_addr(umma::saddr(s_bad), q), 1.0f);
    cluster_sync();   // no CTA leaves while another may read or write its shared memory
    if (*reinterpret_cast<volatile uint32_t *>(s_bad)) {
        // a CTA that gave up may have stopped waiting for columns: all are on
        // their way now, and no CTA leaves before they have landed
        if (warp == 0)
            for (int b = 0; b < 2; ++b) {
                int n = 0;
                for (int g = 0; g < nops; ++g) n += a_buf(g) == b;
                for (int i = (int)(got >> (16 * b) & 0xffffu); i < n; ++i)
                    if (!wait(&arr[b], i & 1)) break;
            }
        cluster_sync();
    }
    if (bad) {
        // a wait gave up: products and weight copies may still run; wait (with
        // a limit) before their TMEM and shared memory are given up, and flag it
        if (warp == 0 && umma::elect_one()) {   // the lane that issued
            umma::commit(drain);
            wait(drain, 0);
        }
        if (tid == 0)   // the last request of each buffer
            for (int g = max(0, loads - S::NBUF); g < loads; ++g)
                wait(&full[g % S::NBUF], (g / S::NBUF) & 1);
        atomicOr(a.status, 1);
    }
    umma::fence_before();
    __syncthreads();
    if (warp == 0) umma::tmem_free(tmem, ncols);
}

// ---- gradients' partial sums over the batch
// CTAs [0, tiles * ks): 128 x 128 tiles of dW_l = dZ_l^T H_{l-1}, l >= 1, split
// z of ks over the batch (both operands K-major: [column][batch]).  The rest:
// sums of dZ over chunks of GRAD_ROWS rows (bias gradients) and, for the first
// layer, of dZ x_f, one thread per column and chunk.  All are summed in split
// and chunk order by k_train_update, so nothing depends on the launch.
struct GradArgs {
    const bf16 *H, *dZ;
    const float *xf;
    int B, ks;
    ParamMap pm;
    float *part;      // [ks][tiles][128][128]
    float *bpart;     // [chunk][layer * 256 + column]
    float *wpart;     // [chunk][256 * 4] first layer
    int *status;
    uint64_t wait_ns; // limit of every mbarrier wait
    int dbg_skip;     // mlp_train_selftest: CTA 0 does not signal stage dbg_skip - 1 (0: never)
};
constexpr int G_STAGES = 3;
constexpr int G_STAGE_BYTES = 2 * 128 * GBK * 2;
constexpr size_t GRADS_SMEM = G_STAGES * G_STAGE_BYTES + 64;

__host__ __device__ inline int grad_tiles(const ParamMap &pm) { return 4 * (pm.nl - 2) + 2; }
// Tile of weight (r, c) of layer l >= 1.
__host__ __device__ inline int grad_tile(int l, int r, int c) { return 4 * (l - 1) + (r >> 7) * 2 + (c >> 7); }
__host__ __device__ inline int grad_sums(const ParamMap &pm) { return pm.nl * 256 - 128; }

__global__ void __launch_bounds__(128) k_train_grads(const __grid_constant__ GradArgs a) {
    extern __shared__ __align__(1024) unsigned char sm[];
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, B = a.B;
    const int tiles = grad_tiles(a.pm);
    if ((int)blockIdx.x >= tiles * a.ks) {
        const int per = grad_sums(a.pm) / 128, e = (int)blockIdx.x - tiles * a.ks;
        const int ch = e / per, i = e % per * 128 + tid, l = i >> 8, c = i & 255;   // block-uniform chunk and layer
        const bf16 *d = a.dZ + ((size_t)l * 256 + c) * B + ch * GRAD_ROWS;
        uint4 q[GRAD_ROWS / 8];
#pragma unroll
        for (int k = 0; k < GRAD_ROWS / 8; ++k) q[k] = reinterpret_cast<const uint4 *>(d)[k];
        float s = 0.f;
        if (l == 0) {
            float4 *xs = reinterpret_cast<float4 *>(sm);
            xs[tid] = reinterpret_cast<const float4 *>(a.xf)[ch * GRAD_ROWS + tid];
            __syncthreads();
            float w0 = 0.f, w1 = 0.f, w2 = 0.f, w3 = 0.f;
#pragma unroll
            for (int k = 0; k < GRAD_ROWS / 8; ++k) {
                const uint32_t u[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float v = __uint_as_float(j & 1 ? u[j / 2] & 0xffff0000u : u[j / 2] << 16);
                    const float4 x = xs[8 * k + j];
                    s += v;
                    w0 += v * x.x;
                    w1 += v * x.y;
                    w2 += v * x.z;
                    w3 += v * x.w;
                }
            }
            reinterpret_cast<float4 *>(a.wpart)[ch * 256 + c] = make_float4(w0, w1, w2, w3);
        } else {
#pragma unroll
            for (int k = 0; k < GRAD_ROWS / 8; ++k) {
                const uint32_t u[4] = {q[k].x, q[k].y, q[k].z, q[k].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) s += __uint_as_float(j & 1 ? u[j / 2] & 0xffff0000u : u[j / 2] << 16);
            }
        }
        a.bpart[(size_t)ch * a.pm.nl * 256 + i] = s;
        return;
    }
    const int tile = (int)blockIdx.x % tiles, z = (int)blockIdx.x / tiles;
    const int l = tile / 4 + 1, mt = tile % 4 / 2, nt = tile % 2;
    uint64_t *mbar = reinterpret_cast<uint64_t *>(sm + G_STAGES * G_STAGE_BYTES);   // [G_STAGES], then the drain
    uint32_t *s_tmem = reinterpret_cast<uint32_t *>(mbar + G_STAGES + 1);
    __shared__ int s_ok;
    if (warp == 0) umma::tmem_alloc(s_tmem, 128);
    if (tid == 0) {
        for (int i = 0; i <= G_STAGES; ++i) umma::mbar_init(&mbar[i], 1);
        umma::mbar_fence_init();
        s_ok = 1;
    }
    umma::fence_before();
    __syncthreads();
    umma::fence_after();
    const uint32_t tmem = *s_tmem;
    const int K = B / a.ks, nk = K / GBK;
    const bf16 *A = a.dZ + ((size_t)l * 256 + mt * 128) * B + (size_t)z * K;
    const bf16 *Bm = a.H + ((size_t)(l - 1) * 256 + nt * 128) * B + (size_t)z * K;
    const uint32_t idesc = umma::idesc_bf16(128, 128);
    const auto fetch = [&](int kt) {
        unsigned char *sa = sm + kt % G_STAGES * G_STAGE_BYTES, *sb = sa + G_STAGE_BYTES / 2;
        for (int c = tid; c < 128 * 8; c += 128) {
            const int r = c >> 3, k8 = c & 7;
            cpa16(sa + tile_off(r, k8), A + (size_t)r * B + kt * GBK + k8 * 8);
            cpa16(sb + tile_off(r, k8), Bm + (size_t)r * B + kt * GBK + k8 * 8);
        }
    };
    for (int kt = 0; kt < G_STAGES - 1; ++kt) {
        if (kt < nk) fetch(kt);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(G_STAGES - 2) : "memory");
        umma::fence_proxy_smem();
        __syncthreads();
        const int s = kt % G_STAGES;
        if (warp == 0 && umma::elect_one()) {
            umma::fence_after();
            const uint32_t a0 = umma::saddr(sm + s * G_STAGE_BYTES), b0 = a0 + G_STAGE_BYTES / 2;
#pragma unroll
            for (int k4 = 0; k4 < GBK / 16; ++k4)
                umma::mma(tmem, umma::desc(a0 + k4 * 256, 128, 1024), umma::desc(b0 + k4 * 256, 128, 1024), idesc,
                          (kt | k4) ? 1u : 0u);
            // (the self-test withholds one signal)
            if (!(a.dbg_skip == kt + 1 && blockIdx.x == 0)) umma::commit(&mbar[s]);
        }
        // the stage fetched next was last read by the products of stage kt - 1
        const int nx = kt + G_STAGES - 1;
        if (nx < nk) {
            if (nx >= G_STAGES && !umma::mbar_wait(&mbar[nx % G_STAGES], (nx / G_STAGES - 1) & 1, a.wait_ns)) s_ok = 0;
            __syncthreads();
            if (!s_ok) break;
            fetch(nx);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (s_ok && !umma::mbar_wait(&mbar[(nk - 1) % G_STAGES], ((nk - 1) / G_STAGES) & 1, a.wait_ns)) s_ok = 0;
    __syncthreads();
    if (!s_ok && warp == 0 && umma::elect_one()) {
        umma::commit(&mbar[G_STAGES]);
        umma::mbar_wait(&mbar[G_STAGES], 0, a.wait_ns);
    }
    __syncthreads();
    umma::fence_after();
    if (s_ok) {
        float *C = a.part + ((size_t)z * tiles + tile) * 16384 + (size_t)(warp * 32 + lane) * 128;
        for (int c0 = 0; c0 < 128; c0 += 16) {
            float v[16];
            umma::ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                reinterpret_cast<float4 *>(C + c0)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        }
    } else if (tid == 0) {
        atomicOr(a.status, 1);
    }
    umma::fence_before();
    __syncthreads();
    if (warp == 0) umma::tmem_free(tmem, 128);
}

// ---- sums of the partials, Adam
struct AdamArgs {
    float lr, b1, b2, c1, c2, eps;
    float *g;          // not NULL: write the gradient here and update nothing
};
struct UpdateArgs {
    ParamMap pm;
    const float *part, *bpart, *wpart;
    int ks, nch;
    float *w, *mom, *var;
    bf16 *Wf[F_MAXL + 1], *Wb[F_MAXL + 1];
    const float *rowloss;
    int B;
    float *loss;       // may be NULL
};

// One thread per parameter; the last block adds the rows' losses.
__global__ void __launch_bounds__(256) k_train_update(const __grid_constant__ UpdateArgs a, const AdamArgs ad) {
    if (blockIdx.x == gridDim.x - 1) {
        if (!a.loss) return;
        __shared__ float s[256];
        float acc = 0.f;
        for (int i = threadIdx.x; i < a.B; i += 256) acc += a.rowloss[i];
        s[threadIdx.x] = acc;
        __syncthreads();
        for (int o = 128; o > 0; o >>= 1) {
            if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
            __syncthreads();
        }
        if (threadIdx.x == 0) *a.loss = s[0];
        return;
    }
    const int i = blockIdx.x * 256 + threadIdx.x;
    const ParamMap pm = a.pm;
    if (i >= pm.count()) return;
    // parameter i: layer l, weight (r, c) or bias r (c < 0)
    int l = i < 1280 ? 0 : 1 + (i - 1280) / 65792;
    if (l > pm.nl - 1) l = pm.nl - 1;
    const int j = i - pm.W(l), nw = pm.out(l) * pm.in(l);
    const int r = j < nw ? j / pm.in(l) : j - nw, c = j < nw ? j % pm.in(l) : -1;
    const float *src;
    size_t stride;
    int nz;
    if (c < 0) {
        src = a.bpart + l * 256 + r;
        stride = (size_t)pm.nl * 256;
        nz = a.nch;
    } else if (l == 0) {
        src = a.wpart + j;
        stride = 1024;
        nz = a.nch;
    } else {
        src = a.part + (size_t)grad_tile(l, r, c) * 16384 + (r & 127) * 128 + (c & 127);
        stride = (size_t)grad_tiles(pm) * 16384;
        nz = a.ks;
    }
    float gr = 0.f;
#pragma unroll 4
    for (int z = 0; z < nz; ++z) gr += src[z * stride];
    if (ad.g) {
        ad.g[i] = gr;
        return;
    }
    const float m = ad.b1 * a.mom[i] + (1.f - ad.b1) * gr;
    const float v = ad.b2 * a.var[i] + (1.f - ad.b2) * gr * gr;
    a.mom[i] = m;
    a.var[i] = v;
    const float nw_ = a.w[i] - ad.lr * (m / ad.c1) / (sqrtf(v / ad.c2) + ad.eps);
    a.w[i] = nw_;
    if (l > 0 && c >= 0) {
        const bf16 h = __float2bfloat16_rn(nw_);
        a.Wf[l][pack_off(r, c, pm.outp(l))] = h;
        a.Wb[l][pack_off(c, r, 256)] = h;
    }
}

}  // namespace mdlg

using namespace mdlg;

// ---------------------------------------------------------------- model
struct mlp_model {
    int nl = 0;                   // linear layers (hidden + 1)
    int ncls = 81;
    float shift[4], scale[4];
    // FP32 master parameters, Adam moments and gradient, packed as `params`
    float *w = nullptr, *mom = nullptr, *var = nullptr, *g = nullptr;
    std::vector<bf16 *> Wf, Wb;   // packed BF16 W and W^T of layers >= 1 (training)
    std::vector<bf16 *> Wp;       // bias and weights in slices for the fused forward pass
    bool packed = false;
    int adam_t = 0;
    // workspace
    long long cap = 0;            // rows
    float *xf = nullptr, *rowloss = nullptr, *Z = nullptr;
    bf16 *H = nullptr, *dZ = nullptr;
    float *part = nullptr, *bpart = nullptr, *wpart = nullptr;   // partial sums of the gradients
    int *status = nullptr;
    std::vector<void *> allocs, ws;
    ParamMap map() const { return ParamMap{nl, ncls}; }
};

namespace {

int malloc_into(std::vector<void *> &v, void **p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes ? bytes : 16);
    if (e != cudaSuccess) return fail(MD_E_NOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
    v.push_back(*p);
    return MD_OK;
}

// Splits of the weight gradients over a batch: as many as leave every split
// two stages of GBK rows at least.
int grad_splits(int B) {
    const int nkt = B / GBK;
    int ks = 1;
    while (ks * 2 <= GRAD_MAX_SPLIT && nkt % (ks * 2) == 0 && nkt / (ks * 2) >= 2) ks *= 2;
    return ks;
}

// Grows the row workspace to hold `rows` rows (multiple of 128).
int ensure_ws(mlp_model *m, long long rows) {
    if (rows <= m->cap) return MD_OK;
    cudaDeviceSynchronize();
    for (void *p : m->ws) cudaFree(p);
    m->ws.clear();
    m->cap = 0;
    const size_t R = (size_t)rows, nch = R / GRAD_ROWS;
    int rc = MD_OK;
    auto A = [&](void **p, size_t bytes) {
        if (rc == MD_OK) rc = malloc_into(m->ws, p, bytes);
    };
    A((void **)&m->xf, R * 4 * sizeof(float));
    A((void **)&m->rowloss, R * sizeof(float));
    A((void **)&m->Z, R * 256 * (m->nl - 1) * sizeof(float));
    A((void **)&m->H, R * 256 * (m->nl - 1) * sizeof(bf16));
    A((void **)&m->dZ, R * 256 * m->nl * sizeof(bf16));
    // a batch of fewer rows may have more splits: room for the most
    A((void **)&m->part, (size_t)std::min<long long>(GRAD_MAX_SPLIT, std::max<long long>(1, rows / GBK / 2)) *
                             grad_tiles(m->map()) * 16384 * sizeof(float));
    A((void **)&m->bpart, nch * m->nl * 256 * sizeof(float));
    A((void **)&m->wpart, nch * 1024 * sizeof(float));
    if (rc) return rc;
    m->cap = rows;
    return MD_OK;
}

int refresh_bf16(mlp_model *m, cudaStream_t st) {
    m->packed = false;
    const ParamMap pm = m->map();
    for (int l = 1; l < m->nl; ++l) {
        const int n = pm.outp(l) * 256;
        k_pack<false><<<(n + 255) / 256, 256, 0, st>>>(m->w + pm.W(l), pm.out(l), pm.outp(l), 1.0f, m->Wf[l]);
        k_pack_t<<<(n + 255) / 256, 256, 0, st>>>(m->w + pm.W(l), pm.out(l), pm.outp(l), m->Wb[l]);
    }
    MD_CUDA_TRY(cudaGetLastError());
    return MD_OK;
}

template <int CS, bool TEST>
int chain_launch(const TrainArgs &a, cudaStream_t st) {
    MD_CUDA_TRY(cudaFuncSetAttribute(k_train_chain<CS, TEST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)TrainShape<CS>::smem));
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CS;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(a.B / 128 * CS);
    cfg.blockDim = dim3(T_THREADS);
    cfg.dynamicSmemBytes = TrainShape<CS>::smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    MD_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_train_chain<CS, TEST>, a));
    return MD_OK;
}

// The three launches of a training step on B rows (B % 128 == 0).  The
// self-test (dbg != 0) ends with the launch that withholds a signal: dbg > 0:
// the chain, its product dbg - 1; dbg < 0: the gradients, a stage that is waited for.
int train_launch(mlp_model *m, const float *X, const float *T, int B, float *loss, const AdamArgs &ad, cudaStream_t st,
                 int dbg = 0, uint64_t wait_ns = GEMM_WAIT_NS) {
    int dev = 0, nsm = 0;
    MD_CUDA_TRY(cudaGetDevice(&dev));
    MD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    TrainArgs t{};
    t.X = X;
    t.T = T;
    t.B = B;
    t.pm = m->map();
    t.shift = make_float4(m->shift[0], m->shift[1], m->shift[2], m->shift[3]);
    t.scale = make_float4(m->scale[0], m->scale[1], m->scale[2], m->scale[3]);
    t.w = m->w;
    for (int l = 1; l < m->nl; ++l) {
        t.Wf[l] = m->Wf[l];
        t.Wb[l] = m->Wb[l];
    }
    t.xf = m->xf;
    t.Z = m->Z;
    t.H = m->H;
    t.dZ = m->dZ;
    t.rowloss = m->rowloss;
    t.inv_batch = 1.0f / (float)B;
    t.status = m->status;
    t.dbg_skip = dbg;
    t.dbg_wait_ns = wait_ns;
    // four CTAs per row block while the device has SMs for them, else two
    // (CTAs beyond the device then queue)
    const bool four = B / 128 * 4 <= nsm;
    int rc = dbg > 0 ? (four ? chain_launch<4, true>(t, st) : chain_launch<2, true>(t, st))
                     : (four ? chain_launch<4, false>(t, st) : chain_launch<2, false>(t, st));
    if (rc || dbg > 0) return rc;
    GradArgs g{};
    g.H = m->H;
    g.dZ = m->dZ;
    g.xf = m->xf;
    g.B = B;
    g.ks = grad_splits(B);
    g.pm = t.pm;
    g.part = m->part;
    g.bpart = m->bpart;
    g.wpart = m->wpart;
    g.status = m->status;
    g.wait_ns = dbg < 0 ? wait_ns : GEMM_WAIT_NS;
    const int nk = B / g.ks / GBK;
    g.dbg_skip = dbg < 0 ? (nk > G_STAGES ? 1 : nk) : 0;
    const int nch = B / GRAD_ROWS;
    MD_CUDA_TRY(cudaFuncSetAttribute(k_train_grads, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GRADS_SMEM));
    k_train_grads<<<grad_tiles(g.pm) * g.ks + grad_sums(g.pm) / 128 * nch, 128, GRADS_SMEM, st>>>(g);
    MD_CUDA_TRY(cudaGetLastError());
    if (dbg < 0) return MD_OK;
    UpdateArgs u{};
    u.pm = t.pm;
    u.part = m->part;
    u.bpart = m->bpart;
    u.wpart = m->wpart;
    u.ks = g.ks;
    u.nch = nch;
    u.w = m->w;
    u.mom = m->mom;
    u.var = m->var;
    for (int l = 1; l < m->nl; ++l) {
        u.Wf[l] = m->Wf[l];
        u.Wb[l] = m->Wb[l];
    }
    u.rowloss = m->rowloss;
    u.B = B;
    u.loss = loss;
    k_train_update<<<(t.pm.count() + 255) / 256 + 1, 256, 0, st>>>(u, ad);
    MD_CUDA_TRY(cudaGetLastError());
    return MD_OK;
}

}  // namespace

extern "C" {

int mlp_create(int32_t n_hidden, int32_t width, int32_t n_classes, const float *shift4,
               const float *scale4, const float *params, mlp_model **out) {
    if (!out || !shift4 || !scale4 || !params || n_hidden < 2 || n_hidden > 15 || width != 256 ||
        n_classes < 2 || n_classes > MLP_MAX_CLASSES)
        return fail(MD_E_ARG, "mlp_create: n_hidden in [2,15], width 256, classes in [2,112]");
    mlp_model *m = new mlp_model();
    m->nl = n_hidden + 1;
    m->ncls = n_classes;
    std::memcpy(m->shift, shift4, sizeof(m->shift));
    std::memcpy(m->scale, scale4, sizeof(m->scale));
    const ParamMap pm = m->map();
    int rc = MD_OK;
    auto A = [&](void **p, size_t bytes) {
        if (rc == MD_OK) rc = malloc_into(m->allocs, p, bytes);
    };
    const size_t np = (size_t)pm.count() * sizeof(float);
    A((void **)&m->w, np);
    A((void **)&m->mom, np);
    A((void **)&m->var, np);
    A((void **)&m->g, np);
    m->Wf.assign(m->nl, nullptr);
    m->Wb = m->Wp = m->Wf;
    for (int l = 0; l < m->nl; ++l) {
        const size_t nw = (size_t)pm.outp(l) * pm.in(l);
        if (l > 0) {
            A((void **)&m->Wf[l], nw * 2);
            A((void **)&m->Wb[l], nw * 2);
            A((void **)&m->Wp[l], (nw + (size_t)pm.outp(l) * 16) * 2);
        } else {
            A((void **)&m->Wp[0], (size_t)pm.outp(0) * 16 * 2);
        }
    }
    A((void **)&m->status, sizeof(int));
    if (rc) {
        mlp_destroy(m);
        return rc;
    }
    cudaMemset(m->mom, 0, np);
    cudaMemset(m->var, 0, np);
    cudaMemset(m->status, 0, sizeof(int));
    rc = mlp_set_params(m, params);
    if (rc) {
        mlp_destroy(m);
        return rc;
    }
    *out = m;
    return MD_OK;
}

void mlp_destroy(mlp_model *m) {
    if (!m) return;
    cudaDeviceSynchronize();
    for (void *p : m->ws) cudaFree(p);
    for (void *p : m->allocs) cudaFree(p);
    delete m;
}

int64_t mlp_param_count(mlp_model *m) { return m ? m->map().count() : 0; }

int mlp_set_params(mlp_model *m, const float *params) {
    if (!m || !params) return fail(MD_E_ARG, "mlp_set_params: NULL argument");
    MD_CUDA_TRY(cudaMemcpy(m->w, params, sizeof(float) * m->map().count(), cudaMemcpyDefault));
    int rc = refresh_bf16(m, nullptr);
    if (rc) return rc;
    MD_CUDA_TRY(cudaDeviceSynchronize());
    return MD_OK;
}

int mlp_get_params(mlp_model *m, float *params) {
    if (!m || !params) return fail(MD_E_ARG, "mlp_get_params: NULL argument");
    MD_CUDA_TRY(cudaDeviceSynchronize());
    MD_CUDA_TRY(cudaMemcpy(params, m->w, sizeof(float) * m->map().count(), cudaMemcpyDefault));
    return MD_OK;
}

int mlp_forward(mlp_model *m, const float *X, int64_t M, float *P_out, void *stream) {
    mdlg::Range range_("mlp_forward");
    if (!m || !X || !P_out || M < 1) return fail(MD_E_ARG, "mlp_forward: bad arguments");
    if ((uintptr_t)X & 15) return fail(MD_E_ARG, "mlp_forward: X must be 16-byte aligned");
    cudaStream_t st = (cudaStream_t)stream;
    if (!m->packed) {
        const ParamMap pm = m->map();
        k_pack0<<<16, 256, 0, st>>>(m->w, m->w + pm.b(0), m->nl > 1 ? 0.5f : 1.0f, m->Wp[0]);
        for (int l = 1; l < m->nl; ++l) {
            const int n = pm.outp(l) * 256;
            const float sc = l < m->nl - 1 ? 0.5f : 1.0f;
            const int nb = pm.outp(l) * 16;   // the bias slice comes first
            k_packb<<<(nb + 255) / 256, 256, 0, st>>>(m->w + pm.b(l), pm.out(l), pm.outp(l), sc, m->Wp[l]);
            k_pack<true><<<(n + 255) / 256, 256, 0, st>>>(m->w + pm.W(l), pm.out(l), pm.outp(l), sc, m->Wp[l] + nb);
        }
        MD_CUDA_TRY(cudaGetLastError());
        m->packed = true;
    }
    FusedArgs a{};
    a.X = X;
    a.M = M;
    a.P = P_out;
    a.ncls = m->ncls;
    a.shift = make_float4(m->shift[0], m->shift[1], m->shift[2], m->shift[3]);
    a.scale = make_float4(m->scale[0], m->scale[1], m->scale[2], m->scale[3]);
    a.nt = m->nl;
    for (int l = 0; l < m->nl; ++l) {
        a.Wp[l] = m->Wp[l];
    }
    a.p_aligned = ((uintptr_t)P_out & 15) == 0;
    a.status = m->status;
    int dev = 0, nsm = 0;   // the calling thread's current device
    MD_CUDA_TRY(cudaGetDevice(&dev));
    MD_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    MD_CUDA_TRY(cudaFuncSetAttribute(k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FUSED_SMEM));
    const long long tiles = (M + 127) / 128;
    const int grid = (int)std::min<long long>(tiles, nsm);
    k_mlp_fused<<<grid, F_THREADS, FUSED_SMEM, st>>>(a);
    MD_CUDA_TRY(cudaGetLastError());
    return MD_OK;
}

int mlp_grad(mlp_model *m, const float *X, const float *T, int32_t B, float *grad_out,
             float *loss_out, void *stream) {
    if (!m || !X || !T || B < 128 || B % 128) return fail(MD_E_ARG, "mlp_grad: batch must be a multiple of 128");
    cudaStream_t st = (cudaStream_t)stream;
    int rc = ensure_ws(m, B);
    if (rc) return rc;
    AdamArgs ad{};
    ad.g = m->g;
    if ((rc = train_launch(m, X, T, B, loss_out, ad, st))) return rc;
    if (grad_out) MD_CUDA_TRY(cudaMemcpyAsync(grad_out, m->g, sizeof(float) * m->map().count(), cudaMemcpyDefault, st));
    return MD_OK;
}

int mlp_train_step(mlp_model *m, const float *X, const float *T, int32_t B, float lr,
                   float *loss_out, void *stream) {
    mdlg::Range range_("mlp_train_step");
    if (!m || !X || !T || B < 128 || B % 128) return fail(MD_E_ARG, "mlp_grad: batch must be a multiple of 128");
    cudaStream_t st = (cudaStream_t)stream;
    int rc = ensure_ws(m, B);
    if (rc) return rc;
    AdamArgs ad{};
    ad.lr = lr;
    ad.b1 = 0.9f;
    ad.b2 = 0.999f;
    ad.eps = 1e-8f;
    ad.c1 = 1.f - powf(ad.b1, (float)(m->adam_t + 1));
    ad.c2 = 1.f - powf(ad.b2, (float)(m->adam_t + 1));
    if ((rc = train_launch(m, X, T, B, loss_out, ad, st))) return rc;
    m->adam_t += 1;
    m->packed = false;
    return MD_OK;
}

int mlp_status(mlp_model *m) {
    if (!m) return fail(MD_E_ARG, "mlp_status: NULL model");
    int s = 0;
    MD_CUDA_TRY(cudaDeviceSynchronize());
    MD_CUDA_TRY(cudaMemcpy(&s, m->status, sizeof(int), cudaMemcpyDeviceToHost));
    if (s) {
        cudaMemset(m->status, 0, sizeof(int));
        return fail(MD_E_TIMEOUT, "tensor-core GEMM wait timed out");
    }
    return MD_OK;
}

int mlp_train_selftest(mlp_model *m, const float *X, const float *T, int32_t B, int32_t where, double limit_s,
                       void *stream) {
    if (!m || !X || !T || B < 128 || B % 128 || where < -1 || where == 0 || where > 2 * (m->nl - 1) ||
        !(limit_s > 0.0) || !(limit_s <= 2.0))
        return fail(MD_E_ARG, "mlp_train_selftest: bad arguments");
    int rc = ensure_ws(m, B);
    if (rc) return rc;
    AdamArgs ad{};
    ad.g = m->g;
    if ((rc = train_launch(m, X, T, B, nullptr, ad, (cudaStream_t)stream, where, (uint64_t)(limit_s * 1e9)))) return rc;
    return mlp_status(m);
}

int bf16_gemm_selftest(const void *A, const void *B, float *C, int32_t M, int32_t N, int32_t K,
                       int32_t *status, double limit_s, void *stream) {
    if (!A || !B || !C || !status || !(limit_s > 0.0) || !(limit_s <= 2.0) || K < 3 * GBK)
        return fail(MD_E_ARG, "bf16_gemm_selftest: bad arguments (K >= 192, 0 < limit_s <= 2)");
    GemmArgs g{};
    g.A = (const bf16 *)A;
    g.B = (const bf16 *)B;
    g.lda = K;
    g.ldb = K;
    g.M = M;
    g.N = N;
    g.K = K;
    g.C = C;
    g.ldc = N;
    g.status = status;
    g.wait_ns = (uint64_t)(limit_s * 1e9);
    g.dbg_skip_commit = 1;   // stage 0
    cudaStream_t st = (cudaStream_t)stream;
    MD_CUDA_TRY(cudaMemsetAsync(status, 0, sizeof(int32_t), st));
    int rc = gemm_launch(g, st);
    if (rc) return rc;
    int32_t h = 0;
    MD_CUDA_TRY(cudaMemcpyAsync(&h, status, sizeof(h), cudaMemcpyDeviceToHost, st));
    MD_CUDA_TRY(cudaStreamSynchronize(st));
    return h ? fail(MD_E_TIMEOUT, "bf16_gemm_selftest: an mbarrier wait ran out (as intended)") : MD_OK;
}

int bf16_gemm_tn(const void *A, const void *B, float *C, int32_t M, int32_t N, int32_t K,
                 int32_t *status, void *stream) {
    if (!A || !B || !C || !status) return fail(MD_E_ARG, "bf16_gemm_tn: NULL argument");
    GemmArgs g{};
    g.A = (const bf16 *)A;
    g.B = (const bf16 *)B;
    g.lda = K;
    g.ldb = K;
    g.M = M;
    g.N = N;
    g.K = K;
    g.C = C;
    g.ldc = N;
    g.status = status;
    return gemm_launch(g, (cudaStream_t)stream);
}

}  // extern "C"
