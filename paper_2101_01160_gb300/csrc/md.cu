// Host side of the MD system: md_init / md_init_batch / md_step / readouts.
//
// One system holds one or more replicas.  md_step enqueues a single
// cooperative launch of the persistent kernel (md_kernels.cuh) that runs all
// requested steps, sampling and cell-list rebuilds on the device; control
// returns to the host only at md_sync or at a readout.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "equilibria.cuh"
#include "md_kernels.cuh"
#include "md_resident.cuh"
#include "md_slab.cuh"

namespace mdlg {

template <typename T>
__global__ void k_init(SysDev S, const double *x, const double *y, const double *vx,
                       const double *vy) {
    using V = typename V2<T>::type;
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot < S.nrep) {
        const RepDev &R = S.reps[slot];
        S.cellcnt[R.cbase + R.nc * R.nc] = R.cap - R.n;
    }
    if (slot >= S.nslots) return;
    const RepDev &R = S.reps[S.gran_rep[slot / GRAN]];
    const int local = slot - R.pbase;
    V *pos = static_cast<V *>(S.pos[0][0]);
    V *vel = static_cast<V *>(S.vel[0]);
    if (local >= R.n) {
        pos[slot] = V{T(0), T(0)};
        vel[slot] = V{T(0), T(0)};
        S.cell[0][slot] = 0u;
        S.pid[0][slot] = -1;
        return;
    }
    const int id = R.ibase + local;
    double X = x[id], Y = y[id];
    X -= R.L * floor(X / R.L);
    Y -= R.L * floor(Y / R.L);
    if (X >= R.L) X -= R.L;
    if (Y >= R.L) Y -= R.L;
    int cx = (int)floor(X / R.h), cy = (int)floor(Y / R.h);
    cx = min(max(cx, 0), R.nc - 1);
    cy = min(max(cy, 0), R.nc - 1);
    pos[slot] = V{(T)(X - (double)cx * R.h), (T)(Y - (double)cy * R.h)};
    vel[slot] = V{(T)vx[id], (T)vy[id]};
    S.cell[0][slot] = (uint32_t)cx | ((uint32_t)cy << 16);
    S.pid[0][slot] = id;
}

// Energy partials of one replica summed in a fixed order by one CTA.
__device__ __forceinline__ void sum_energy_cta(const double *epart, int g0, int g1, double *out4) {
    __shared__ double sh[4][256];
    double a[4] = {0, 0, 0, 0};
    for (int g = g0 + threadIdx.x; g < g1; g += 256)
        for (int k = 0; k < 4; ++k) a[k] += epart[(long long)g * 4 + k];
    for (int k = 0; k < 4; ++k) sh[k][threadIdx.x] = a[k];
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if ((int)threadIdx.x < o)
            for (int k = 0; k < 4; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 4) out4[threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_sum_energy(const double *epart, int g0, int g1, double *out4) {
    sum_energy_cta(epart, g0, g1, out4);
}

// every replica at once, one CTA per replica: the same sums as k_sum_energy
__global__ void k_sum_energy_batch(const double *epart, const RepDev *reps, double *out) {
    const RepDev &R = reps[blockIdx.x];
    sum_energy_cta(epart, R.pbase / 32, (R.pbase + R.cap) / 32, out + 4 * (size_t)blockIdx.x);
}

struct FeqArgs {
    const int32_t *hist;          // [MD_NBLK][nb] of one (rep, lg, dx)
    const unsigned long long *ovf;
    const double *mom;            // [ngran32][n_lg][2]
    int g0, g1, n_lg, lg, nb, W, sym;
    double n;                     // particles of the replica
    long long nwin;
    long long wblk[MD_NBLK];      // windows per block
    double dx_eff;
    double *out;                  // [nb] P, [nb] stderr, [8] stats
};

// Normalised measured equilibrium (Eq. theory_feq per particle), batch-means
// error bars over blocks of windows, optional symmetric-set averaging
// (Sec. 5), moments mu2, mu4 and a^2 (Eq. a2_n_ua).  One CTA.
constexpr int FEQ_THREADS = 256;

// Sums of the moment partials of groups [g0, g1), in thread 0 (both f_eq
// kernels: the same threads, strides and tree, so the same bits).
__device__ __forceinline__ void feq_moments(const double *mom, int g0, int g1, int n_lg, int lg, double &m2, double &m4) {
    const double2 *p = reinterpret_cast<const double2 *>(mom) + lg;
    m2 = m4 = 0.0;
#pragma unroll 8
    for (int g = g0 + (int)threadIdx.x; g < g1; g += FEQ_THREADS) {
        const double2 m = p[(long long)g * n_lg];
        m2 += m.x;
        m4 += m.y;
    }
    block_sum2(m2, m4);
}

__global__ void __launch_bounds__(FEQ_THREADS) k_feq_measured(FeqArgs A) {
    double m2, m4;
    feq_moments(A.mom, A.g0, A.g1, A.n_lg, A.lg, m2, m4);
    const double samples = A.n * (double)A.nwin;
    const int side = 2 * A.W + 1;
    for (int i = threadIdx.x; i < A.nb; i += blockDim.x) {
        int mem[8];
        int nm = 0;
        if (A.sym) {
            const int a = abs(i % side - A.W), b = abs(i / side - A.W);
            const int lo = min(a, b), hi = max(a, b);
            for (int j = 0; j < A.nb && nm < 8; ++j) {
                const int c = abs(j % side - A.W), d = abs(j / side - A.W);
                if (min(c, d) == lo && max(c, d) == hi) mem[nm++] = j;
            }
        } else {
            mem[nm++] = i;
        }
        long long tot = 0;
        double pb[MD_NBLK];
        for (int b = 0; b < MD_NBLK; ++b) {
            long long hb = 0;
            for (int m = 0; m < nm; ++m) hb += A.hist[b * A.nb + mem[m]];
            tot += hb;
            pb[b] = A.wblk[b] > 0 ? (double)hb / ((double)nm * A.n * (double)A.wblk[b]) : 0.0;
        }
        const double P = samples > 0 ? (double)tot / ((double)nm * samples) : 0.0;
        double num = 0.0, wsum = 0.0;
        int used = 0;
        for (int b = 0; b < MD_NBLK; ++b) {
            if (A.wblk[b] <= 0) continue;
            const double w = (double)A.wblk[b];
            num += w * w * (pb[b] - P) * (pb[b] - P);
            wsum += w;
            ++used;
        }
        A.out[i] = P;
        A.out[A.nb + i] = used > 1 ? sqrt(num / (wsum * wsum) * (double)used / (double)(used - 1)) : 0.0;
    }
    if (threadIdx.x == 0) {
        double *st = A.out + 2 * A.nb;
        const double mu2 = samples > 0 ? m2 / (2.0 * samples) : 0.0;
        const double mu4 = samples > 0 ? m4 / (2.0 * samples) : 0.0;
        st[0] = mu2;
        st[1] = mu4;
        st[2] = mu2 / (A.dx_eff * A.dx_eff);
        st[3] = (double)(*A.ovf);
    }
}

__global__ void k_hist_total(const int32_t *hist, int nb, long long *out) {
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        long long t = 0;
        for (int b = 0; b < MD_NBLK; ++b) t += hist[b * nb + i];
        out[i] = t;
    }
}

__global__ void k_copy_snapshot(const uint32_t *sc, const void *so, int f64, long long ntot,
                                const int32_t *nc_of_id, int32_t *cell, void *ox, void *oy) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ntot) return;
    const uint32_t pk = sc[i];
    cell[i] = (int32_t)(pk >> 16) * nc_of_id[i] + (int32_t)(pk & 0xffffu);
    if (f64) {
        const double2 v = static_cast<const double2 *>(so)[i];
        static_cast<double *>(ox)[i] = v.x;
        static_cast<double *>(oy)[i] = v.y;
    } else {
        const float2 v = static_cast<const float2 *>(so)[i];
        static_cast<float *>(ox)[i] = v.x;
        static_cast<float *>(oy)[i] = v.y;
    }
}

__global__ void k_nc_of_id(SysDev S, int32_t *nc_of_id) {
    const int slot = blockIdx.x * blockDim.x + threadIdx.x;
    if (slot >= S.nslots) return;
    const RepDev &R = S.reps[S.gran_rep[slot / GRAN]];
    const int local = slot - R.pbase;
    if (local < R.n) nc_of_id[R.ibase + local] = R.nc;
}


// ---------------------------------------------------------------- batched f_eq stage
// For every replica, on the device, one CTA each: the measured equilibrium
// (Eq. theory_feq per particle, optionally averaged over symmetric sets),
// the moments mu2, mu4 and a^2 (Eq. a2_n_ua), lambda from Eq. (lambda_eq)
// (root 2), the Gaussian (Eq. feq_gaussian) and WSG (Eq. f_eq_wsg)
// equilibria at that a^2 and lambda, and their distance to the measured one
// (max |difference| and Eq. kullback_leibler).
//
// What bounds it is the FP64 pipe (a warp instruction every 15 clocks of an
// SM) and, for few replicas, the chain of its phases.  So the WSG sum takes
// the strided window (at most 137 terms, wsg_stride), a term's exponentials
// and error functions are evaluated at |v| = 1 .. W+1 only (u = 0: both
// equilibria depend on |vx|, |vy|), one (term, point) per thread, the 2D
// products are summed once per symmetric set {|vx|, |vy|}, and the Gaussian
// is one more row of the table.  Measured: 256 replicas 291 -> 57 us, one
// replica of 262,144 particles 123 -> 25 us (three kernels before).
constexpr int FEQB_THREADS = FEQ_THREADS;
constexpr int FEQB_STATS = 16;
constexpr int FEQB_SPLIT = 8;     // partial sums over the terms per symmetric set

struct FeqBatchArgs {
    const RepDev *reps;
    const int32_t *hist;           // [nrep][n_lg][n_dx][MD_NBLK][nb]
    const unsigned long long *ovf; // [nrep][n_lg][n_dx]
    const double *mom;             // [ngran32][n_lg][2]
    int n_lg, n_dx, lg, dxi, nb, W, sym;
    long long nwin;
    double *out;                   // [nrep][3 nb + FEQB_STATS]
};

// Sums of a and b over the CTA (fixed tree), in every thread.
__device__ __forceinline__ void feqb_sum2(double &a, double &b, double *s_r) {
    block_sum2(a, b);
    if (threadIdx.x == 0) {
        s_r[0] = a;
        s_r[1] = b;
    }
    __syncthreads();
    a = s_r[0];
    b = s_r[1];
    __syncthreads();
}

__global__ void __launch_bounds__(FEQB_THREADS) k_feq_batch(FeqBatchArgs A) {
    constexpr int ROWS = WSG_MAX_TERMS + 1;             // terms of a chunk and the Gaussian
    constexpr int PTS = MD_MAX_W + 2;                   // |v| = 0 .. W + 1
    constexpr int SETS = (MD_MAX_W + 1) * (MD_MAX_W + 2) / 2;
    __shared__ double s_var[ROWS], s_w[ROWS], s_E[ROWS][PTS], s_R[ROWS][PTS];
    __shared__ double s_part[SETS * FEQB_SPLIT], s_wsg[SETS], s_G[MD_MAX_W + 1], s_par[4], s_r[2];
    __shared__ long long s_tot[(2 * MD_MAX_W + 1) * (2 * MD_MAX_W + 1)];
    const int r = blockIdx.x, tid = threadIdx.x;
    const RepDev &R = A.reps[r];
    double *out = A.out + (long long)r * (3 * A.nb + FEQB_STATS);
    const int32_t *hist = A.hist + ((((long long)r * A.n_lg + A.lg) * A.n_dx + A.dxi) * MD_NBLK) * A.nb;
    const double samples = (double)R.n * (double)A.nwin;
    const int side = 2 * A.W + 1, W = A.W;
    // counts of every class over the blocks, requested before the moments
    for (int i = tid; i < A.nb; i += FEQB_THREADS) {
        int v[MD_NBLK];
#pragma unroll
        for (int b = 0; b < MD_NBLK; ++b) v[b] = hist[b * A.nb + i];
        long long t = 0;
#pragma unroll
        for (int b = 0; b < MD_NBLK; ++b) t += v[b];
        s_tot[i] = t;
    }
    // moments, a^2, lambda
    double m2, m4;
    feq_moments(A.mom, R.pbase / 32, (R.pbase + R.cap) / 32, A.n_lg, A.lg, m2, m4);
    if (tid == 0) {
        const double mu2 = samples > 0 ? m2 / (2.0 * samples) : 0.0;
        const double mu4 = samples > 0 ? m4 / (2.0 * samples) : 0.0;
        const double dx = R.dxl[A.dxi];
        double lam = 0.0, st = 0.0;
        const double k = mu2 > 0 ? mu4 / (mu2 * mu2) : 0.0;
        if (!(k > 3.0)) {
            st = 1.0;
        } else if (k > 3.75) {
            lam = 1.0;
            st = 2.0;
        } else {
            lam = lambda_root(mu2, mu4, 2);
            if (lam > 1e5) {
                lam = 1e5;   // the mixture is then a single Gaussian to ~1e-5
                st = 3.0;
            }
        }
        s_par[1] = mu2 / (dx * dx);
        s_par[2] = lam;
        out[3 * A.nb + 0] = mu2;
        out[3 * A.nb + 1] = mu4;
        out[3 * A.nb + 2] = s_par[1];
        out[3 * A.nb + 3] = lam;
        out[3 * A.nb + 8] = (double)A.nwin;
        out[3 * A.nb + 9] = samples;
        out[3 * A.nb + 10] = (double)A.ovf[((long long)r * A.n_lg + A.lg) * A.n_dx + A.dxi];
        out[3 * A.nb + 11] = dx;
        out[3 * A.nb + 12] = st;
    }
    __syncthreads();
    const double a2 = s_par[1], lam = s_par[2];
    const int nsets = (W + 1) * (W + 2) / 2;             // (lo <= hi): index hi (hi + 1) / 2 + lo
    const int terms = wsg_terms(lam), cmin = wsg_cmin(lam), dc = wsg_stride(lam);
    for (int e = tid; e < nsets; e += FEQB_THREADS) s_wsg[e] = 0.0;
    for (int j0 = 0; j0 < terms && a2 > 0; j0 += WSG_MAX_TERMS) {
        // rows 0 .. nt-1: terms of the chunk; row nt: the Gaussian
        const int nt = min(WSG_MAX_TERMS, terms - j0);
        for (int t = tid; t <= nt; t += FEQB_THREADS) {
            const int c = cmin + (j0 + t) * dc;
            s_w[t] = t < nt ? (double)dc * poisson_weight(c, lam) : 0.0;
            s_var[t] = t < nt ? a2 * ((double)c + 1.0) / (lam + 1.0) : a2;
            s_E[t][0] = 1.0;
            s_R[t][0] = 0.0;
        }
        __syncthreads();
        for (int e = tid; e < (nt + 1) * (W + 1); e += FEQB_THREADS) {
            const int t = e / (W + 1), q = e % (W + 1) + 1;
            const double p = (double)q, var2 = 2.0 * s_var[t];
            s_E[t][q] = exp(-(p * p) / var2);
            s_R[t][q] = erf(p / sqrt(var2));
        }
        __syncthreads();
        // 1D factors (cell_gauss_1d) of |v| = 0 .. W, in place over E: a pass
        // to registers, then the write
        constexpr int FPT = (ROWS * (MD_MAX_W + 1) + FEQB_THREADS - 1) / FEQB_THREADS;
        double f[FPT];
#pragma unroll
        for (int k = 0; k < FPT; ++k) {
            const int e = tid + k * FEQB_THREADS;
            if (e < (nt + 1) * (W + 1)) {
                const int t = e / (W + 1), v = e % (W + 1), lo = v ? v - 1 : 1;
                const double u = (double)v, um = u - 1.0, up = u + 1.0;
                const double norm = sqrt(s_var[t]) * 0.39894228040143267794;
                const double E = s_E[t][lo] - 2.0 * s_E[t][v] + s_E[t][v + 1];
                const double Rm = v ? s_R[t][lo] : -s_R[t][1], eu = s_R[t][v];
                f[k] = norm * E + 0.5 * um * (Rm - eu) + 0.5 * up * (s_R[t][v + 1] - eu);
            }
        }
        __syncthreads();
#pragma unroll
        for (int k = 0; k < FPT; ++k) {
            const int e = tid + k * FEQB_THREADS;
            if (e < (nt + 1) * (W + 1)) s_E[e / (W + 1)][e % (W + 1)] = f[k];
        }
        __syncthreads();
        for (int e = tid; e < nsets * FEQB_SPLIT; e += FEQB_THREADS) {
            const int set = e / FEQB_SPLIT, sp = e % FEQB_SPLIT;
            int hi = 0;
            while ((hi + 1) * (hi + 2) / 2 <= set) ++hi;
            const int lo = set - hi * (hi + 1) / 2;
            double acc = 0.0;
            for (int t = sp; t < nt; t += FEQB_SPLIT) acc += s_w[t] * (s_E[t][lo] * s_E[t][hi]);
            s_part[e] = acc;
        }
        if (tid <= W) s_G[tid] = s_E[nt][tid];
        __syncthreads();
        for (int e = tid; e < nsets; e += FEQB_THREADS) {
            double acc = s_wsg[e];
            for (int sp = 0; sp < FEQB_SPLIT; ++sp) acc += s_part[e * FEQB_SPLIT + sp];
            s_wsg[e] = acc;
        }
        __syncthreads();
    }
    __syncthreads();
    double mg = 0.0, kg = 0.0, mw = 0.0, kw = 0.0, sum = 0.0, zero = 0.0;
    for (int i = tid; i < A.nb; i += FEQB_THREADS) {
        const int x = abs(i % side - W), y = abs(i / side - W);
        const int lo = min(x, y), hi = max(x, y);
        long long tot = 0;
        int nm = 1;
        if (A.sym) {
            nm = 0;
            for (int q = 0; q < 8; ++q) {                 // (+-lo, +-hi), (+-hi, +-lo), each once
                const int sx = (q & 1 ? -1 : 1) * (q & 4 ? hi : lo), sy = (q & 2 ? -1 : 1) * (q & 4 ? lo : hi);
                if (((q & 1) && sx == 0) || ((q & 2) && sy == 0) || ((q & 4) && lo == hi)) continue;
                tot += s_tot[(sy + W) * side + sx + W];
                ++nm;
            }
        } else {
            tot = s_tot[i];
        }
        const double P = samples > 0 ? (double)tot / ((double)nm * samples) : 0.0;
        const double G = a2 > 0 ? s_G[x] * s_G[y] : 0.0;
        const double Wg = s_wsg[hi * (hi + 1) / 2 + lo];
        out[i] = P;
        out[A.nb + i] = G;
        out[2 * A.nb + i] = Wg;
        mg = fmax(mg, fabs(P - G));
        mw = fmax(mw, fabs(P - Wg));
        if (P > 0.0) {
            kg += P * log(P / G);
            kw += P * log(P / Wg);
        }
        sum += P;
    }
    feqb_sum2(kg, kw, s_r);
    feqb_sum2(sum, zero, s_r);
    for (int o = 16; o > 0; o >>= 1) {
        mg = fmax(mg, __shfl_xor_sync(0xffffffffu, mg, o));
        mw = fmax(mw, __shfl_xor_sync(0xffffffffu, mw, o));
    }
    if ((tid & 31) == 0) {
        s_part[tid >> 5] = mg;
        s_part[32 + (tid >> 5)] = mw;
    }
    __syncthreads();
    if (tid == 0) {
        for (int w = 1; w < FEQB_THREADS / 32; ++w) {
            mg = fmax(mg, s_part[w]);
            mw = fmax(mw, s_part[32 + w]);
        }
        out[3 * A.nb + 4] = mg;
        out[3 * A.nb + 5] = kg;
        out[3 * A.nb + 6] = mw;
        out[3 * A.nb + 7] = kw;
        out[3 * A.nb + 13] = sum;
    }
}

// ---------------------------------------------------------------- bootstrap
// Block-bootstrap standard error of the measured equilibrium of every
// replica: the error-bar blocks of windows that hold data are resampled with
// replacement (as many draws as used blocks), each resample's P_i = drawn
// counts / (n * drawn windows), optionally averaged over i's symmetric set;
// sigma_i = sample standard deviation over the B resamples (divisor B - 1).
// Draw c of replica rep is SplitMix64 (Steele, Lea and Flood 2014) used as a
// counter-based generator: the output function of seed + (c + 1) * gamma,
// gamma = 0x9e3779b97f4a7c15, c = ((rep * 2^20 + b) * 64 + k) for slot k of
// resample b; block = (draw >> 32) * used >> 32.
//
// A resample's counts are sum_u m_u h[u][i] over the used blocks u, m_u how
// often it drew u, so the draws are made once per resample (not once per
// class) and a class costs nu integer multiply-adds in shared memory.  With
// symmetric sets only one class of each set is computed (15 of 81 at W = 4).
// The P of a chunk of resamples are formed by all threads; one thread per
// class then adds them in resample order, so sigma has the bits of the plain
// loop.  All P are kept in shared memory between the mean and the deviation
// pass where they fit (BOOT_KEEP_BYTES), else they are formed again.
// Grid: (replica, tile of BOOT_CLASSES classes).  What bounds it: the FP64
// divisions (one per resample and class) and the class threads' chains of
// additions.  256 replicas x 200 resamples x 32 blocks, symmetric sets: the
// f_eq stage with its error bars takes 0.46 ms instead of 6.90 ms, of which
// 6.51 ms went to this kernel while every class repeated the draws.
__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t c) {
    uint64_t z = seed + (c + 1u) * 0x9e3779b97f4a7c15ull;
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

struct BootArgs {
    const RepDev *reps;
    const int32_t *hist;   // [nrep][n_lg][n_dx][MD_NBLK][nb]
    int n_lg, n_dx, lg, dxi, nb, W, sym, B;
    uint64_t seed;
    long long wblk[MD_NBLK];
    double *sigma;         // [nrep][nb]
};

constexpr int BOOT_THREADS = 256;
constexpr int BOOT_CHUNK = 64;       // resamples per chunk (a multiple of 4)
constexpr int BOOT_CLASSES = 64;     // classes per CTA
constexpr size_t BOOT_KEEP_BYTES = 100 * 1024;

// Classes computed: all, or one per symmetric set (|vx| <= |vy| pairs).
inline int boot_classes(int W, bool sym) { return sym ? (W + 1) * (W + 2) / 2 : (2 * W + 1) * (2 * W + 1); }
inline size_t boot_p_bytes(int rows, int ncls) { return sizeof(double) * (size_t)rows * std::min(ncls, BOOT_CLASSES); }

// Counts of 4 resamples of one class: acc[q] = sum_u mult[u][b + q] H[u][i].
// IT = int where every sum fits 31 bits, long long otherwise.
template <typename IT>
__device__ __forceinline__ void boot_counts(const long long *H, int ct, int i, const int *mult, int b, int nu,
                                            long long (&out)[4]) {
    IT acc[4] = {0, 0, 0, 0};
    for (int u = 0; u < nu; ++u) {
        const IT h = (IT)H[u * ct + i];
        const int4 m = *reinterpret_cast<const int4 *>(&mult[u * BOOT_CHUNK + b]);
        acc[0] += (IT)m.x * h;
        acc[1] += (IT)m.y * h;
        acc[2] += (IT)m.z * h;
        acc[3] += (IT)m.w * h;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) out[q] = (long long)acc[q];
}

__global__ void __launch_bounds__(BOOT_THREADS) k_feq_bootstrap(BootArgs A, int ncls, int keep) {
    extern __shared__ __align__(16) double s_P[];   // [keep ? B : BOOT_CHUNK][ct]
    __shared__ long long s_H[MD_NBLK * BOOT_CLASSES];
    __shared__ __align__(16) int s_mult[MD_NBLK * BOOT_CHUNK];
    __shared__ double s_ws[BOOT_CHUNK];
    __shared__ double s_dn[BOOT_CLASSES];           // members * n of each class
    __shared__ int s_used[MD_NBLK];
    __shared__ int s_nu, s_wide;
    const int r = blockIdx.x, tid = threadIdx.x;
    const int i0 = blockIdx.y * BOOT_CLASSES, ct = min(BOOT_CLASSES, ncls - i0);
    const int side = 2 * A.W + 1;
    if (tid == 0) {
        int nu = 0;
        for (int k = 0; k < MD_NBLK; ++k)
            if (A.wblk[k] > 0) s_used[nu++] = k;
        s_nu = nu;
        s_wide = 0;
    }
    __syncthreads();
    const int nu = s_nu;
    const double n = (double)A.reps[r].n;
    const int32_t *h = A.hist + ((((long long)r * A.n_lg + A.lg) * A.n_dx + A.dxi) * MD_NBLK) * A.nb;
    // block counts of the tile's classes; a symmetric set's members are the
    // (+-a, +-b), (+-b, +-a) cells, each counted once
    for (int e = tid; e < ct * nu; e += BOOT_THREADS) {
        const int c = e % ct, u = e / ct;
        const int32_t *hu = h + (long long)s_used[u] * A.nb;
        long long t = 0;
        int nm = 1;
        if (A.sym) {
            int b = 0;                              // set (a, b), a <= b: index b (b + 1) / 2 + a
            while ((b + 1) * (b + 2) / 2 <= i0 + c) ++b;
            const int a = i0 + c - b * (b + 1) / 2;
            nm = 0;
            for (int q = 0; q < 8; ++q) {
                const int x = (q & 1 ? -1 : 1) * (q & 4 ? b : a), y = (q & 2 ? -1 : 1) * (q & 4 ? a : b);
                const bool twice = ((q & 1) && x == 0) || ((q & 2) && y == 0) || ((q & 4) && a == b);
                if (twice) continue;
                t += hu[(y + A.W) * side + x + A.W];
                ++nm;
            }
        } else {
            t = hu[i0 + c];
        }
        s_H[u * ct + c] = t;
        if (t > (1ll << 31) / (MD_NBLK + 1)) s_wide = 1;   // MD_NBLK draws of it could pass 31 bits
        if (u == 0) s_dn[c] = (double)nm * n;
    }
    __syncthreads();
    const bool wide = s_wide != 0;
    double mean = 0.0, ss = 0.0;                    // of class tid, tid < ct
    for (int pass = 0; pass < 2 && nu > 0; ++pass) {
        for (int b0 = 0; b0 < A.B; b0 += BOOT_CHUNK) {
            const int nbr = min(BOOT_CHUNK, A.B - b0);
            double *P = s_P + (keep ? (size_t)b0 * ct : 0);
            if (pass == 0 || !keep) {
                for (int e = tid; e < nu * BOOT_CHUNK; e += BOOT_THREADS) s_mult[e] = 0;
                __syncthreads();
                for (int e = tid; e < nbr * nu; e += BOOT_THREADS) {
                    const int b = e / nu, k = e % nu;
                    const uint64_t c = (((uint64_t)r << 20) + (uint64_t)(b0 + b)) * 64u + (uint64_t)k;
                    const uint64_t x = splitmix64(A.seed, c);
                    atomicAdd(&s_mult[(int)(((x >> 32) * (uint64_t)nu) >> 32) * BOOT_CHUNK + b], 1);
                }
                __syncthreads();
                if (tid < nbr) {
                    long long ws = 0;
                    for (int u = 0; u < nu; ++u) ws += (long long)s_mult[u * BOOT_CHUNK + tid] * A.wblk[s_used[u]];
                    s_ws[tid] = (double)ws;
                }
                __syncthreads();
                for (int e = tid; e < (nbr + 3) / 4 * ct; e += BOOT_THREADS) {
                    const int i = e % ct, b = e / ct * 4;
                    long long hs[4];
                    if (wide)
                        boot_counts<long long>(s_H, ct, i, s_mult, b, nu, hs);
                    else
                        boot_counts<int>(s_H, ct, i, s_mult, b, nu, hs);
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (b + q < nbr) P[(size_t)(b + q) * ct + i] = (double)hs[q] / (s_dn[i] * s_ws[b + q]);
                }
                __syncthreads();
            }
            if (tid < ct) {
                if (pass == 0) {
#pragma unroll 8
                    for (int b = 0; b < nbr; ++b) mean += P[(size_t)b * ct + tid];
                } else {
#pragma unroll 8
                    for (int b = 0; b < nbr; ++b) {
                        const double d = P[(size_t)b * ct + tid] - mean;
                        ss = __dadd_rn(ss, __dmul_rn(d, d));   // rounded as the plain definition
                    }
                }
            }
            if (!keep) __syncthreads();             // the chunk's buffer is written again
        }
        if (pass == 0) mean /= (double)A.B;
    }
    if (tid < ct) s_dn[tid] = nu > 0 ? sqrt(ss / (double)(A.B - 1)) : 0.0;
    __syncthreads();
    double *out = A.sigma + (long long)r * A.nb;
    for (int j = tid; j < A.nb; j += BOOT_THREADS) {
        int c = j;
        if (A.sym) {
            const int x = abs(j % side - A.W), y = abs(j / side - A.W);
            const int lo = min(x, y), hi = max(x, y);
            c = hi * (hi + 1) / 2 + lo;
        }
        if (c >= i0 && c < i0 + ct) out[j] = s_dn[c - i0];
    }
}

}  // namespace mdlg

using namespace mdlg;

struct md_system {
    int prec = 0, nrep = 0, W = 0, nb = 0, n_lg = 0, n_dx = 0, block_windows = 1;
    int lg_every[MD_MAX_LG] = {0};
    long long n_equil = 0;
    std::vector<RepDev> reps;
    long long ntot = 0;
    int nslots = 0, total_cells = 0;
    cudaStream_t st = nullptr;
    int dev = 0, nsm = 1;
    int block = 256, grid = 1, ppt = 1, K = 16, stage = 1;
    long long chunk_cap = 0;
    int4 *d_chunks = nullptr;
    size_t smem = 0;
    long long step = 0;
    int phase_half = 0;
    std::vector<void *> allocs;
    SysDev sd{};
    RepDev *d_reps = nullptr;
    int32_t *d_gran = nullptr;
    Control *d_ctl = nullptr;
    int *h_status = nullptr;     // pinned: the landing place of Control::status .. slab_ends
    double *d_epart = nullptr;
    double *d_small = nullptr;   // readout scratch (2*nb + 8 doubles, 4 energy)
    long long *d_hist64 = nullptr;
    int32_t *d_nc_of_id = nullptr;
    // resident engine (md_tune staging 4): plan, buffers, launch shape; the
    // global engine's cell lists need a sort-only rebuild after its launches
    int engine = 0;                   // 0 = k_md_persistent, 1 = k_md_resident
    bool needs_sort = false;
    // the neighbour lists' layout depends on the launch shape (staged: slot
    // order; global: sorted within each chunk of the chunk table), so a new
    // shape's first launch rebuilds them (sort only)
    bool lists_valid = false;
    // The rebuild count does not depend on the engine: it includes the sort of
    // a new launch shape's first step (shape_new) and the sort behind a
    // resident launch or a loaded checkpoint (sort_counts), and no sort that
    // is made only because the slab engine ran
    bool shape_new = false, sort_counts = false;
    // slab engine (a single replica): its plan and buffers (slab_ok: it has
    // one), whether md_step may take it, and whether the state is as its last
    // launch left it
    SlabDev sl{};
    size_t slab_smem = 0;
    bool slab_ok = false, slab_on = true, slab_last = false;
    // A state that outgrows the slabs' room makes every slab launch a detour: after
    // a synchronisation that finds one ended early, the next slab_wait calls that
    // would take the engine run globally; twice as many after each such try
    int slab_ends = 0, slab_wait = 0, slab_backoff = 0;
    bool slab_tried = false;     // a slab launch since the last synchronisation
    std::vector<void *> res_allocs;
    ResDev rd{};
    int res_grid = 0;
    size_t res_smem = 0;
    int res_slabs = 0, res_max_g = 0;
    std::vector<ResJob> res_jobs;     // the plan's slabs, in device order
    std::vector<double> res_cost;     // measured per-replica slab times of the current plan, if any
};

namespace {

int dalloc(md_system *s, void **p, size_t bytes) {
    if (bytes == 0) bytes = 16;
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaSuccess) {
        *p = nullptr;
        return fail(MD_E_NOMEM, "cudaMalloc(%zu): %s", bytes, cudaGetErrorString(e));
    }
    s->allocs.push_back(*p);
    return MD_OK;
}

// staging 3 = global staging with the full-occupancy register budget (FP32
// only; in FP64 it is the same kernel as staging 2)
const void *persistent_fn(int prec, int block, int stage) {
    if (prec == MD_FP64)
        return block == 128 ? (const void *)k_md_persistent<double, 128, false>
                            : (const void *)k_md_persistent<double, 256, false>;
    if (stage == 3)
        return block == 128 ? (const void *)k_md_persistent<float, 128, true>
                            : (const void *)k_md_persistent<float, 256, true>;
    return block == 128 ? (const void *)k_md_persistent<float, 128, false>
                        : (const void *)k_md_persistent<float, 256, false>;
}

// Per-replica constants from the parameters (slot, cell and id bases are
// set by the caller).
RepDev make_rep(const md_params &q, int prec, int n_dx) {
    RepDev R{};
    R.nc = (int)std::floor(q.box_L / (q.rc + q.skin));
    double h = q.box_L / R.nc;
    if (prec == MD_FP32_CELLOFF) h = (double)(float)h;
    R.h = h;
    R.L = (double)R.nc * h;
    R.n = (int)q.n;
    R.cap = (int)((q.n + SLOT_PAD - 1) / SLOT_PAD * SLOT_PAD);
    R.dt = q.dt;
    R.hk = q.dt / (2.0 * q.mass);
    R.rc2 = q.rc * q.rc;
    R.eps = q.eps;
    R.sig2 = q.sigma * q.sigma;
    const double sc2 = q.sigma * q.sigma / (q.rc * q.rc), sc6 = sc2 * sc2 * sc2;
    R.vshift = 4.0 * q.eps * (sc6 * sc6 - sc6);
    R.mass = q.mass;
    R.rv2 = (q.rc + q.skin) * (q.rc + q.skin);
    R.half_skin = 0.5 * q.skin;
    for (int d = 0; d < n_dx; ++d) {
        R.lx[d] = q.lx[d];
        R.dxl[d] = R.L / (double)q.lx[d];
        R.dxl_invf[d] = (float)(1.0 / R.dxl[d]);
    }
    R.hf = (float)h;
    R.dtf = (float)R.dt;
    R.hkf = (float)R.hk;
    R.rc2f = (float)R.rc2;
    R.epsf = (float)R.eps;
    R.sig2f = (float)R.sig2;
    R.rv2f = (float)R.rv2;
    return R;
}

// ---- resident engine plan -------------------------------------------------
// Cuts every replica into g slabs of whole MD-cell rows, the fewest that fit
// one CTA's shared memory each with room to spare (particles 1.2x the
// expected count of the largest slab plus 64, halo rows twice the mean row
// population plus 64, list entries 1.8x the mean neighbour count within
// rc + skin), then deals the slabs to `grid` CTAs by list scheduling: the
// replicas in order of decreasing g and estimated time, each on the
// contiguous CTA range that frees up first.  Every CTA runs its slabs in
// order of their planned start, so the slabs of one replica meet in the
// same order on all their CTAs (no cycle of waits).
struct ResPlan {
    std::vector<ResJob> jobs;        // by CTA, in execution order
    std::vector<int32_t> start;      // [grid + 1]
    int hmax = 0, slabs = 0, max_g = 0;
    double makespan = 0.0;
};

static int round_up(long long v, int m) { return (int)((v + m - 1) / m * m); }

int plan_resident(const std::vector<RepDev> &all, int grid, size_t avail, ResPlan &P,
                  const std::vector<double> *measured = nullptr) {
    struct Rep {
        int r, g, p_cap, h_cap;
        double cost;
    };
    std::vector<Rep> reps;
    for (int r = 0; r < (int)all.size(); ++r) {
        const RepDev &R = all[r];
        const double dens = (double)R.n / (R.L * R.L);
        const double cbar = M_PI * R.rv2 * dens;
        const double rowpop = (double)R.n / R.nc;
        Rep best{r, 0, 0, 0, 0.0};
        for (int g = 1; g <= 1024; ++g) {
            if (g > 1 && (R.nc / g < 2 || g > R.cap / 32)) break;
            const int rows = (R.nc + g - 1) / g;
            if ((g == 1 ? R.nc : rows + 2) > RES_NCC) continue;
            const double pmax = (double)R.n * rows / R.nc;
            const double want = 1.2 * pmax + 64.0;
            if (want > RES_PCAP) continue;
            const int p_cap = std::min(RES_PCAP, round_up((long long)std::ceil(want), 32));
            const int h_cap = g == 1 ? 0 : std::min(4096, round_up((long long)std::ceil(2.0 * rowpop + 64.0), 32));
            if (p_cap + 2 * h_cap > (int)RES_IDX + 1) continue;   // 14-bit list indices
            const long long e_need = (long long)std::ceil(1.8 * cbar * p_cap) + 256;
            if (res_slab_bytes(p_cap, h_cap, (int)std::min<long long>(e_need, 1 << 30)) > avail) continue;
            best = Rep{r, g, p_cap, h_cap, pmax * (40.0 + 14.0 * cbar) + (g > 1 ? 4000.0 : 0.0)};
            // a measured time of the replica's slabs replaces the model
            if (measured && r < (int)measured->size() && (*measured)[r] > 0.0) best.cost = (*measured)[r];
            break;
        }
        if (best.g == 0)
            return fail(MD_E_LIMIT, "resident engine: replica %d (n = %d, %d cell rows) fits no slab plan", r, R.n,
                        R.nc);
        reps.push_back(best);
    }
    std::stable_sort(reps.begin(), reps.end(), [](const Rep &a, const Rep &b) {
        return a.g != b.g ? a.g > b.g : a.cost > b.cost;
    });
    std::vector<double> free_at(grid, 0.0);
    struct Placed {
        double t;
        ResJob j;
    };
    std::vector<std::vector<Placed>> per_cta(grid);
    P.hmax = 32;
    P.slabs = 0;
    P.max_g = 0;
    for (const Rep &q : reps) {
        if (q.g > grid) return fail(MD_E_LIMIT, "resident engine: replica %d needs %d CTAs > %d", q.r, q.g, grid);
        int c0 = 0;
        double best_t = 1e300, best_idle = 1e300;
        for (int c = 0; c + q.g <= grid; ++c) {
            double t = 0.0;
            for (int k = 0; k < q.g; ++k) t = std::max(t, free_at[c + k]);
            double idle = 0.0;
            for (int k = 0; k < q.g; ++k) idle += t - free_at[c + k];
            if (t < best_t || (t == best_t && idle < best_idle)) {
                best_t = t;
                best_idle = idle;
                c0 = c;
            }
        }
        const RepDev &R = all[q.r];
        for (int k = 0; k < q.g; ++k) {
            ResJob j;
            j.rep = q.r;
            j.g = q.g;
            j.k = k;
            j.r0 = (int)((long long)k * R.nc / q.g);
            j.r1 = (int)((long long)(k + 1) * R.nc / q.g);
            j.p_cap = q.p_cap;
            j.h_cap = q.h_cap;
            j.cta0 = c0;
            per_cta[c0 + k].push_back(Placed{best_t, j});
            free_at[c0 + k] = best_t + q.cost;
        }
        P.hmax = std::max(P.hmax, q.h_cap);
        P.slabs += q.g;
        P.max_g = std::max(P.max_g, q.g);
    }
    P.jobs.clear();
    P.start.assign(grid + 1, 0);
    P.makespan = 0.0;
    for (int c = 0; c < grid; ++c) {
        std::stable_sort(per_cta[c].begin(), per_cta[c].end(),
                         [](const Placed &a, const Placed &b) { return a.t < b.t; });
        P.start[c] = (int)P.jobs.size();
        for (const Placed &x : per_cta[c]) P.jobs.push_back(x.j);
        P.makespan = std::max(P.makespan, free_at[c]);
    }
    P.start[grid] = (int)P.jobs.size();
    return MD_OK;
}

void free_resident(md_system *s) {
    for (void *p : s->res_allocs) cudaFree(p);
    s->res_allocs.clear();
    s->rd = ResDev{};
    s->res_grid = 0;
}

int configure_resident(md_system *s, const std::vector<double> *measured = nullptr) {
    if (s->prec != MD_FP32_CELLOFF) return fail(MD_E_ARG, "the resident engine (staging 4) is FP32 only");
    int optin = 0, per_sm = 0;
    MD_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->dev));
    MD_CUDA_TRY(cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, s->dev));
    cudaFuncAttributes fa{};
    MD_CUDA_TRY(cudaFuncGetAttributes(&fa, k_md_resident));
    // RES_CTAS_PER_SM CTAs share an SM's shared memory (1 KB of it is
    // reserved per CTA)
    const size_t smem = std::min((size_t)optin, (size_t)per_sm / RES_CTAS_PER_SM - 1024) - fa.sharedSizeBytes;
    const size_t hb = smem_hist_bytes(s->n_lg, s->n_dx, s->nb);
    if (hb + 4096 > smem) return fail(MD_E_LIMIT, "resident engine: histograms leave no shared memory");
    MD_CUDA_TRY(cudaFuncSetAttribute(k_md_resident, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    MD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_md_resident, RES_THREADS, smem));
    if (occ < RES_CTAS_PER_SM) return fail(MD_E_CUDA, "resident kernel: %d of %d CTAs fit on an SM", occ, RES_CTAS_PER_SM);
    const int grid = s->nsm * RES_CTAS_PER_SM;
    ResPlan P;
    int rc = plan_resident(s->reps, grid, smem - hb, P, measured);
    if (rc) return rc;
    MD_CUDA_TRY(cudaStreamSynchronize(s->st));   // no launch may still use the old buffers
    free_resident(s);
    ResDev &D = s->rd;
    auto A = [&](void **ptr, size_t bytes) {
        if (rc) return;
        if (cudaMalloc(ptr, bytes ? bytes : 16) != cudaSuccess) {
            *ptr = nullptr;
            rc = fail(MD_E_NOMEM, "resident engine: cudaMalloc(%zu)", bytes);
            return;
        }
        s->res_allocs.push_back(*ptr);
    };
    const size_t hm = (size_t)P.hmax;
    A((void **)&D.jobs, sizeof(ResJob) * P.jobs.size());
    A((void **)&D.job_start, sizeof(int32_t) * P.start.size());
    A((void **)&D.halo_off, sizeof(float2) * grid * 4 * hm);
    A((void **)&D.halo_ci, sizeof(uint2) * grid * 2 * hm);
    A((void **)&D.halo_n, sizeof(int32_t) * grid * 2);
    A((void **)&D.mig_a, sizeof(float4) * grid * 2 * hm);
    A((void **)&D.mig_b, sizeof(uint2) * grid * 2 * hm);
    A((void **)&D.mig_n, sizeof(int32_t) * grid * 2);
    A((void **)&D.slab_n, sizeof(int32_t) * grid);
    A((void **)&D.gbar, sizeof(unsigned) * 2 * (size_t)s->nrep);
    A((void **)&D.job_ns, sizeof(unsigned long long) * std::max<size_t>(1, P.jobs.size()));
    if (rc) {
        free_resident(s);
        return rc;
    }
    D.hmax = P.hmax;
    D.smem_bytes = (int)smem;
    MD_CUDA_TRY(cudaMemcpyAsync((void *)D.jobs, P.jobs.data(), sizeof(ResJob) * P.jobs.size(),
                                cudaMemcpyHostToDevice, s->st));
    MD_CUDA_TRY(cudaMemcpyAsync((void *)D.job_start, P.start.data(), sizeof(int32_t) * P.start.size(),
                                cudaMemcpyHostToDevice, s->st));
    MD_CUDA_TRY(cudaMemsetAsync(D.gbar, 0, sizeof(unsigned) * 2 * (size_t)s->nrep, s->st));
    s->res_grid = grid;
    s->res_smem = smem;
    s->res_slabs = P.slabs;
    s->res_max_g = P.max_g;
    s->res_jobs = P.jobs;
    s->res_cost = measured ? *measured : std::vector<double>();
    s->engine = 1;   // the global engine keeps its own launch shape for its other uses
    return MD_OK;
}

int launch_resident(md_system *s, long long nsteps) {
    for (long long done = 0; done < nsteps;) {
        long long step0 = s->step + done;
        long long n = std::min(RES_MAX_STEPS, nsteps - done);
        int phase = done ? 1 : s->phase_half;
        void *args[] = {&s->sd, &s->rd, &step0, &n, &phase};
        MD_CUDA_TRY(cudaLaunchCooperativeKernel((const void *)k_md_resident, dim3(s->res_grid), dim3(RES_THREADS),
                                                args, s->res_smem, s->st));
        k_res_flip<<<1, 1, 0, s->st>>>(s->d_ctl);
        MD_CUDA_TRY(cudaGetLastError());
        done += n;
    }
    s->needs_sort = s->sort_counts = true;
    s->slab_last = false;   // the slots are in this engine's order now
    return MD_OK;
}

int configure_launch(md_system *s, int block, int ppt, int stage) {
    if (stage == 4) return configure_resident(s);
    if (block != 128 && block != 256) return fail(MD_E_ARG, "block_threads must be 128 or 256");
    if (ppt < 1 || ppt > 8) return fail(MD_E_ARG, "per_thread must be in [1, 8]");
    if (stage < 1 || stage > 3) return fail(MD_E_ARG, "staging must be 1, 2, 3 or 4");
    const void *fn = persistent_fn(s->prec, block, stage);
    const int chunk = ppt * block;
    // chunk table: ppt*block consecutive slots of one replica
    std::vector<int4> ch;
    for (int r = 0; r < s->nrep; ++r) {
        const RepDev &R = s->reps[r];
        for (int a = R.pbase; a < R.pbase + R.n; a += chunk)
            ch.push_back(make_int4(r, a, std::min(a + chunk, R.pbase + R.n), 0));
    }
    if ((long long)ch.size() > s->chunk_cap) return fail(MD_E_LIMIT, "chunk table overflow");
    const long long nch = (long long)ch.size();
    const size_t smem = s->prec == MD_FP64
                            ? smem_bytes<double>(s->n_lg, s->n_dx, s->nb, chunk, stage == 1)
                            : smem_bytes<float>(s->n_lg, s->n_dx, s->nb, chunk, stage == 1);
    if (smem > 227 * 1024) return fail(MD_E_LIMIT, "shared memory per CTA exceeds 227 KB");
    MD_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int occ = 0;
    MD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, block, smem));
    if (occ < 1) return fail(MD_E_CUDA, "persistent kernel does not fit on an SM");
    const long long maxco = (long long)occ * s->nsm;
    // Every SM gets the same number of CTAs (the full resident grid, unless
    // there are fewer chunks): an SM finishes a step's force pass when all of
    // its CTAs' work is done, so an SM with one CTA more would set the pace
    // of the grid barrier.  The chunk dealing below evens out the per-CTA sums.
    const long long q = (nch + maxco - 1) / maxco;
    const long long grid = std::min<long long>(4096, std::max<long long>(1, std::min<long long>(maxco, nch)));
    if (q > MAX_CPC) return fail(MD_E_LIMIT, "more than %d chunks per CTA: raise per_thread", MAX_CPC);
    // CTA b owns table entries b, b + grid, b + 2 grid, ... (staged shapes;
    // also the sampling pass and the sort of a rebuild).  Chunks differ in
    // cost by the replicas' densities (neighbours per particle), so they are
    // dealt by decreasing estimated cost, the CTA order reversed every other
    // round, which evens out the per-CTA sums and the wait at the step's grid
    // barrier.  The dynamic distribution of the global-memory shapes takes
    // the chunks in table order, so the costliest come first.  Which CTA
    // computes a chunk does not change any result.
    {
        std::vector<double> cost(nch);
        for (long long k = 0; k < nch; ++k) {
            const RepDev &R = s->reps[ch[k].x];
            const double nbr = M_PI * R.rv2 * (double)R.n / (R.L * R.L);
            cost[k] = (double)(ch[k].z - ch[k].y) * (6.0 + nbr);
        }
        std::vector<long long> order(nch);
        for (long long k = 0; k < nch; ++k) order[k] = k;
        std::stable_sort(order.begin(), order.end(),
                         [&](long long a, long long b) { return cost[a] > cost[b]; });
        std::vector<int4> dealt(nch);
        for (long long k = 0; k < nch; ++k) {
            const long long round = k / grid, w = k % grid;
            const bool full = (round + 1) * grid <= nch;
            const long long b = (full && (round & 1)) ? grid - 1 - w : w;
            dealt[round * grid + b] = ch[order[k]];
        }
        ch.swap(dealt);
    }
    MD_CUDA_TRY(cudaMemcpyAsync(s->d_chunks, ch.data(), sizeof(int4) * ch.size(),
                                cudaMemcpyHostToDevice, s->st));
    s->smem = smem;
    s->grid = (int)grid;
    s->block = block;
    s->ppt = ppt;
    s->sd.chunks = s->d_chunks;
    s->sd.nchunks = (int)nch;
    // global-memory shapes: the later half of the dealing's rounds (its
    // cheapest chunks) is claimed (a measured choice on a 256-replica batch:
    // a third and a half claimed about equal, none or all 3-10 % slower)
    {
        const long long rounds = (nch + grid - 1) / grid;
        const long long keep = stage == 1 ? rounds : rounds / 2;
        // the shared work word holds a claimed chunk's index in 22 bits
        s->sd.nstatic = (int)std::min<long long>(nch, std::max(keep * grid, nch - (1ll << 21)));
    }
    s->sd.ppt = ppt;
    s->sd.stage = stage == 1;
    s->stage = stage;
    s->engine = 0;
    s->lists_valid = false;   // chunk table and list layout change with the shape
    s->shape_new = true;
    return MD_OK;
}

int launch_persistent(md_system *s, long long nsteps, int force_rebuild, const long long *left = nullptr);

// The global engine's invariants (slots sorted by cell, by id inside a cell,
// cell_start, Verlet lists) after a resident launch: a sort-only rebuild,
// which moves no particle's cell and changes no value.
int ensure_sorted(md_system *s) {
    if (!s->needs_sort) return MD_OK;
    s->needs_sort = false;
    // behind the slab engine without the lists: its next launch builds its own
    return launch_persistent(s, 0, s->slab_last ? RB_SORT : RB_NONE);
}

int launch_persistent(md_system *s, long long nsteps, int force_rebuild, const long long *left) {
    s->slab_last = false;
    if (force_rebuild != RB_ALL && force_rebuild != RB_SORT && (s->needs_sort || !s->lists_valid)) force_rebuild = RB_NONE;
    s->needs_sort = false;
    s->lists_valid = force_rebuild != RB_SORT;
    if (force_rebuild == RB_NONE && !s->sort_counts && !s->shape_new) force_rebuild |= RB_QUIET;
    s->sort_counts = false;
    if (s->lists_valid) s->shape_new = false;
    const void *fn = persistent_fn(s->prec, s->block, s->stage);
    long long step0 = s->step;
    int phase = s->phase_half;
    void *args[] = {&s->sd, &step0, &nsteps, &phase, &force_rebuild, &left};
    // the steps' maxima and the chunk claims start from zero: the slot of the
    // first step may hold a maximum from before another engine's steps
    constexpr size_t from = offsetof(Control, vmax), to = offsetof(Control, claims) + sizeof(Control::claims);
    MD_CUDA_TRY(cudaMemsetAsync(s->d_ctl->vmax, 0, to - from, s->st));
    MD_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(s->grid), dim3(s->block), args, s->smem, s->st));
    return MD_OK;
}

// ---- slab engine ------------------------------------------------------------
const void *slab_fn(int prec, bool cluster) {
    if (prec == MD_FP64) return (const void *)k_md_slab<double, false>;
    return cluster ? (const void *)k_md_slab<float, true> : (const void *)k_md_slab<float, false>;
}
SlabLayout slab_layout_of(const md_system *s, int p_cap, int h_cap, int e_cap, int ncells) {
    const size_t hb = smem_hist_bytes(s->n_lg, s->n_dx, s->nb);
    return s->prec == MD_FP64 ? slab_layout<double>(hb, p_cap, h_cap, e_cap, ncells)
                              : slab_layout<float>(hb, p_cap, h_cap, e_cap, ncells);
}

// One cooperative launch (every CTA resident), or one cluster.
cudaLaunchConfig_t slab_config(md_system *s, cudaLaunchAttribute *at) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(s->sl.g);
    cfg.blockDim = dim3(s->sl.threads);
    cfg.dynamicSmemBytes = s->slab_smem;
    cfg.stream = s->st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (s->sl.cluster) {
        at->id = cudaLaunchAttributeClusterDimension;
        at->val.clusterDim.x = s->sl.g;
        at->val.clusterDim.y = at->val.clusterDim.z = 1;
    } else {
        at->id = cudaLaunchAttributeCooperative;
        at->val.cooperative = 1;
    }
    return cfg;
}

// Plans the slabs of a single replica: as many as SMs, of at least two cell
// rows in FP32 and one in FP64 (whose force pass is long enough to pay for
// more slabs), with all the room the SM's shared memory gives beyond what the
// mean density needs (at least 1.05 times the largest slab's mean count and
// 1.1 times a row's, plus five standard deviations of a Poisson count; lists
// 1.25 times the mean neighbour count plus 2 per particle).  No plan where
// that does not fit, e.g. more than about 4,000 FP32 particles per SM.
int plan_slab(md_system *s, bool may_cluster = true) {
    if (s->nrep != 1) return MD_OK;
    const RepDev &R = s->reps[0];
    int g = std::min(std::min(s->nsm, s->prec == MD_FP64 ? R.nc : R.nc / 2), R.cap / 32);
    if (g < 2) g = 1;
    // A cluster's exchange is shorter but leaves 16 SMs.  In FP32 it pays to
    // about 500 particles a slab (us/step, cluster against grid: 1,024
    // particles 3.2/4.3, 4,096 3.7/4.8, 2,000 at phi 0.3 4.4/5.4, 8,000
    // 5.2/5.3, 16,384 8.2/5.7).  In FP64 the pairs want every SM's pipe
    // (1,024 6.3/6.4, 2,048 7.7/6.7, 4,096 10.1/7.1): never.
    bool cluster = false;
    if (may_cluster && g > 1 && s->prec != MD_FP64) {
        const int gc = std::min(g, SLAB_CLUSTER);
        const double pc = (double)R.n * ((R.nc + gc - 1) / gc) / R.nc;
        cluster = pc <= 512.0;
        if (cluster) g = gc;
    }
    const void *fn = slab_fn(s->prec, cluster);
    int optin = 0;
    MD_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->dev));
    cudaFuncAttributes fa{};
    MD_CUDA_TRY(cudaFuncGetAttributes(&fa, fn));
    const size_t smem = (size_t)optin - fa.sharedSizeBytes;
    const int rows = (R.nc + g - 1) / g, ncells = (g == 1 ? R.nc : rows + 2) * R.nc;
    const double pmax = (double)R.n * rows / R.nc, row = (double)R.n / R.nc;
    const double cbar = M_PI * R.rv2 * (double)R.n / (R.L * R.L);
    const double p_want = 1.05 * pmax + 5.0 * std::sqrt(pmax) + 32.0;
    const double h_want = g == 1 ? 0.0 : 1.1 * row + 5.0 * std::sqrt(row) + 32.0;
    // FP64 shares a particle's pairs among lanes, so small slabs take more warps than particles
    const int lo = s->prec == MD_FP64 ? 256 : 128;
    const int hi = s->prec == MD_FP64 ? SLAB_THREADS<double, false>
                                      : (cluster ? SLAB_THREADS<float, true> : SLAB_THREADS<float, false>);
    // FP32: one particle per thread also where a slab holds more than its mean
    const double want = std::ceil(s->prec == MD_FP64 ? 4.0 * pmax : pmax + 3.0 * std::sqrt(pmax));
    const int threads = std::min(hi, std::max(lo, round_up((long long)want, 32)));
    // FP64 is bound by its pipe, so the fullest slab counts (whole rows: up to
    // twice the mean), and long lists leave the global engine fewer idle lanes.
    // Microseconds per step of both, fitted to runs from 1,024 to 262,144
    // particles at phi 0.08 to 0.3 (on starts of few collisions, 262,144 at 0.08:
    // 44 against 71 us; 99,856 at 0.2: 57 against 66; 150,000 at 0.3: 139 against
    // 86; 16,384 at 0.3: 30 against 25; both grow with the gas's correlations, 56
    // and 93 at 262,144).  FP32 slabs were faster at all of them.
    if (s->prec == MD_FP64) {
        const long long chunks = (R.n + 255) / 256, waves = (chunks + 2 * s->nsm - 1) / (2 * s->nsm);
        const double slab = 5.0 + pmax * (0.0091 * cbar - 0.0054);
        const double global = chunks <= s->nsm ? 9.3 + 1.43 * cbar : waves * (11.5 + 2.9 * cbar);
        if (slab > global) return MD_OK;
    }
    SlabDev D{};
    for (double f = 3.0; f > 0.99 && !D.p_cap; f -= 0.05) {
        const int p = (int)std::min<double>(R.n, std::ceil(f * p_want));
        const int h = (int)std::min<double>(R.n, std::ceil(f * h_want));
        const double e = std::ceil(p * (1.25 * cbar + 2.0)) + 256.0;
        if (p + 2 * h >= SLAB_MAX_IDX || e > 1e6) continue;
        if (slab_layout_of(s, p, h, (int)e, ncells).end > smem) continue;
        D.p_cap = p;
        D.h_cap = std::max(h, 1);
        D.e_cap = (int)e;
    }
    if (!D.p_cap) return MD_OK;
    D.g = g;
    D.ncells = ncells;
    D.threads = threads;
    const size_t vsz = s->prec == MD_FP64 ? sizeof(double2) : sizeof(float2), gh = (size_t)g * D.h_cap;
    int rc = MD_OK;
    auto A = [&](void **p, size_t bytes) {
        if (rc == MD_OK) rc = dalloc(s, p, bytes);
    };
    A((void **)&D.word, sizeof(unsigned long long) * 2 * g * g);
    A(&D.halo_off, vsz * 4 * gh);
    A((void **)&D.halo_ci, sizeof(uint2) * 2 * gh);
    A((void **)&D.halo_n, sizeof(int32_t) * 2 * g);
    A(&D.mig_off, vsz * 2 * gh);
    A(&D.mig_vel, vsz * 2 * gh);
    A((void **)&D.mig_ci, sizeof(uint2) * 2 * gh);
    A((void **)&D.mig_n, sizeof(int32_t) * 2 * g);
    A((void **)&D.slab_n, sizeof(int32_t) * g);
    A((void **)&D.left, sizeof(long long));
    if (rc) return rc;
    s->slab_smem = slab_layout_of(s, D.p_cap, D.h_cap, D.e_cap, ncells).end;
    MD_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes));
    int occ = 0;
    MD_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, threads, s->slab_smem));
    D.cluster = cluster;
    s->sl = D;
    if (cluster) {
        MD_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        cudaLaunchAttribute at{};
        cudaLaunchConfig_t cfg = slab_config(s, &at);
        int nclu = 0;
        MD_CUDA_TRY(cudaOccupancyMaxActiveClusters(&nclu, fn, &cfg));
        if (nclu < 1) return plan_slab(s, false);
    }
    s->slab_ok = occ >= 1;
    return MD_OK;
}

int launch_slab(md_system *s, long long nsteps) {
    if (!s->slab_last) {
        // cell_start must describe the slots' order
        int rc = ensure_sorted(s);
        if (rc) return rc;
    }
    long long step0 = s->step;
    int phase = s->phase_half;
    s->sl.counted = s->shape_new;
    s->shape_new = false;
    void *args[] = {&s->sd, &s->sl, &step0, &nsteps, &phase};
    if (!s->sl.cluster)
        MD_CUDA_TRY(cudaMemsetAsync(s->sl.word, 0, sizeof(unsigned long long) * 2 * s->sl.g * s->sl.g, s->st));
    cudaLaunchAttribute at{};
    const cudaLaunchConfig_t cfg = slab_config(s, &at);
    MD_CUDA_TRY(cudaLaunchKernelExC(&cfg, slab_fn(s->prec, s->sl.cluster), args));
    int rc = launch_persistent(s, nsteps, RB_NONE, s->sl.left);
    if (rc) return rc;
    s->needs_sort = true;
    s->slab_last = true;
    s->slab_tried = true;
    return MD_OK;
}

// A slab launch loads, builds its lists, writes back and is followed by the
// (empty) global launch: 15 to 70 us more than a global launch costs.  A readout
// or a short call after it has to sort: 20 to 90 us.  It gains 3 to 25 us per
// step.  `enter`: steps from which a call pays for itself and the sort behind it,
// from a sorted state; `stay`: steps from which a call pays for itself on a state
// that the slab engine left.  Measured break-evens (1,024 to 262,144 particles, phi
// 0.08 to 0.3): FP64 and clusters enter 8 to 16 (one case of 24), stay 4 to 8; the
// FP32 grid enters 12 to 32 (one case of 40), stays 11 to 28.  Single steps behind a slab call,
// FP32, 99,856 particles: 71 us each while they stayed, 20 now.
int64_t slab_enter(const md_system *s) { return s->prec == MD_FP64 || s->sl.cluster ? 16 : 32; }
int64_t slab_stay(const md_system *s) { return s->prec == MD_FP64 || s->sl.cluster ? 8 : 20; }

bool takes_slab(md_system *s, int64_t nsteps) {
    if (s->engine != 0 || !s->slab_ok || !s->slab_on || nsteps < (s->slab_last ? slab_stay(s) : slab_enter(s)))
        return false;
    if (s->slab_wait == 0) return true;
    --s->slab_wait;
    return false;
}

int status_to_code(int ds) {
    if (ds & DS_TIMEOUT) return fail(MD_E_TIMEOUT, "device barrier wait timed out");
    if (ds & DS_CAPACITY)
        return fail(MD_E_LIMIT, "resident engine: a slab outgrew its planned capacity (state undefined)");
    if (ds & DS_NONFINITE) return fail(MD_E_NONFINITE, "non-finite position encountered");
    if (ds & DS_SKIN) return fail(MD_E_SKIN, "a particle moved more than one cell in one step");
    if (ds & DS_NBR_OVERFLOW)
        return fail(MD_E_LIMIT, "neighbour list overflow: raise md_params.nbr_max");
    return MD_OK;
}

constexpr size_t STATUS_BYTES = offsetof(Control, slab_ends) + sizeof(int) - offsetof(Control, status);

int sync_status(md_system *s) {
    // the status word follows the work into pinned memory: one wait
    MD_CUDA_TRY(cudaMemcpyAsync(s->h_status, &s->d_ctl->status, STATUS_BYTES, cudaMemcpyDeviceToHost, s->st));
    MD_CUDA_TRY(cudaStreamSynchronize(s->st));
    const int ds = *s->h_status, ends = s->h_status[STATUS_BYTES / sizeof(int) - 1];
    if (s->slab_tried) {
        const bool early = ends != s->slab_ends;
        s->slab_backoff = early ? std::min(std::max(32, 2 * s->slab_backoff), 1 << 20) : 0;
        s->slab_wait = s->slab_backoff;
    }
    s->slab_ends = ends;
    s->slab_tried = false;
    if (ds) {
        MD_CUDA_TRY(cudaMemset(&s->d_ctl->status, 0, sizeof(int)));
        // a wait that gave up leaves the arrival count behind; no kernel of
        // the system runs now, so it is cleared for the next launch
        if (ds & DS_TIMEOUT) MD_CUDA_TRY(cudaMemset(&s->d_ctl->bar_count, 0, sizeof(unsigned)));
        if ((ds & (DS_TIMEOUT | DS_CAPACITY)) && s->rd.gbar)
            MD_CUDA_TRY(cudaMemset(s->rd.gbar, 0, sizeof(unsigned) * 2 * (size_t)s->nrep));
        return status_to_code(ds);
    }
    return MD_OK;
}

int check_params(const md_params *p, int r, const md_params *p0) {
    if (p->n < 2 || p->n > (1ll << 30)) return fail(MD_E_ARG, "replica %d: n out of [2, 2^30]", r);
    if (!(p->box_L > 0) || !(p->dt > 0) || !(p->rc > 0) || !(p->sigma > 0) || !(p->mass > 0) ||
        !(p->eps >= 0) || !(p->skin > 0))
        return fail(MD_E_ARG, "replica %d: box_L, dt, rc, sigma, mass, skin must be > 0, eps >= 0", r);
    if (p->precision != MD_FP64 && p->precision != MD_FP32_CELLOFF)
        return fail(MD_E_ARG, "replica %d: unknown precision", r);
    if (p->W < 1 || p->W > MD_MAX_W) return fail(MD_E_ARG, "W out of [1,%d]", MD_MAX_W);
    if (p->n_lg < 0 || p->n_lg > MD_MAX_LG) return fail(MD_E_ARG, "n_lg out of [0,%d]", MD_MAX_LG);
    if (p->n_dx < 1 || p->n_dx > MD_MAX_DX) return fail(MD_E_ARG, "n_dx out of [1,%d]", MD_MAX_DX);
    for (int k = 0; k < p->n_lg; ++k)
        if (p->lg_every[k] < 1) return fail(MD_E_ARG, "lg_every[%d] must be >= 1", k);
    for (int d = 0; d < p->n_dx; ++d)
        if (p->lx[d] < 1) return fail(MD_E_ARG, "replica %d: lx[%d] must be >= 1", r, d);
    if (p->n_equil < 0) return fail(MD_E_ARG, "n_equil must be >= 0");
    if (p->block_windows < 1) return fail(MD_E_ARG, "block_windows must be >= 1");
    const long long nc = (long long)std::floor(p->box_L / (p->rc + p->skin));
    if (nc < 3) return fail(MD_E_ARG, "replica %d: box must hold >= 3 cells of rc+skin", r);
    if (nc > 32767) return fail(MD_E_LIMIT, "replica %d: more than 32767 cells per edge", r);
    if (p0) {
        if (p->precision != p0->precision || p->W != p0->W || p->n_equil != p0->n_equil ||
            p->n_lg != p0->n_lg || p->n_dx != p0->n_dx || p->block_windows != p0->block_windows)
            return fail(MD_E_ARG, "replica %d: batch-wide parameters differ from replica 0", r);
        for (int k = 0; k < p->n_lg; ++k)
            if (p->lg_every[k] != p0->lg_every[k])
                return fail(MD_E_ARG, "replica %d: lg_every differs from replica 0", r);
    }
    return MD_OK;
}

int observe(md_system *s, ObsArgs a);

int upload_state(md_system *s, const double *x, const double *y, const double *vx,
                 const double *vy) {
    if (!x || !y || !vx || !vy) return fail(MD_E_ARG, "state arrays must not be NULL");
    const size_t bytes = sizeof(double) * (size_t)s->ntot;
    double *tmp = nullptr;
    MD_CUDA_TRY(scratch_alloc((void **)&tmp, 4 * bytes, s->st));
    int rc = MD_OK;
    const double *src[4] = {x, y, vx, vy};
    for (int k = 0; k < 4 && rc == MD_OK; ++k) {
        cudaError_t e = cudaMemcpyAsync(tmp + k * s->ntot, src[k], bytes, cudaMemcpyDefault, s->st);
        if (e != cudaSuccess) rc = fail(MD_E_CUDA, "state upload: %s", cudaGetErrorString(e));
    }
    if (rc == MD_OK) {
        // fresh cell list: positions go to set 0, buffer 0
        cudaMemsetAsync(&s->d_ctl->set, 0, 2 * sizeof(int), s->st);
        const int nthr = 256;
        const int nblk = (s->nslots + nthr - 1) / nthr;
        if (s->prec == MD_FP64)
            k_init<double><<<nblk, nthr, 0, s->st>>>(s->sd, tmp, tmp + s->ntot, tmp + 2 * s->ntot,
                                                     tmp + 3 * s->ntot);
        else
            k_init<float><<<nblk, nthr, 0, s->st>>>(s->sd, tmp, tmp + s->ntot, tmp + 2 * s->ntot,
                                                    tmp + 3 * s->ntot);
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) rc = fail(MD_E_CUDA, "init kernel: %s", cudaGetErrorString(e));
    }
    if (rc == MD_OK) rc = launch_persistent(s, 0, 1);
    scratch_free(tmp, s->st);
    if (rc) return rc;
    s->phase_half = 0;
    s->slab_wait = s->slab_backoff = 0;   // another state, another chance
    s->slab_tried = false;
    // a state placed on a sampling boundary starts the next window there
    unsigned mask = 0;
    for (int k = 0; k < s->n_lg; ++k)
        if (s->step >= s->n_equil && (s->step - s->n_equil) % s->lg_every[k] == 0) mask |= 1u << k;
    if (mask) {
        ObsArgs a{};
        a.snap_mask = mask;
        rc = observe(s, a);
        if (rc) return rc;
    }
    return sync_status(s);
}

// Runs the observation kernel; completes the half kick when needed.
int observe(md_system *s, ObsArgs a) {
    int rc = ensure_sorted(s);
    if (rc) return rc;
    a.complete = s->phase_half;
    const int nthr = 256;
    const int nblk = s->nslots / nthr;
    const bool pe = a.epart || a.fabs_sum;
    const auto k = s->prec == MD_FP64 ? (pe ? k_observe<double, true> : k_observe<double, false>)
                                      : (pe ? k_observe<float, true> : k_observe<float, false>);
    k<<<nblk, nthr, 0, s->st>>>(s->sd, a);
    MD_CUDA_TRY(cudaGetLastError());
    s->phase_half = 0;
    return MD_OK;
}

// Particles per thread in a chunk: one, i.e. chunks of one block, which
// keeps the staging buffers small and deals the most chunks round-robin.
int default_ppt(const md_system *) { return 1; }

long long windows_done(const md_system *s, int k) {
    const long long t = s->step - s->n_equil;
    if (t < 0) return 0;
    return t / s->lg_every[k];
}

}  // namespace

extern "C" {

int md_init_batch(const md_params *p, int32_t n_rep, const double *x, const double *y,
                  const double *vx, const double *vy, void *stream, md_system **out) {
    mdlg::Range range_("md_init_batch");
    if (!p || !out || n_rep < 1) return fail(MD_E_ARG, "md_init_batch: bad arguments");
    if (n_rep > MD_MAX_REP) return fail(MD_E_LIMIT, "md_init_batch: more than %d replicas", MD_MAX_REP);
    *out = nullptr;
    for (int r = 0; r < n_rep; ++r) {
        int rc = check_params(&p[r], r, r ? &p[0] : nullptr);
        if (rc) return rc;
    }
    md_system *s = new md_system();
    s->st = (cudaStream_t)stream;
    s->prec = p[0].precision;
    s->nrep = n_rep;
    s->W = p[0].W;
    s->nb = (2 * s->W + 1) * (2 * s->W + 1);
    s->n_lg = p[0].n_lg;
    s->n_dx = p[0].n_dx;
    s->block_windows = p[0].block_windows;
    s->n_equil = p[0].n_equil;
    for (int k = 0; k < s->n_lg; ++k) s->lg_every[k] = p[0].lg_every[k];
    long long pbase = 0, cbase = 0, ibase = 0;
    for (int r = 0; r < n_rep; ++r) {
        const md_params &q = p[r];
        RepDev R = make_rep(q, s->prec, s->n_dx);
        R.pbase = (int)pbase;
        R.cbase = (int)cbase;
        R.ibase = (int)ibase;
        s->reps.push_back(R);
        pbase += R.cap;
        cbase += (long long)R.nc * R.nc + 1;
        ibase += q.n;
    }
    if (pbase >= (1ll << 31) - SLOT_PAD || cbase >= (1ll << 31) - 1) {
        delete s;
        return fail(MD_E_LIMIT, "md_init_batch: more than 2^31 slots or cells");
    }
    // neighbour-list capacity: three times the mean count within rv plus
    // eight standard deviations (clustered replicas), or the caller's value
    double kmax = 16.0;
    for (int r = 0; r < n_rep; ++r) {
        const md_params &q = p[r];
        const double rv = q.rc + q.skin;
        const double mean = M_PI * rv * rv * (double)q.n / (s->reps[r].L * s->reps[r].L);
        kmax = std::max(kmax, 3.0 * mean + 8.0 * std::sqrt(mean) + 8.0);
        if (q.nbr_max > 0) kmax = std::max(kmax, (double)q.nbr_max);
    }
    s->K = (int)std::min(1024.0, std::ceil(kmax / 4.0) * 4.0);
    s->nslots = (int)pbase;
    s->total_cells = (int)cbase;
    s->ntot = ibase;
    int rc = MD_OK;
    cudaError_t e = cudaGetDevice(&s->dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&s->nsm, cudaDevAttrMultiProcessorCount, s->dev);
    if (e != cudaSuccess) {
        delete s;
        return fail(MD_E_CUDA, "md_init_batch: %s", cudaGetErrorString(e));
    }
    const size_t vsz = s->prec == MD_FP64 ? sizeof(double2) : sizeof(float2);
    const size_t ns = (size_t)s->nslots, nlg = (size_t)std::max(1, s->n_lg);
    const size_t ngr = ns / 32;
    SysDev &S = s->sd;
#define ALLOC(ptr, bytes) \
    if (rc == MD_OK) rc = dalloc(s, (void **)&(ptr), (bytes))
    ALLOC(s->d_reps, sizeof(RepDev) * n_rep);
    ALLOC(s->d_gran, sizeof(int32_t) * (ns / GRAN));
    ALLOC(s->d_ctl, sizeof(Control));
    for (int k = 0; k < 2; ++k) {
        ALLOC(S.cell[k], sizeof(uint32_t) * ns);
        ALLOC(S.pid[k], sizeof(int32_t) * ns);
        ALLOC(S.vel[k], vsz * ns);
        ALLOC(S.pos[k][0], vsz * ns);
        ALLOC(S.pos[k][1], vsz * ns);
    }
    ALLOC(S.cellcnt, sizeof(int32_t) * s->total_cells);
    ALLOC(S.cell_start, sizeof(int32_t) * (s->total_cells + 1));
    ALLOC(S.newcell, sizeof(int32_t) * ns);
    ALLOC(S.rank, sizeof(int32_t) * ns);
    ALLOC(S.perm, sizeof(int32_t) * ns);
    ALLOC(S.nbr, sizeof(uint32_t) * ns * (size_t)s->K);
    ALLOC(S.nn, sizeof(int32_t) * (ns + 16));   // staged four at a time
    ALLOC(S.cnt_id, sizeof(int32_t) * (size_t)s->ntot);
    s->chunk_cap = (long long)(ns / 128) + n_rep + 1;
    ALLOC(s->d_chunks, sizeof(int4) * s->chunk_cap);
    ALLOC(S.blocksum, sizeof(int32_t) * 4096);
    ALLOC(S.snap_cell, sizeof(uint32_t) * nlg * s->ntot);
    ALLOC(S.snap_off, vsz * nlg * s->ntot);
    const size_t nhist = (size_t)n_rep * nlg * s->n_dx * MD_NBLK * s->nb;
    ALLOC(S.hist, sizeof(int32_t) * nhist);
    ALLOC(S.ovf, sizeof(unsigned long long) * n_rep * nlg * s->n_dx);
    ALLOC(S.mom, sizeof(double) * ngr * nlg * 2);
    ALLOC(S.vmax_rep, sizeof(unsigned) * 3 * (size_t)n_rep);
    ALLOC(S.disp_rep, sizeof(double) * (size_t)n_rep);
    ALLOC(s->d_epart, sizeof(double) * ngr * 4);
    ALLOC(s->d_small, sizeof(double) * (2 * s->nb + 16));
    ALLOC(s->d_hist64, sizeof(long long) * s->nb);
    ALLOC(s->d_nc_of_id, sizeof(int32_t) * s->ntot);
#undef ALLOC
    if (rc == MD_OK && cudaMallocHost((void **)&s->h_status, STATUS_BYTES) != cudaSuccess) {
        s->h_status = nullptr;
        rc = fail(MD_E_NOMEM, "md_init_batch: pinned memory");
    }
    if (rc) {
        md_destroy(s);
        return rc;
    }
    std::vector<int32_t> gran(ns / GRAN);
    for (int r = 0; r < n_rep; ++r)
        for (int g = s->reps[r].pbase / GRAN; g < (s->reps[r].pbase + s->reps[r].cap) / GRAN; ++g)
            gran[g] = r;
    S.reps = s->d_reps;
    S.gran_rep = s->d_gran;
    S.ctl = s->d_ctl;
    S.nslots = s->nslots;
    S.nrep = n_rep;
    S.total_cells = s->total_cells;
    S.n_lg = s->n_lg;
    S.n_dx = s->n_dx;
    S.W = s->W;
    S.nb = s->nb;
    S.block_windows = s->block_windows;
    S.n_equil = s->n_equil;
    for (int k = 0; k < MD_MAX_LG; ++k) S.lg_every[k] = s->lg_every[k];
    S.ntot = s->ntot;
    S.K = s->K;
    S.timeout_ns = 4000000000ull;
    S.dbg_leave_cta = -1;
    auto tryc = [&](cudaError_t er) {
        if (er != cudaSuccess && rc == MD_OK) rc = fail(MD_E_CUDA, "md_init_batch: %s", cudaGetErrorString(er));
    };
    tryc(cudaMemcpyAsync(s->d_reps, s->reps.data(), sizeof(RepDev) * n_rep, cudaMemcpyHostToDevice, s->st));
    tryc(cudaMemcpyAsync(s->d_gran, gran.data(), sizeof(int32_t) * gran.size(), cudaMemcpyHostToDevice, s->st));
    tryc(cudaMemsetAsync(s->d_ctl, 0, sizeof(Control), s->st));
    tryc(cudaMemsetAsync(S.perm, 0xff, sizeof(int32_t) * ns, s->st));   // padding slots: -1
    tryc(cudaMemsetAsync(S.nn, 0, sizeof(int32_t) * (ns + 16), s->st));
    tryc(cudaMemsetAsync(S.cnt_id, 0, sizeof(int32_t) * (size_t)s->ntot, s->st));
    tryc(cudaMemsetAsync(S.cellcnt, 0, sizeof(int32_t) * s->total_cells, s->st));
    tryc(cudaMemsetAsync(S.hist, 0, sizeof(int32_t) * nhist, s->st));
    tryc(cudaMemsetAsync(S.ovf, 0, sizeof(unsigned long long) * n_rep * nlg * s->n_dx, s->st));
    tryc(cudaMemsetAsync(S.mom, 0, sizeof(double) * ngr * nlg * 2, s->st));
    tryc(cudaMemsetAsync(S.vmax_rep, 0, sizeof(unsigned) * 3 * (size_t)n_rep, s->st));
    tryc(cudaMemsetAsync(S.disp_rep, 0, sizeof(double) * (size_t)n_rep, s->st));
    tryc(cudaMemsetAsync(S.snap_cell, 0, sizeof(uint32_t) * nlg * s->ntot, s->st));
    tryc(cudaMemsetAsync(S.snap_off, 0, vsz * nlg * s->ntot, s->st));
    if (rc == MD_OK) {
        k_nc_of_id<<<(s->nslots + 255) / 256, 256, 0, s->st>>>(S, s->d_nc_of_id);
        tryc(cudaGetLastError());
    }
    if (rc == MD_OK) rc = configure_launch(s, 256, default_ppt(s), 1);
    if (rc == MD_OK) rc = plan_slab(s);
    if (rc == MD_OK) rc = upload_state(s, x, y, vx, vy);
    if (rc) {
        md_destroy(s);
        return rc;
    }
    *out = s;
    return MD_OK;
}

int md_resident_plan(const md_params *p, int32_t n_rep, int32_t grid, int64_t smem_bytes, int32_t *jobs_out,
                     int32_t max_jobs, int32_t *start_out, double *makespan) {
    if (!p || n_rep < 1 || n_rep > MD_MAX_REP || grid < 1 || smem_bytes < 4096 || !jobs_out || !start_out ||
        max_jobs < 0)
        return fail(MD_E_ARG, "md_resident_plan: bad arguments");
    std::vector<RepDev> reps;
    for (int r = 0; r < n_rep; ++r) {
        int rc = check_params(&p[r], r, r ? &p[0] : nullptr);
        if (rc) return rc;
        reps.push_back(make_rep(p[r], p[0].precision, p[0].n_dx));
    }
    const int nb = (2 * p[0].W + 1) * (2 * p[0].W + 1);
    const size_t hb = smem_hist_bytes(p[0].n_lg, p[0].n_dx, nb);
    if ((size_t)smem_bytes <= hb) return fail(MD_E_LIMIT, "md_resident_plan: no shared memory left");
    ResPlan P;
    int rc = plan_resident(reps, grid, (size_t)smem_bytes - hb, P);
    if (rc) return rc;
    if ((int)P.jobs.size() > max_jobs) return fail(MD_E_LIMIT, "md_resident_plan: %d slabs > max_jobs", (int)P.jobs.size());
    for (size_t j = 0; j < P.jobs.size(); ++j) {
        const ResJob &J = P.jobs[j];
        const int32_t v[8] = {J.rep, J.g, J.k, J.r0, J.r1, J.p_cap, J.h_cap, J.cta0};
        std::memcpy(jobs_out + 8 * j, v, sizeof(v));
    }
    std::memcpy(start_out, P.start.data(), sizeof(int32_t) * P.start.size());
    if (makespan) *makespan = P.makespan;
    return MD_OK;
}

int md_init(const md_params *p, const double *x, const double *y, const double *vx,
            const double *vy, void *stream, md_system **out) {
    return md_init_batch(p, 1, x, y, vx, vy, stream, out);
}

void md_destroy(md_system *s) {
    if (!s) return;
    if (s->st) cudaStreamSynchronize(s->st);
    free_resident(s);
    for (void *p : s->allocs) cudaFree(p);
    if (s->h_status) cudaFreeHost(s->h_status);
    delete s;
}

int md_step(md_system *s, int64_t nsteps) {
    mdlg::Range range_("md_step");
    if (!s || nsteps < 0) return fail(MD_E_ARG, "md_step: bad arguments");
    if (nsteps == 0) return MD_OK;
    int rc = s->engine == 1 ? launch_resident(s, nsteps)
                            : (takes_slab(s, nsteps) ? launch_slab(s, nsteps) : launch_persistent(s, nsteps, 0));
    if (rc) return rc;
    s->step += nsteps;
    s->phase_half = 1;
    return MD_OK;
}

int md_tune(md_system *s, int32_t block_threads, int32_t per_thread, int32_t staging) {
    if (!s) return fail(MD_E_ARG, "md_tune: NULL system");
    if (block_threads == 0) block_threads = 256;
    if (per_thread == 0) per_thread = default_ppt(s);
    const bool slab = staging == 0;   // the default: the slab engine where a single replica has a plan
    if (staging == 0) staging = 1;
    const int rc = configure_launch(s, block_threads, per_thread, staging);
    if (rc == MD_OK && staging <= 3) s->slab_on = slab;   // (a refused call changes nothing)
    return rc;
}

// ---- checkpoint ---------------------------------------------------------------
// Layout of a checkpoint (host memory): header, then the arrays in the order
// of ckpt_parts.  The state is stored slot by slot in the current set, sorted
// by cell and by id inside a cell (a resident launch's order is sorted
// first), so a load followed by a sort that moves nothing restores the slot
// order, and with it every later force sum and moment partial.
struct CkptHeader {
    uint64_t magic;
    int64_t step, ntot, n_rebuilds;
    int32_t version, prec, nrep, nslots, n_lg, n_dx, nb, phase_half;
};
constexpr uint64_t CKPT_MAGIC = 0x4d444c4743484b31ull;   // "MDLGCHK1"

struct CkptPart {
    void *dev;
    size_t bytes;
};

static std::vector<CkptPart> ckpt_parts(md_system *s, int set, int cur) {
    const SysDev &S = s->sd;
    const size_t vsz = s->prec == MD_FP64 ? sizeof(double2) : sizeof(float2);
    const size_t ns = (size_t)s->nslots, nlg = (size_t)std::max(1, s->n_lg);
    const size_t nhist = (size_t)s->nrep * nlg * s->n_dx * MD_NBLK * s->nb;
    return {{S.cell[set], sizeof(uint32_t) * ns},
            {S.pid[set], sizeof(int32_t) * ns},
            {S.vel[set], vsz * ns},
            {S.pos[set][cur], vsz * ns},
            {S.disp_rep, sizeof(double) * (size_t)s->nrep},
            {S.snap_cell, sizeof(uint32_t) * nlg * (size_t)s->ntot},
            {S.snap_off, vsz * nlg * (size_t)s->ntot},
            {S.hist, sizeof(int32_t) * nhist},
            {S.ovf, sizeof(unsigned long long) * (size_t)s->nrep * nlg * s->n_dx},
            {S.mom, sizeof(double) * (ns / 32) * nlg * 2}};
}

int md_checkpoint_bytes(md_system *s, int64_t *bytes) {
    if (!s || !bytes) return fail(MD_E_ARG, "md_checkpoint_bytes: NULL argument");
    size_t b = sizeof(CkptHeader);
    for (const CkptPart &p : ckpt_parts(s, 0, 0)) b += p.bytes;
    *bytes = (int64_t)b;
    return MD_OK;
}

int md_checkpoint_save(md_system *s, void *buf) {
    mdlg::Range range_("md_checkpoint_save");
    if (!s || !buf) return fail(MD_E_ARG, "md_checkpoint_save: NULL argument");
    int rc = ensure_sorted(s);
    if (rc) return rc;
    rc = sync_status(s);
    if (rc) return rc;
    Control c;
    MD_CUDA_TRY(cudaMemcpy(&c, s->d_ctl, sizeof(Control), cudaMemcpyDeviceToHost));
    CkptHeader h{};
    h.magic = CKPT_MAGIC;
    h.version = 1;
    h.step = s->step;
    h.ntot = s->ntot;
    h.n_rebuilds = c.n_rebuilds;
    h.prec = s->prec;
    h.nrep = s->nrep;
    h.nslots = s->nslots;
    h.n_lg = s->n_lg;
    h.n_dx = s->n_dx;
    h.nb = s->nb;
    h.phase_half = s->phase_half;
    unsigned char *o = static_cast<unsigned char *>(buf);
    std::memcpy(o, &h, sizeof(h));
    o += sizeof(h);
    for (const CkptPart &p : ckpt_parts(s, c.set, c.cur)) {
        MD_CUDA_TRY(cudaMemcpy(o, p.dev, p.bytes, cudaMemcpyDeviceToHost));
        o += p.bytes;
    }
    return MD_OK;
}

int md_checkpoint_load(md_system *s, const void *buf) {
    mdlg::Range range_("md_checkpoint_load");
    if (!s || !buf) return fail(MD_E_ARG, "md_checkpoint_load: NULL argument");
    CkptHeader h;
    std::memcpy(&h, buf, sizeof(h));
    if (h.magic != CKPT_MAGIC || h.version != 1) return fail(MD_E_ARG, "md_checkpoint_load: not a checkpoint");
    if (h.ntot != s->ntot || h.prec != s->prec || h.nrep != s->nrep || h.nslots != s->nslots ||
        h.n_lg != s->n_lg || h.n_dx != s->n_dx || h.nb != s->nb)
        return fail(MD_E_ARG, "md_checkpoint_load: the checkpoint was made by a system of other parameters");
    int rc = sync_status(s);
    if (rc) return rc;
    // the state goes to set 0, buffer 0; then a sort that moves no particle
    MD_CUDA_TRY(cudaMemset(&s->d_ctl->set, 0, 2 * sizeof(int)));
    const unsigned char *o = static_cast<const unsigned char *>(buf) + sizeof(h);
    for (const CkptPart &p : ckpt_parts(s, 0, 0)) {
        MD_CUDA_TRY(cudaMemcpy(p.dev, o, p.bytes, cudaMemcpyHostToDevice));
        o += p.bytes;
    }
    MD_CUDA_TRY(cudaMemcpy(&s->d_ctl->n_rebuilds, &h.n_rebuilds, sizeof(long long), cudaMemcpyHostToDevice));
    MD_CUDA_TRY(cudaMemset(s->sd.vmax_rep, 0, sizeof(unsigned) * 3 * (size_t)s->nrep));
    s->step = h.step;
    s->phase_half = h.phase_half;
    s->needs_sort = s->sort_counts = true;
    s->slab_last = false;
    s->slab_wait = s->slab_backoff = 0;
    rc = ensure_sorted(s);
    if (rc) return rc;
    return sync_status(s);
}

int md_barrier_selftest(md_system *s, double limit_s) {
    if (!s || !(limit_s > 0.0) || !(limit_s <= 4.0)) return fail(MD_E_ARG, "md_barrier_selftest: bad arguments");
    if (s->grid < 2) return fail(MD_E_ARG, "md_barrier_selftest: needs a launch of at least 2 CTAs");
    int rc = sync_status(s);
    if (rc) return rc;
    const uint64_t keep = s->sd.timeout_ns;
    s->sd.timeout_ns = (uint64_t)(limit_s * 1e9);
    s->sd.dbg_leave_cta = 0;
    rc = launch_persistent(s, 1, 0);   // the global engine's grid barrier
    s->sd.dbg_leave_cta = -1;
    s->sd.timeout_ns = keep;
    if (rc) return rc;
    s->step += 1;
    s->phase_half = 1;
    return sync_status(s);
}

int md_slab_selftest(md_system *s, double limit_s) {
    if (!s || !(limit_s > 0.0) || !(limit_s <= 4.0)) return fail(MD_E_ARG, "md_slab_selftest: bad arguments");
    if (!s->slab_ok || s->sl.cluster || s->sl.g < 2)
        return fail(MD_E_ARG, "md_slab_selftest: needs a system whose slabs meet through mailboxes");
    int rc = sync_status(s);
    if (rc) return rc;
    if ((rc = ensure_sorted(s))) return rc;
    const uint64_t keep = s->sd.timeout_ns;
    s->sd.timeout_ns = (uint64_t)(limit_s * 1e9);
    s->sd.dbg_leave_cta = 0;
    rc = launch_slab(s, 1);
    s->sd.dbg_leave_cta = -1;
    s->sd.timeout_ns = keep;
    if (rc) return rc;
    return sync_status(s);
}

int md_sync(md_system *s) {
    if (!s) return fail(MD_E_ARG, "md_sync: NULL system");
    return sync_status(s);
}

int md_info(md_system *s, md_info_t *o) {
    if (!s || !o) return fail(MD_E_ARG, "md_info: NULL argument");
    MD_CUDA_TRY(cudaStreamSynchronize(s->st));
    Control c;
    MD_CUDA_TRY(cudaMemcpy(&c, s->d_ctl, sizeof(Control), cudaMemcpyDeviceToHost));
    o->n_total = s->ntot;
    o->step = s->step;
    o->n_rebuilds = c.n_rebuilds;
    o->n_rep = s->nrep;
    o->precision = s->prec;
    o->grid_blocks = s->grid;
    o->block_threads = s->block;
    return MD_OK;
}

int md_rep_info(md_system *s, int32_t rep, md_rep_info_t *o) {
    if (!s || !o || rep < 0 || rep >= s->nrep) return fail(MD_E_ARG, "md_rep_info: bad arguments");
    const RepDev &R = s->reps[rep];
    o->n = R.n;
    o->L_eff = R.L;
    o->h = R.h;
    o->ncell = R.nc;
    o->reserved = 0;
    for (int d = 0; d < MD_MAX_DX; ++d) o->dx_eff[d] = d < s->n_dx ? R.dxl[d] : 0.0;
    return MD_OK;
}

int md_get_state(md_system *s, double *x, double *y, double *vx, double *vy) {
    if (!s || !x || !y || !vx || !vy) return fail(MD_E_ARG, "md_get_state: NULL argument");
    const size_t bytes = sizeof(double) * s->ntot;
    double *tmp = nullptr;
    MD_CUDA_TRY(scratch_alloc((void **)&tmp, 4 * bytes, s->st));
    ObsArgs a{};
    a.x = tmp;
    a.y = tmp + s->ntot;
    a.vx = tmp + 2 * s->ntot;
    a.vy = tmp + 3 * s->ntot;
    int rc = observe(s, a);
    double *dst[4] = {x, y, vx, vy};
    for (int k = 0; k < 4 && rc == MD_OK; ++k) {
        cudaError_t e = cudaMemcpyAsync(dst[k], tmp + k * s->ntot, bytes, cudaMemcpyDefault, s->st);
        if (e != cudaSuccess) rc = fail(MD_E_CUDA, "md_get_state: %s", cudaGetErrorString(e));
    }
    scratch_free(tmp, s->st);
    if (rc) return rc;
    return sync_status(s);
}

int md_set_state(md_system *s, const double *x, const double *y, const double *vx,
                 const double *vy) {
    if (!s) return fail(MD_E_ARG, "md_set_state: NULL system");
    return upload_state(s, x, y, vx, vy);
}

int md_get_raw(md_system *s, int32_t *cell, void *off_x, void *off_y) {
    if (!s || !cell || !off_x || !off_y) return fail(MD_E_ARG, "md_get_raw: NULL argument");
    ObsArgs a{};
    a.raw_cell = cell;
    a.raw_x = off_x;
    a.raw_y = off_y;
    int rc = observe(s, a);
    if (rc) return rc;
    return sync_status(s);
}

int md_get_snapshot(md_system *s, int32_t lg, int32_t *cell, void *off_x, void *off_y) {
    if (!s || !cell || !off_x || !off_y || lg < 0 || lg >= s->n_lg)
        return fail(MD_E_ARG, "md_get_snapshot: bad arguments");
    const size_t vsz = s->prec == MD_FP64 ? sizeof(double2) : sizeof(float2);
    k_copy_snapshot<<<(unsigned)((s->ntot + 255) / 256), 256, 0, s->st>>>(
        s->sd.snap_cell + (size_t)lg * s->ntot, (const char *)s->sd.snap_off + vsz * lg * s->ntot,
        s->prec == MD_FP64, s->ntot, s->d_nc_of_id, cell, off_x, off_y);
    MD_CUDA_TRY(cudaGetLastError());
    return sync_status(s);
}

int md_forces(md_system *s, double *fx, double *fy, double *fabs_sum) {
    if (!s || !fx || !fy) return fail(MD_E_ARG, "md_forces: NULL argument");
    const size_t bytes = sizeof(double) * s->ntot;
    double *tmp = nullptr;
    MD_CUDA_TRY(scratch_alloc((void **)&tmp, 3 * bytes, s->st));
    ObsArgs a{};
    a.fx = tmp;
    a.fy = tmp + s->ntot;
    a.fabs_sum = tmp + 2 * s->ntot;
    int rc = observe(s, a);
    double *dst[3] = {fx, fy, fabs_sum};
    for (int k = 0; k < 3 && rc == MD_OK; ++k) {
        if (!dst[k]) continue;
        cudaError_t e = cudaMemcpyAsync(dst[k], tmp + k * s->ntot, bytes, cudaMemcpyDefault, s->st);
        if (e != cudaSuccess) rc = fail(MD_E_CUDA, "md_forces: %s", cudaGetErrorString(e));
    }
    scratch_free(tmp, s->st);
    if (rc) return rc;
    return sync_status(s);
}

int md_step_forces(md_system *s, int64_t nsteps, double *fx, double *fy) {
    mdlg::Range range_("md_step_forces");
    if (!s || nsteps < 1 || !fx || !fy) return fail(MD_E_ARG, "md_step_forces: bad arguments");
    const size_t bytes = sizeof(double) * s->ntot;
    double *tmp = nullptr;
    MD_CUDA_TRY(scratch_alloc((void **)&tmp, 2 * bytes, s->st));
    s->sd.dbg_fx = tmp;
    s->sd.dbg_fy = tmp + s->ntot;
    int rc = md_step(s, nsteps);
    s->sd.dbg_fx = s->sd.dbg_fy = nullptr;
    double *dst[2] = {fx, fy};
    for (int k = 0; k < 2 && rc == MD_OK; ++k) {
        cudaError_t e = cudaMemcpyAsync(dst[k], tmp + k * s->ntot, bytes, cudaMemcpyDefault, s->st);
        if (e != cudaSuccess) rc = fail(MD_E_CUDA, "md_step_forces: %s", cudaGetErrorString(e));
    }
    scratch_free(tmp, s->st);
    if (rc) return rc;
    return sync_status(s);
}

int md_energy(md_system *s, int32_t rep, double *out4) {
    if (!s || !out4 || rep < 0 || rep >= s->nrep) return fail(MD_E_ARG, "md_energy: bad arguments");
    ObsArgs a{};
    a.epart = s->d_epart;
    int rc = observe(s, a);
    if (rc) return rc;
    const RepDev &R = s->reps[rep];
    k_sum_energy<<<1, 256, 0, s->st>>>(s->d_epart, R.pbase / 32, (R.pbase + R.cap) / 32, s->d_small);
    MD_CUDA_TRY(cudaGetLastError());
    MD_CUDA_TRY(cudaMemcpyAsync(out4, s->d_small, 4 * sizeof(double), cudaMemcpyDeviceToHost, s->st));
    return sync_status(s);
}

int md_energy_batch(md_system *s, double *out) {
    mdlg::Range range_("md_energy_batch");
    if (!s || !out) return fail(MD_E_ARG, "md_energy_batch: bad arguments");
    ObsArgs a{};
    a.epart = s->d_epart;
    int rc = observe(s, a);
    if (rc) return rc;
    const size_t bytes = sizeof(double) * 4 * (size_t)s->nrep;
    cudaPointerAttributes at{};
    const bool dev = cudaPointerGetAttributes(&at, out) == cudaSuccess && at.type == cudaMemoryTypeDevice;
    cudaGetLastError();
    double *dst = out;
    if (!dev) MD_CUDA_TRY(scratch_alloc((void **)&dst, bytes, s->st));
    k_sum_energy_batch<<<s->nrep, 256, 0, s->st>>>(s->d_epart, s->d_reps, dst);
    cudaError_t e = cudaGetLastError();
    if (!dev) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(out, dst, bytes, cudaMemcpyDeviceToHost, s->st);
        scratch_free(dst, s->st);
    }
    if (e != cudaSuccess) return fail(MD_E_CUDA, "md_energy_batch: %s", cudaGetErrorString(e));
    return sync_status(s);
}

int md_hist_raw(md_system *s, int32_t rep, int32_t lg, int32_t dxi, int64_t *hist,
                int64_t *overflow, int64_t *n_windows) {
    if (!s || !hist || rep < 0 || rep >= s->nrep || lg < 0 || lg >= s->n_lg || dxi < 0 ||
        dxi >= s->n_dx)
        return fail(MD_E_ARG, "md_hist_raw: bad arguments");
    const size_t base = ((size_t)(rep * s->n_lg + lg) * s->n_dx + dxi);
    k_hist_total<<<1, 256, 0, s->st>>>(s->sd.hist + base * MD_NBLK * s->nb, s->nb, s->d_hist64);
    MD_CUDA_TRY(cudaGetLastError());
    MD_CUDA_TRY(cudaMemcpyAsync(hist, s->d_hist64, sizeof(int64_t) * s->nb, cudaMemcpyDeviceToHost, s->st));
    unsigned long long ov = 0;
    MD_CUDA_TRY(cudaMemcpyAsync(&ov, s->sd.ovf + base, sizeof(ov), cudaMemcpyDeviceToHost, s->st));
    int rc = sync_status(s);
    if (rc) return rc;
    if (overflow) *overflow = (int64_t)ov;
    if (n_windows) *n_windows = windows_done(s, lg);
    return MD_OK;
}

int feq_measured(md_system *s, int32_t rep, int32_t lg, int32_t dxi, int32_t symmetrize,
                 double *P_out, double *stderr_out, md_feq_stats *stats) {
    mdlg::Range range_("feq_measured");
    if (!s || !P_out || rep < 0 || rep >= s->nrep || lg < 0 || lg >= s->n_lg || dxi < 0 ||
        dxi >= s->n_dx)
        return fail(MD_E_ARG, "feq_measured: bad arguments");
    const RepDev &R = s->reps[rep];
    const size_t base = ((size_t)(rep * s->n_lg + lg) * s->n_dx + dxi);
    FeqArgs A{};
    A.hist = s->sd.hist + base * MD_NBLK * s->nb;
    A.ovf = s->sd.ovf + base;
    A.mom = s->sd.mom;
    A.g0 = R.pbase / 32;
    A.g1 = (R.pbase + R.cap) / 32;
    A.n_lg = s->n_lg;
    A.lg = lg;
    A.nb = s->nb;
    A.W = s->W;
    A.sym = symmetrize != 0;
    A.n = (double)R.n;
    A.nwin = windows_done(s, lg);
    int used = 0;
    for (long long w = 0; w < A.nwin; ++w) {
        const int b = (int)((w / s->block_windows) % MD_NBLK);
        if (A.wblk[b]++ == 0) ++used;
    }
    A.dx_eff = R.dxl[dxi];
    A.out = s->d_small;
    k_feq_measured<<<1, FEQ_THREADS, 0, s->st>>>(A);
    MD_CUDA_TRY(cudaGetLastError());
    std::vector<double> h(2 * s->nb + 8);
    MD_CUDA_TRY(cudaMemcpyAsync(h.data(), s->d_small, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, s->st));
    int rc = sync_status(s);
    if (rc) return rc;
    std::memcpy(P_out, h.data(), sizeof(double) * s->nb);
    if (stderr_out) std::memcpy(stderr_out, h.data() + s->nb, sizeof(double) * s->nb);
    if (stats) {
        const double *st = h.data() + 2 * s->nb;
        stats->mu2 = st[0];
        stats->mu4 = st[1];
        stats->a2 = st[2];
        stats->dx_eff = A.dx_eff;
        stats->n_windows = A.nwin;
        stats->n_overflow = (int64_t)st[3];
        stats->n_samples = (int64_t)R.n * A.nwin;
        stats->n_blocks_used = used;
    }
    return MD_OK;
}

int md_hist_blocks(md_system *s, int32_t rep, int32_t lg, int32_t dxi, int32_t *hist, int64_t *wblk) {
    if (!s || !hist || !wblk || rep < 0 || rep >= s->nrep || lg < 0 || lg >= s->n_lg || dxi < 0 ||
        dxi >= s->n_dx)
        return fail(MD_E_ARG, "md_hist_blocks: bad arguments");
    const size_t base = ((size_t)(rep * s->n_lg + lg) * s->n_dx + dxi);
    MD_CUDA_TRY(cudaMemcpyAsync(hist, s->sd.hist + base * MD_NBLK * s->nb, sizeof(int32_t) * MD_NBLK * s->nb,
                                cudaMemcpyDeviceToHost, s->st));
    int rc = sync_status(s);
    if (rc) return rc;
    for (int b = 0; b < MD_NBLK; ++b) wblk[b] = 0;
    for (long long w = 0; w < windows_done(s, lg); ++w) wblk[(w / s->block_windows) % MD_NBLK] += 1;
    return MD_OK;
}

int feq_bootstrap(md_system *s, int32_t lg, int32_t dxi, int32_t symmetrize, int32_t n_resamples, uint64_t seed,
                  double *sigma_out) {
    mdlg::Range range_("feq_bootstrap");
    if (!s || !sigma_out || lg < 0 || lg >= s->n_lg || dxi < 0 || dxi >= s->n_dx || n_resamples < 2 ||
        n_resamples > (1 << 20))
        return fail(MD_E_ARG, "feq_bootstrap: bad arguments");
    BootArgs A{};
    A.reps = s->d_reps;
    A.hist = s->sd.hist;
    A.n_lg = s->n_lg;
    A.n_dx = s->n_dx;
    A.lg = lg;
    A.dxi = dxi;
    A.nb = s->nb;
    A.W = s->W;
    A.sym = symmetrize != 0;
    A.B = n_resamples;
    A.seed = seed;
    for (long long w = 0; w < windows_done(s, lg); ++w) A.wblk[(w / s->block_windows) % MD_NBLK] += 1;
    const size_t bytes = sizeof(double) * (size_t)s->nrep * s->nb;
    cudaPointerAttributes at{};
    const bool dev = cudaPointerGetAttributes(&at, sigma_out) == cudaSuccess && at.type == cudaMemoryTypeDevice;
    cudaGetLastError();
    double *dst = sigma_out;
    if (!dev) MD_CUDA_TRY(scratch_alloc((void **)&dst, bytes, s->st));
    A.sigma = dst;
    const int ncls = boot_classes(s->W, A.sym);
    const int keep = boot_p_bytes(A.B, ncls) <= BOOT_KEEP_BYTES;
    const size_t smem = boot_p_bytes(keep ? A.B : BOOT_CHUNK, ncls);
    cudaError_t e = cudaFuncSetAttribute(k_feq_bootstrap, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)BOOT_KEEP_BYTES);
    if (e == cudaSuccess) {
        k_feq_bootstrap<<<dim3(s->nrep, (ncls + BOOT_CLASSES - 1) / BOOT_CLASSES), BOOT_THREADS, smem, s->st>>>(
            A, ncls, keep);
        e = cudaGetLastError();
    }
    if (!dev) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(sigma_out, dst, bytes, cudaMemcpyDeviceToHost, s->st);
        scratch_free(dst, s->st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    }
    if (e != cudaSuccess) return fail(MD_E_CUDA, "feq_bootstrap: %s", cudaGetErrorString(e));
    return MD_OK;
}

int feq_batch(md_system *s, int32_t lg, int32_t dxi, int32_t symmetrize, double *out) {
    mdlg::Range range_("feq_batch");
    if (!s || !out || lg < 0 || lg >= s->n_lg || dxi < 0 || dxi >= s->n_dx)
        return fail(MD_E_ARG, "feq_batch: bad arguments");
    FeqBatchArgs A{};
    A.reps = s->d_reps;
    A.hist = s->sd.hist;
    A.ovf = s->sd.ovf;
    A.mom = s->sd.mom;
    A.n_lg = s->n_lg;
    A.n_dx = s->n_dx;
    A.lg = lg;
    A.dxi = dxi;
    A.nb = s->nb;
    A.W = s->W;
    A.sym = symmetrize != 0;
    A.nwin = windows_done(s, lg);
    const size_t bytes = sizeof(double) * (size_t)s->nrep * (3 * s->nb + FEQB_STATS);
    cudaPointerAttributes at{};
    const bool dev = cudaPointerGetAttributes(&at, out) == cudaSuccess && at.type == cudaMemoryTypeDevice;
    cudaGetLastError();
    double *dst = out;
    if (!dev) MD_CUDA_TRY(scratch_alloc((void **)&dst, bytes, s->st));
    A.out = dst;
    k_feq_batch<<<s->nrep, FEQB_THREADS, 0, s->st>>>(A);
    cudaError_t e = cudaGetLastError();
    if (!dev) {
        if (e == cudaSuccess) e = cudaMemcpyAsync(out, dst, bytes, cudaMemcpyDeviceToHost, s->st);
        scratch_free(dst, s->st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->st);
    }
    if (e != cudaSuccess) return fail(MD_E_CUDA, "feq_batch: %s", cudaGetErrorString(e));
    return MD_OK;
}

// ---- autotuner ------------------------------------------------------------
// Launch shapes tried: block {256, 128} x per_thread {1, 2, 4} x staging
// {shared, global}.  The best shape per (precision, replicas, particle
// count rounded to a power of two, list capacity) is kept for the process.
namespace {
std::mutex g_tune_mu;
std::map<std::tuple<int, int, int, int>, std::tuple<int, int, int>> g_tune_cache;
std::map<std::tuple<int, int, int, int>, std::vector<double>> g_tune_costs;   // resident slab times
// whether the slab engine was the fastest, kept by a system that has a plan for
// it (of the systems under one key some have none)
std::map<std::tuple<int, int, int, int>, bool> g_tune_slab;
}

int md_autotune(md_system *s, int64_t steps_per_trial, int32_t *best3) {
    mdlg::Range range_("md_autotune");
    if (!s || steps_per_trial < 1) return fail(MD_E_ARG, "md_autotune: bad arguments");
    int lg2 = 0;
    while ((1ll << lg2) < s->ntot) ++lg2;
    const auto key = std::make_tuple(s->prec, s->nrep, lg2, s->K);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tune_cache.find(key);
        if (it != g_tune_cache.end()) {
            auto ic = g_tune_costs.find(key);
            int rc = std::get<2>(it->second) == 4 && ic != g_tune_costs.end() && !ic->second.empty() &&
                             (int)ic->second.size() == s->nrep
                         ? configure_resident(s, &ic->second)
                         : configure_launch(s, std::get<0>(it->second), std::get<1>(it->second),
                                            std::get<2>(it->second));
            if (rc) return rc;
            const auto is = g_tune_slab.find(key);   // none: the library's choice, as without a tuner
            s->slab_on = is == g_tune_slab.end() || is->second;
            if (best3) {
                best3[0] = std::get<0>(it->second);
                best3[1] = std::get<1>(it->second);
                best3[2] = std::get<2>(it->second);
            }
            return MD_OK;
        }
    }
    cudaEvent_t e0, e1;
    MD_CUDA_TRY(cudaEventCreate(&e0));
    MD_CUDA_TRY(cudaEventCreate(&e1));
    float best_ms = 1e30f;
    int bb = 256, bp = 1, bs = 1;
    const int blocks[2] = {256, 128}, ppts[3] = {1, 2, 4}, stages[3] = {1, 2, 3};
    int rc = MD_OK;
    s->slab_on = false;
    for (int b : blocks)
        for (int p : ppts)
            for (int st : stages) {
                if (st == 3 && s->prec == MD_FP64) continue;               // same kernel as 2
                if (configure_launch(s, b, p, st) != MD_OK) continue;   // shape does not fit
                rc = md_step(s, steps_per_trial);                          // settles caches
                if (rc) break;
                cudaEventRecord(e0, s->st);
                rc = md_step(s, steps_per_trial);
                if (rc) break;
                cudaEventRecord(e1, s->st);
                cudaEventSynchronize(e1);
                float ms = 0.0f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (ms < best_ms) {
                    best_ms = ms;
                    bb = b;
                    bp = p;
                    bs = st;
                }
            }
    // the slab engine of a single replica, against the fastest global shape timed
    // again: the state has gone on since that shape's trial, and a step's cost
    // with it (the first trial runs on the caller's start, a lattice as a rule,
    // with few pairs in range: FP64, 262,144 particles, 39 us a step there and 71
    // later, when the slab engine's 55 used to lose).  Twice in turn: a trial of 50
    // steps holds one rebuild or two.  Near ties go to the slab engine, whose
    // launch weighs less in a program's longer calls (86,281 FP32 particles: 0.49
    // and 0.47-0.49 ms for 50 steps, 0.89 and 0.77 for 80 and a readout); short
    // calls are kept from it by slab_enter.
    bool slab = false;
    if (rc == MD_OK && s->slab_ok && configure_launch(s, bb, bp, bs) == MD_OK) {
        float ms[2] = {0.0f, 0.0f};
        s->slab_wait = 0;
        for (int k = 0; k < 4 && rc == MD_OK; ++k) {
            s->slab_on = k & 1;
            rc = md_step(s, steps_per_trial);
            cudaEventRecord(e0, s->st);
            if (rc == MD_OK) rc = md_step(s, steps_per_trial);
            cudaEventRecord(e1, s->st);
            cudaEventSynchronize(e1);
            float t = 0.0f;
            cudaEventElapsedTime(&t, e0, e1);
            ms[k & 1] += t;
        }
        slab = ms[1] < 1.05f * ms[0];
    }
    if (steps_per_trial < slab_enter(s)) slab = s->slab_ok;   // too short to have run there
    s->slab_on = slab;
    // the shared-memory-resident engine (batched FP32 ensembles): a trial
    // with the modelled slab costs, then one with the schedule re-planned
    // from the slabs' measured times (the per-replica work split this
    // tunes; no result depends on the schedule)
    std::vector<double> res_cost;
    if (rc == MD_OK && s->prec == MD_FP32_CELLOFF && s->nrep >= 2 && configure_launch(s, 256, 1, 4) == MD_OK) {
        for (int trial = 0; trial < 2 && rc == MD_OK; ++trial) {
            rc = md_step(s, steps_per_trial);
            if (rc) break;
            cudaEventRecord(e0, s->st);
            rc = md_step(s, steps_per_trial);
            cudaEventRecord(e1, s->st);
            cudaEventSynchronize(e1);
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rc == MD_OK && ms < best_ms) {
                best_ms = ms;
                bb = 256;
                bp = 1;
                bs = 4;
                res_cost.clear();
                if (trial == 1) res_cost = s->res_cost;
            }
            if (trial == 0 && rc == MD_OK) {
                // per replica: the longest of its slabs in the last launch
                std::vector<unsigned long long> ns(s->res_jobs.size());
                if (cudaMemcpy(ns.data(), s->rd.job_ns, sizeof(unsigned long long) * ns.size(),
                               cudaMemcpyDeviceToHost) != cudaSuccess)
                    break;
                std::vector<double> cost(s->nrep, 0.0);
                for (size_t j = 0; j < ns.size(); ++j)
                    cost[s->res_jobs[j].rep] = std::max(cost[s->res_jobs[j].rep], (double)ns[j]);
                if (configure_resident(s, &cost) != MD_OK) break;
            }
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (rc) return rc;
    rc = sync_status(s);
    if (rc) return rc;
    rc = bs == 4 && !res_cost.empty() ? configure_resident(s, &res_cost) : configure_launch(s, bb, bp, bs);
    if (rc) return rc;
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tune_cache[key] = std::make_tuple(bb, bp, bs);
        if (s->slab_ok) g_tune_slab[key] = slab;
        g_tune_costs[key] = res_cost;
    }
    if (best3) {
        best3[0] = bb;
        best3[1] = bp;
        best3[2] = bs;
    }
    return MD_OK;
}

}  // extern "C"

