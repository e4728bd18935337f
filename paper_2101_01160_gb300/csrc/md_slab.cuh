// The slab engine: md_step of a single replica in one cooperative launch with
// the whole state in shared memory (Sec. 4 MD with the Sec. 2 sampling fused),
// FP32 and FP64.  Included by md.cu only.
//
// The replica is cut into as many horizontal slabs of whole MD-cell rows as
// there are SMs (of two rows or more in FP32, of one or more in FP64), one slab
// per CTA for the whole launch.  What a step of the global engine spends on a system of up to a few
// hundred thousand particles is latency: list and position gathers through L2
// and a barrier of 600 CTAs.  Here the gathers are shared-memory reads and the
// CTAs exchange three things per step, each through one L2 round trip:
//   * the new offsets of their first and last rows (the neighbours' halo);
//   * the step's largest |v| dt in half skins, in a 64-bit word that also says
//     which exchange it belongs to and that every CTA stores into every other
//     CTA's mailbox: the barrier and the grid-wide maximum are one exchange,
//     no atomic is serialised, and a CTA polls only lines that nobody else
//     reads (slab_sync; 152 CTAs polling one word per CTA took 6 us, this takes
//     3.5 us with the imbalance of the slabs).
// A small FP32 replica's slabs are one thread-block cluster (at most 16 CTAs):
// the exchange is then stores into the CTAs' shared memory and a cluster
// barrier, 1,860 clocks a step against 3,140 (1,024 particles, 16 slabs/32).
// A step has two phases: forces and kick (velocities are private to their
// particle), then, after a CTA barrier, drift in place, so offsets are held
// once.
//
// Measured per step, best of three global shapes -> slabs (phi 0.0784, T 20,
// calls of 800 steps after 2,000): FP32 1,024 particles 6.0 -> 3.1 us, 99,856
// 10.8 -> 7.6 us, 262,144 17.0 -> 10.5 us; FP64 1,024 11.7 -> 6.2 us, 99,856 42
// -> 29 us, 262,144 93 -> 56 us.  By clock stamps in a run of 9.9 us a step
// (262,144 FP32 particles) the forces take 2.9, the exchange 3.3, halo and drift
// 2.1, the rebuilds (one in 22 steps) 1.6.
//
// FP64.  GB300 issues one FP64 warp instruction per 15 clocks and SM, so what
// counts is how many of its lanes work.  A warp first tests its particles'
// list entries in FP32 (float copies of the offsets, cutoff widened by the
// error bound), then takes the surviving pairs 32 at a time, one per lane
// whichever particle they belong to, and the owners add their pairs' forces in
// list order (shuffles).  Lists are tested in FP32 too: they may hold a few
// pairs beyond rv, which changes no force.
//
// The trajectory is, bit for bit, the global engine's: the same rebuild rule,
// canonicalisation and kick/drift arithmetic, and each force is summed over
// the same pairs in the same order (3x3 stencil row by row, column by column,
// by id inside a cell; pairs beyond rc add nothing).  The moments of a window
// are summed per slab in double-double, so their rounding does not depend on
// the particles' order inside a slab.
//
// A slab whose particles, boundary rows, migrants or lists outgrow the planned
// room ends the launch for all slabs at that point, which is always one where
// the state is consistent: the slabs write it back and *left says how many
// steps remain; the global engine, launched behind every slab launch, runs
// them (none as a rule: it then returns at once).  So does one whose list grows
// beyond the caller's nbr_max at a rebuild: the global engine builds the lists
// of that state again and reports it.
#pragma once

#include "md_kernels.cuh"
#include "md_resident.cuh"

namespace mdlg {

constexpr int SLAB_MAX_THREADS = 768;
// FP64 is bound by its pipe, which 16 warps keep busy with twice the registers,
// and a cluster's CTAs hold a few hundred particles.  The FP32 grid spills two
// words at 768 threads (80 registers) and many at 1,024 (64): 262,144 particles
// 13.3 -> 13.1 us, 16,384 at phi 0.3 7.4 -> 6.6 us.
template <typename T, bool CL> constexpr int SLAB_THREADS = sizeof(T) == 8 || CL ? 512 : 768;
constexpr int SLAB_CLUSTER = 16;        // most CTAs of a cluster
constexpr int SLAB_MAX_IDX = 1 << 14;   // list entries: 14-bit index, 2-bit column tag

struct SlabDev {
    unsigned long long *word;   // [2][g receivers][g senders]: exchange number << 32 | payload (zeroed before a launch)
    void *halo_off;             // V2<T> [g][2 sides][2 parities][h_cap]
    uint2 *halo_ci;             // [g][2][h_cap]: cell, id
    int32_t *halo_n;            // [g][2]
    void *mig_off, *mig_vel;    // V2<T> [g][2 directions][h_cap]
    uint2 *mig_ci;              // [g][2][h_cap]
    int32_t *mig_n;             // [g][2]
    int32_t *slab_n;            // [g]: particles of each slab in the state written back
    long long *left;            // steps that the launch leaves to the global engine
    int32_t g, p_cap, h_cap, e_cap, ncells, threads, cluster;   // ncells: MD cells of the largest slab with its halo rows
    int32_t counted;            // rebuilds that this launch adds to the count besides its own (0 or 1)
};

// Byte offsets of a slab's arrays in dynamic shared memory (after the
// histograms).  Own particles: indices [0, p_cap); halo: [p_cap, p_cap + 2
// h_cap), the upper neighbour's first row, then the lower one's last.
struct SlabLayout {
    uint32_t off, foff, vel, cell, id, lst, rend, bpos, mem, ccs, ent, end;   // ccs: ncells + 1
};
template <typename T>
__host__ __device__ inline SlabLayout slab_layout(size_t base, int p_cap, int h_cap, int e_cap, int ncells) {
    SlabLayout L;
    const size_t ph = (size_t)p_cap + 2 * (size_t)h_cap;
    size_t p = base;
    const auto take = [&](size_t bytes) {
        const uint32_t at = (uint32_t)p;
        p += align16(bytes);
        return at;
    };
    L.off = take(ph * 2 * sizeof(T));
    L.foff = sizeof(T) == 8 ? take(ph * sizeof(float2)) : L.off;
    L.vel = take((size_t)p_cap * 2 * sizeof(T));
    L.cell = take(ph * sizeof(uint32_t));
    L.id = take(ph * sizeof(int32_t));
    L.lst = take(((size_t)p_cap + 1) * sizeof(uint32_t));
    L.rend = take((size_t)p_cap * sizeof(uint16_t));
    L.bpos = take((size_t)p_cap * sizeof(uint16_t));
    L.mem = take(ph * sizeof(uint16_t));
    L.ccs = take(((size_t)ncells + 1) * sizeof(int32_t));
    L.ent = take((size_t)e_cap * sizeof(uint16_t));
    L.end = (uint32_t)p;
    return L;
}

template <typename T> struct SlabMem {
    using V = typename V2<T>::type;
    SlabLayout L;
    __device__ __forceinline__ V *off() const { return reinterpret_cast<V *>(res_smem + L.off); }
    __device__ __forceinline__ float2 *foff() const { return reinterpret_cast<float2 *>(res_smem + L.foff); }
    __device__ __forceinline__ V *vel() const { return reinterpret_cast<V *>(res_smem + L.vel); }
    __device__ __forceinline__ uint32_t *cell() const { return reinterpret_cast<uint32_t *>(res_smem + L.cell); }
    __device__ __forceinline__ int32_t *id() const { return reinterpret_cast<int32_t *>(res_smem + L.id); }
    __device__ __forceinline__ uint32_t *lst() const { return reinterpret_cast<uint32_t *>(res_smem + L.lst); }
    __device__ __forceinline__ uint16_t *rend() const { return reinterpret_cast<uint16_t *>(res_smem + L.rend); }
    __device__ __forceinline__ uint16_t *bpos() const { return reinterpret_cast<uint16_t *>(res_smem + L.bpos); }
    __device__ __forceinline__ uint16_t *mem() const { return reinterpret_cast<uint16_t *>(res_smem + L.mem); }
    __device__ __forceinline__ int32_t *ccs() const { return reinterpret_cast<int32_t *>(res_smem + L.ccs); }
    __device__ __forceinline__ uint16_t *ent() const { return reinterpret_cast<uint16_t *>(res_smem + L.ent); }
    // sets the offset of particle j (own or halo) and its float copy
    __device__ __forceinline__ void put_off(int j, V o) const {
        off()[j] = o;
        if (sizeof(T) == 8) foff()[j] = make_float2((float)o.x, (float)o.y);
    }
};

// What a CTA keeps about its slab besides the arrays (uniform over the CTA).
struct SlabCta {
    int k, g, r0, r1, up, down;   // slab, slabs, MD-cell rows [r0, r1), neighbours
    int last;                     // published row of the lower neighbour that is its last: 1, or 0 if it has one row
    int p, nh[2], par;            // own particles, halo particles, parity of the published offsets
    unsigned seq;                 // exchanges done
    unsigned *box;                // cluster: the others' payloads, [2][SLAB_CLUSTER] in shared memory
};

__device__ __forceinline__ unsigned long long ld_acquire_gpu64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// This CTA's mailbox of the current exchange, one word per sender.
__device__ __forceinline__ unsigned long long *slab_mail(const SlabDev &D, const SlabCta &X) {
    return D.word + ((size_t)(X.seq & 1u) * X.g + X.k) * X.g;
}

// One exchange: posts this CTA's payload (thread 0's), waits for every CTA's
// and returns the largest; what a CTA wrote to global memory before is visible to all
// after.  A word is not overwritten before its CTA has read it: the
// next-but-one exchange's, of the same parity, is posted only after the next,
// which a CTA posts after reading its mailbox of this one.  The wait is
// bounded (S.timeout_ns): a CTA that waits longer flags DS_TIMEOUT, and every
// CTA leaves the kernel at its next exchange (ok = false).  A cluster meets at
// the hardware's barrier instead: its CTAs run at the same time, and every one
// makes the same exchanges (what they branch on is exchanged).
template <bool CL>
__device__ __forceinline__ unsigned slab_sync(const SysDev &S, const SlabDev &D, SlabCta &X, unsigned payload,
                                              bool &ok) {
    __shared__ unsigned s_wmax[SLAB_MAX_THREADS / 32], s_pay;
    __shared__ int s_fail;
    if constexpr (CL) {
        // one 32-bit word per sender in every CTA's shared memory, by parity
        // of the exchange; the barrier releases and acquires for the cluster
        const unsigned par = ++X.seq & 1u;
        if (threadIdx.x == 0) s_pay = payload;
        __syncthreads();
        if ((int)threadIdx.x < X.g) {
            uint32_t at;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                         : "=r"(at)
                         : "r"(smem_u32(&X.box[par * SLAB_CLUSTER + X.k])), "r"(threadIdx.x));
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(s_pay) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        unsigned r = 0;
        for (int j = 0; j < X.g; ++j) r = max(r, X.box[par * SLAB_CLUSTER + j]);
        ok = true;
        return r;
    }
    const int tid = threadIdx.x;
    const unsigned seq = ++X.seq;
    unsigned long long *w = slab_mail(D, X);
    if (tid == 0) {
        s_fail = 0;
        s_pay = payload;
    }
    __syncthreads();
    // the release of each store covers what the whole CTA wrote before the barrier
    for (int t = tid; t < X.g; t += blockDim.x)
        st_release_gpu64(w + ((long long)t - X.k) * X.g + X.k, (unsigned long long)seq << 32 | s_pay);
    const int pollers = (X.g + 31) & ~31;   // whole warps
    unsigned m = 0;
    for (int t = tid; t < pollers; t += blockDim.x) {
        unsigned long long v = 0;
        if (t < X.g) {
            uint64_t t0 = 0;
            unsigned spins = 0;
            while ((unsigned)((v = ld_acquire_gpu64(&w[t])) >> 32) != seq) {
                if ((++spins & 255u) == 0) {
                    const uint64_t now = global_ns();
                    if (t0 == 0) t0 = now;
                    if ((*(volatile int *)&S.ctl->status) & DS_TIMEOUT) {
                        s_fail = 1;
                        break;
                    }
                    if (now - t0 > S.timeout_ns) {
                        atomicOr(&S.ctl->status, (int)DS_TIMEOUT);
                        s_fail = 1;
                        break;
                    }
                }
            }
        }
        m = max(m, (unsigned)v);
    }
    if (tid < pollers) {
        m = __reduce_max_sync(0xffffffffu, m);
        if ((tid & 31) == 0) s_wmax[tid >> 5] = m;
    }
    __syncthreads();
    unsigned r = 0;
    for (int i = 0; i < min(pollers, (int)blockDim.x) >> 5; ++i) r = max(r, s_wmax[i]);
    ok = s_fail == 0;
    return r;
}

// Sum of `own` over the CTAs before this one, from the words of the last
// exchange (whose payloads were the CTAs' own values).
template <bool CL>
__device__ __forceinline__ int slab_before(const SlabDev &D, const SlabCta &X) {
    int o = 0;
    if constexpr (CL) {
        for (int j = 0; j < X.k; ++j) o += (int)X.box[(X.seq & 1u) * SLAB_CLUSTER + j];
        return o;
    }
    const unsigned long long *w = slab_mail(D, X);
    for (int j = 0; j < X.k; ++j) o += (int)(unsigned)ld_acquire_gpu64(&w[j]);
    return o;
}

// ---------------------------------------------------------------- halo
// Publishes the first and the last row of the slab (cells, ids, offsets).
// Returns whether they fit, and whether every particle lies in the slab's rows
// (the lists index cells by row; slots in another order than the slabs' leave
// all steps to the global engine, which sorts).
template <typename T>
__device__ bool slab_publish_rows(const SlabDev &D, const SlabMem<T> &M, const SlabCta &X) {
    using V = typename V2<T>::type;
    __shared__ int s_n[2];
    if (X.g == 1) return true;
    if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
    __syncthreads();
    V *pub = static_cast<V *>(D.halo_off);
    for (int i = threadIdx.x; i < X.p; i += blockDim.x) {
        const uint32_t c = M.cell()[i];
        const int cy = (int)(c >> 16);
        // (a slab of one row publishes it once, as its first, for both neighbours)
        const int side = cy == X.r0 ? 0 : (cy == X.r1 - 1 ? 1 : -1);
        uint16_t b = RES_NOB;
        if (cy < X.r0 || cy >= X.r1) atomicAdd(&s_n[0], D.h_cap + 1);   // a stranger: does not fit
        if (side >= 0) {
            const int at = atomicAdd(&s_n[side], 1);   // the order of a halo changes no result
            if (at < D.h_cap) {
                b = (uint16_t)(side << 15 | at);
                D.halo_ci[((size_t)X.k * 2 + side) * D.h_cap + at] = make_uint2(c, (uint32_t)M.id()[i]);
                pub[(((size_t)X.k * 2 + side) * 2 + X.par) * D.h_cap + at] = M.off()[i];
            }
        }
        M.bpos()[i] = b;
    }
    __syncthreads();
    if (threadIdx.x < 2) D.halo_n[X.k * 2 + threadIdx.x] = s_n[threadIdx.x];
    return s_n[0] <= D.h_cap && s_n[1] <= D.h_cap;
}

// Reads the neighbours' published rows into the halo.
template <typename T>
__device__ void slab_read_rows(const SlabDev &D, const SlabMem<T> &M, SlabCta &X) {
    using V = typename V2<T>::type;
    X.nh[0] = X.nh[1] = 0;
    if (X.g > 1) {
        const V *pub = static_cast<const V *>(D.halo_off);
        const int src[2] = {X.up * 2, X.down * 2 + X.last};   // the up neighbour's first row, the down one's last
        for (int h = 0; h < 2; ++h) {
            const int n = *(volatile int32_t *)&D.halo_n[src[h]];
            X.nh[h] = n;
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const uint2 ci = __ldcg(&D.halo_ci[(size_t)src[h] * D.h_cap + i]);
                const int j = D.p_cap + h * D.h_cap + i;
                M.cell()[j] = ci.x;
                M.id()[j] = (int32_t)ci.y;
                M.put_off(j, __ldcg(&pub[((size_t)src[h] * 2 + X.par) * D.h_cap + i]));
            }
        }
    }
    __syncthreads();
}

// The neighbours' new offsets after a step.
template <typename T>
__device__ __forceinline__ void slab_read_offsets(const SlabDev &D, const SlabMem<T> &M, const SlabCta &X) {
    using V = typename V2<T>::type;
    if (X.g > 1) {
        const V *pub = static_cast<const V *>(D.halo_off);
        const V *p0 = pub + (((size_t)X.up * 2 + 0) * 2 + X.par) * D.h_cap;
        const V *p1 = pub + (((size_t)X.down * 2 + X.last) * 2 + X.par) * D.h_cap;
        const int n0 = X.nh[0], n = n0 + X.nh[1];
        for (int t = threadIdx.x; t < n; t += blockDim.x) {
            const bool lo = t < n0;
            M.put_off(D.p_cap + (lo ? t : D.h_cap + t - n0), __ldcg(lo ? p0 + t : p1 + t - n0));
        }
    }
    __syncthreads();
}

// ---------------------------------------------------------------- lists
// Member m of a stencil row (slab_lists): a place in the sorted members, or
// for a row across the periodic edge its place in the order of its columns.
__device__ __forceinline__ int slab_member(const uint16_t *mem, const int32_t *ccs, int row, int cx, int nc, int wrapped,
                                           int m1, int m2, int m) {
    if (wrapped) {
        if (m < m1) m += ccs[row + wrap1(cx - 1, nc)];
        else if (m < m2) m += ccs[row + cx] - m1;
        else m += ccs[row + wrap1(cx + 1, nc)] - m2;
    }
    return mem[m];
}

// Neighbour lists of the own particles in stencil order (rows dy = -1, 0, 1,
// columns dx = -1, 0, 1, by id inside a cell): a counting sort of own and halo
// particles by MD cell (rows of the slab and one either side), ids sorted
// inside a cell, then one run over the three cells of each stencil row whose
// hits are kept as bits, so the entries are written as soon as the counts
// before them are known.  FP32 distances; with T = double the radius is widened by
// the bound of their rounding.  Returns whether they fit, none longer than kmax.
template <typename T>
__device__ bool slab_lists(const RepDev &R, const SlabDev &D, const SlabMem<T> &M, const SlabCta &X, int kmax, int *s_w) {
    const int nc = R.nc, nt = (int)blockDim.x;
    const int G = X.g == 1 ? nc : (X.r1 - X.r0) + 2, ncells = G * nc;
    uint16_t *mem = M.mem();
    int32_t *ccs = M.ccs();
    const uint32_t *cell = M.cell();
    const int32_t *id = M.id();
    const auto relrow = [&](int cy) {
        if (X.g == 1) return cy;
        int r = cy - X.r0 + 1;
        if (r < 0) r += nc;
        else if (r >= nc) r -= nc;
        return r;
    };
    // particle t of own, upper halo, lower halo, and its cell in the grid
    const int n0 = X.p + X.nh[0], np = n0 + X.nh[1];
    const auto index = [&](int t) { return t < X.p ? t : (t < n0 ? D.p_cap + t - X.p : D.p_cap + D.h_cap + t - n0); };
    const auto grid_cell = [&](int t, int j) {   // a halo's row by the side it came from
        const uint32_t c = cell[j];
        const int r = t < X.p ? relrow((int)(c >> 16)) : (t < n0 ? G - 1 : 0);
        return r * nc + (int)(c & 0xffffu);
    };
    for (int c = threadIdx.x; c <= ncells; c += nt) ccs[c] = 0;
    __syncthreads();
    for (int t = threadIdx.x; t < np; t += nt) atomicAdd(&ccs[grid_cell(t, index(t))], 1);
    __syncthreads();
    {
        // inclusive sums; the decrementing scatter below leaves ccs[c] = first member of c
        int carry = 0;
        for (int c0 = 0; c0 < ncells; c0 += 4 * nt) {
            const int c = c0 + 4 * (int)threadIdx.x;
            int v[4], sum = 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = c + q < ncells ? ccs[c + q] : 0;
                sum += v[q];
            }
            int tot;
            int ex = carry + block_excl_scan(sum, s_w, &tot);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                ex += v[q];
                if (c + q < ncells) ccs[c + q] = ex;
            }
            carry += tot;
        }
        if (threadIdx.x == 0) ccs[ncells] = carry;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < np; t += nt) {
        const int j = index(t);
        mem[atomicSub(&ccs[grid_cell(t, j)], 1) - 1] = (uint16_t)j;
    }
    __syncthreads();
    for (int c = threadIdx.x; c < ncells; c += nt) {
        const int a = ccs[c], b = ccs[c + 1];
        for (int m = a + 1; m < b; ++m) {
            const uint16_t v = mem[m];
            const int ki = id[v];
            int q = m - 1;
            while (q >= a && id[mem[q]] > ki) {
                mem[q + 1] = mem[q];
                --q;
            }
            mem[q + 1] = v;
        }
    }
    __syncthreads();
    const float h = R.hf;
    // coordinates of pairs within the stencil stay below 2.5 h, so an FP32
    // r^2 is off by less than 2^-19 h^2 (four roundings per component)
    const float rv2 = sizeof(T) == 8 ? R.rv2f + h * h * 0x1p-18f : R.rv2f;
    const float2 *fo = M.foff();
    uint16_t *ent = M.ent();
    uint32_t *lst = M.lst();
    bool over = false;
    int e0 = 0;
    for (int base = 0; base < X.p; base += nt) {
        const int i = base + (int)threadIdx.x;
        // members of the three stencil rows within the radius, one bit each;
        // a row's members are [a, a + len), its columns start at a, m1, m2
        unsigned long long hit[3] = {0ull, 0ull, 0ull};
        int a[3], m1[3], m2[3], wrapped = 0;
        uint32_t rows = 0;
        int cnt = 0;
        if (i < X.p) {
            const uint32_t ci = cell[i];
            const int cx = (int)(ci & 0xffffu), rr = relrow((int)(ci >> 16));
            const float2 oi = fo[i];
            const float sxm = -h - oi.x, sx0 = -oi.x, sxp = h - oi.x;
            wrapped = cx < 1 || cx > nc - 2;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int row = (X.g == 1 ? wrap1(rr + q - 1, nc) : rr + q - 1) * nc;
                const float sy = q == 0 ? -h - oi.y : (q == 1 ? -oi.y : h - oi.y);
                int len;
                if (!wrapped) {
                    const int c = row + cx - 1;
                    a[q] = ccs[c];
                    m1[q] = ccs[c + 1];
                    m2[q] = ccs[c + 2];
                    len = ccs[c + 3] - a[q];
                } else {   // columns across the periodic edge: members by their place in the row's order
                    const int l = row + wrap1(cx - 1, nc), r = row + wrap1(cx + 1, nc);
                    a[q] = 0;
                    m1[q] = ccs[l + 1] - ccs[l];
                    m2[q] = m1[q] + ccs[row + cx + 1] - ccs[row + cx];
                    len = m2[q] + ccs[r + 1] - ccs[r];
                }
                over |= len > 64;
                const auto member = [&](int m) { return slab_member(mem, ccs, row, cx, nc, wrapped, m1[q], m2[q], m); };
                for (int t0 = 0; t0 < min(len, 64); t0 += 4) {   // four members' loads at a time
                    int j[4];
                    float2 o[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) j[u] = member(a[q] + min(t0 + u, len - 1));
#pragma unroll
                    for (int u = 0; u < 4; ++u) o[u] = fo[j[u]];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int m = a[q] + t0 + u;
                        const float rx = o[u].x + (m < m1[q] ? sxm : (m < m2[q] ? sx0 : sxp)), ry = o[u].y + sy;
                        if (t0 + u < len && rx * rx + ry * ry < rv2 && j[u] != i) hit[q] |= 1ull << (t0 + u);
                    }
                }
                cnt += __popcll(hit[q]);
                if (q < 2) rows |= (uint32_t)min(cnt, 255) << (8 * q);
            }
            over |= cnt > kmax;
        }
        int tot;
        const int at = e0 + block_excl_scan(cnt, s_w, &tot);
        if (i < X.p) {
            lst[i] = (uint32_t)at;
            M.rend()[i] = (uint16_t)rows;
            const uint32_t ci = cell[i];
            const int cx = (int)(ci & 0xffffu), rr = relrow((int)(ci >> 16));
            int e = at;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int row = (X.g == 1 ? wrap1(rr + q - 1, nc) : rr + q - 1) * nc;
                for (unsigned long long w = hit[q]; w; w &= w - 1ull) {
                    const int m = a[q] + __ffsll((long long)w) - 1;
                    const int j = slab_member(mem, ccs, row, cx, nc, wrapped, m1[q], m2[q], m);
                    if (e < D.e_cap) ent[e] = (uint16_t)((uint32_t)j | (m < m1[q] ? 0u : (m < m2[q] ? 1u << 14 : 2u << 14)));
                    ++e;
                }
            }
        }
        e0 += tot;
    }
    if (threadIdx.x == 0) lst[X.p] = (uint32_t)e0;
    over |= e0 > D.e_cap;
    return !__syncthreads_or(over);
}

// ---------------------------------------------------------------- forces
// The constants of a step in the state's precision.
template <typename T> struct SlabPar {
    T h, rc2, eps24, sig2, hk, dt;
    float vscale, rc2f;   // rc2f: the FP32 test's cutoff, widened (T = double)
};

// First kick(s) of one particle (kick_drift's arithmetic without the drift).
template <typename T>
__device__ __forceinline__ void slab_kick(const SlabPar<T> &P, typename V2<T>::type *vel, int i, T fx, T fy, bool first,
                                          float &vm, bool &bad) {
    typename V2<T>::type v = vel[i];
    if (!first) {
        v.x = axpyT(v.x, P.hk, fx);
        v.y = axpyT(v.y, P.hk, fy);
    }
    v.x = axpyT(v.x, P.hk, fx);
    v.y = axpyT(v.y, P.hk, fy);
    vel[i] = v;
    const float vx = (float)v.x, vy = (float)v.y;
    const float sp = __fmul_rn(sqrtf(__fmaf_rn(vx, vx, __fmul_rn(vy, vy))), P.vscale);
    vm = fmaxf(vm, sp);
    bad |= !(sp < 1e30f);
}

// FP32: one thread per particle (the arithmetic of lj_list_from).
__device__ __forceinline__ void slab_forces(const SysDev &S, const SlabMem<float> &M, const SlabCta &X,
                                            const SlabPar<float> &P, bool first, bool dbg, float &vm, bool &bad) {
    const float2 *off = M.off();
    const uint16_t *ent = M.ent();
    for (int i = threadIdx.x; i < X.p; i += blockDim.x) {
        const float2 oi = off[i];
        const float sx0 = -P.h - oi.x, sx1 = -oi.x, sx2 = P.h - oi.x;
        const float sy0 = -P.h - oi.y, sy1 = -oi.y, sy2 = P.h - oi.y;
        const uint32_t st = M.lst()[i], en = M.lst()[i + 1], re = M.rend()[i];
        const uint32_t e1 = st + (re & 0xffu), e2 = st + (re >> 8);
        float fx = 0.0f, fy = 0.0f;
        double pe_unused = 0.0, fa_unused = 0.0;
        // batches of U entries, all their loads issued before the arithmetic
        constexpr int U = 4;
        for (uint32_t e = st; e < en; e += U) {
            uint32_t v[U];
            float2 o[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = ent[min(e + u, en - 1)];
#pragma unroll
            for (int u = 0; u < U; ++u) o[u] = off[v[u] & RES_IDX];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (e + u < en) {
                    const uint32_t t = v[u] >> 14;
                    const float sx = t == 0 ? sx0 : (t == 1 ? sx1 : sx2);
                    const float sy = e + u < e1 ? sy0 : (e + u < e2 ? sy1 : sy2);
                    lj_pair_acc<float, false>(o[u].x + sx, o[u].y + sy, P.rc2, P.eps24, P.sig2, fx, fy, 0.0, pe_unused,
                                              fa_unused);
                }
            }
        }
        if (dbg) {
            S.dbg_fx[M.id()[i]] = (double)fx;
            S.dbg_fy[M.id()[i]] = (double)fy;
        }
        slab_kick<float>(P, M.vel(), i, fx, fy, first, vm, bad);
    }
}

// The k-th (from 0) set bit of m1:m0; past the last, entries from 64 on.
__device__ __forceinline__ uint32_t slab_kth(uint32_t m0, uint32_t m1, uint32_t k) {
    const uint32_t n0 = __popc(m0), n = n0 + __popc(m1);
    if (k >= n) return 64u + k - n;
    const bool up = k >= n0;
    uint32_t w = up ? m1 : m0, at = up ? 32u : 0u;
    if (up) k -= n0;
#pragma unroll
    for (int step = 16; step; step >>= 1) {
        const uint32_t c = __popc(w & ((1u << step) - 1u));
        if (k >= c) {
            k -= c;
            w >>= step;
            at += step;
        }
    }
    return at;
}

// FP64: per warp up to 32 owners (fewer in a small slab, so that all warps
// share the work); pairs 32 at a time over the warp's lanes.
__device__ __forceinline__ void slab_forces(const SysDev &S, const SlabMem<double> &M, const SlabCta &X,
                                            const SlabPar<double> &P, bool first, bool dbg, float &vm, bool &bad) {
    const double2 *off = M.off();
    const float2 *fo = M.foff();
    const uint16_t *ent = M.ent();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int pw = X.p <= 8 * nw ? 8 : (X.p <= 16 * nw ? 16 : 32);
    const float hf = (float)P.h;
    for (int base = warp * pw; base < X.p; base += nw * pw) {
        const int i = base + lane;
        const bool own = lane < pw && i < X.p;
        uint32_t st = 0, len = 0, r1 = 0, r2 = 0;
        unsigned long long mask = 0;   // entries within the widened cutoff (entries past 63: all)
        if (own) {
            const float2 oi = fo[i];
            st = M.lst()[i];
            len = M.lst()[i + 1] - st;
            const uint32_t re = M.rend()[i];
            r1 = re & 0xffu;
            r2 = re >> 8;
            for (uint32_t e0 = 0; e0 < min(len, 64u); e0 += 4) {   // four entries' loads at a time
                uint32_t v[4];
                float2 o[4];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) v[u] = ent[st + min(e0 + u, len - 1)];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) o[u] = fo[v[u] & RES_IDX];
#pragma unroll
                for (uint32_t u = 0; u < 4; ++u) {
                    const uint32_t e = e0 + u, row = (e >= r1) + (e >= r2);
                    const float rx = o[u].x + __fmaf_rn((float)((int)(v[u] >> 14) - 1), hf, -oi.x);
                    const float ry = o[u].y + __fmaf_rn((float)((int)row - 1), hf, -oi.y);
                    if (e < len && rx * rx + ry * ry < P.rc2f) mask |= 1ull << e;
                }
            }
        }
        const uint32_t more = len > 64u ? len - 64u : 0u;
        const int cnt = __popcll(mask) + (int)more;
        int incl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        const int excl = incl - cnt;
        double fx = 0.0, fy = 0.0;
        for (int c0 = 0; c0 < total; c0 += 32) {
            // this lane's pair: its owner by bisection of the running counts,
            // its entry as the owner's k-th surviving one.  (Owners writing
            // their pairs into a window took 14,470 clocks a step in a dense
            // system, 2,000 particles at phi 0.3: one lane at a time; this way the
            // whole step went from 16.2 to 14.7 us.)
            const int q = c0 + lane;
            int o = 0;
#pragma unroll
            for (int step = 16; step; step >>= 1)
                if (__shfl_sync(0xffffffffu, incl, o + step - 1) <= q) o += step;
            const uint32_t k = (uint32_t)(q - __shfl_sync(0xffffffffu, excl, o));
            const uint32_t m0 = __shfl_sync(0xffffffffu, (uint32_t)mask, o);
            const uint32_t m1 = __shfl_sync(0xffffffffu, (uint32_t)(mask >> 32), o);
            const uint32_t est = __shfl_sync(0xffffffffu, st, o), rows = __shfl_sync(0xffffffffu, r1 | r2 << 8, o);
            double fr = 0.0, rx = 0.0, ry = 0.0;
            if (q < total) {
                const uint32_t e = slab_kth(m0, m1, k), v = ent[est + e];
                const double2 oi = off[base + o], oj = off[v & RES_IDX];
                const uint32_t tx = v >> 14, ty = (e >= (rows & 0xffu)) + (e >= rows >> 8);
                const double hx = tx == 0 ? -P.h : (tx == 1 ? 0.0 : P.h), hy = ty == 0 ? -P.h : (ty == 1 ? 0.0 : P.h);
                rx = oj.x + __dsub_rn(hx, oi.x);
                ry = oj.y + __dsub_rn(hy, oi.y);
                const double r2 = __fma_rn(rx, rx, ry * ry);
                double s6;
                if (within(r2, P.rc2)) fr = lj_pair_fr<double>(r2, P.eps24, P.sig2, s6);
            }
            const int first_pos = max(excl, c0), n = min(incl, c0 + 32) - first_pos;   // this owner's pairs here
            const int nmax = __reduce_max_sync(0xffffffffu, n);
            for (int k = 0; k < nmax; ++k) {
                const int src = first_pos - c0 + k;           // taken modulo 32 by the shuffle
                const double f = __shfl_sync(0xffffffffu, fr, src), x = __shfl_sync(0xffffffffu, rx, src),
                             y = __shfl_sync(0xffffffffu, ry, src);
                if (k < n && f != 0.0) {
                    fx = __fma_rn(-f, x, fx);
                    fy = __fma_rn(-f, y, fy);
                }
            }
        }
        if (own) {
            if (dbg) {
                S.dbg_fx[M.id()[i]] = fx;
                S.dbg_fy[M.id()[i]] = fy;
            }
            slab_kick<double>(P, M.vel(), i, fx, fy, first, vm, bad);
        }
    }
}

// ---------------------------------------------------------------- moments
struct DD {   // unevaluated sum hi + lo
    double hi, lo;
};
__device__ __forceinline__ void dd_add(DD &a, double hi, double lo) {
    const double s = __dadd_rn(a.hi, hi), bb = __dsub_rn(s, a.hi);
    const double e = __dadd_rn(__dsub_rn(a.hi, __dsub_rn(s, bb)), __dsub_rn(hi, bb));
    const double l = __dadd_rn(__dadd_rn(a.lo, lo), e);
    a.hi = __dadd_rn(s, l);
    a.lo = __dsub_rn(l, __dsub_rn(a.hi, s));
}

// ---------------------------------------------------------------- kernel
template <typename T, bool CL>
__global__ void __launch_bounds__(SLAB_THREADS<T, CL>, 1)
    k_md_slab(SysDev S, SlabDev D, long long step0, long long nsteps, int phase_half) {
    using V = typename V2<T>::type;
    __shared__ int s_w[33];
    __shared__ unsigned s_vm[SLAB_MAX_THREADS / 32];
    __shared__ double s_dd[4][SLAB_MAX_THREADS / 32];
    __shared__ unsigned s_due[2];                  // by step parity: the next step's is written while this one's is read
    __shared__ long long s_win[MD_MAX_LG], s_next[MD_MAX_LG];   // window that ends, and the step count at which the next ends
    __shared__ int s_before;
    Control *C = S.ctl;
    const RepDev &R = S.reps[0];
    const int tid = threadIdx.x, lane = tid & 31, nt = (int)blockDim.x, nw = nt >> 5;
    const int set = C->set, gcur = C->cur, nset = set ^ 1, slab_order = C->slab_order;
    const int per_lg = S.n_dx * S.nb;
    int *sh_hist = reinterpret_cast<int *>(res_smem);
    SlabMem<T> M;
    M.L = slab_layout<T>(smem_hist_bytes(S.n_lg, S.n_dx, S.nb), D.p_cap, D.h_cap, D.e_cap, D.ncells);
    SlabCta X;
    X.k = (int)blockIdx.x;
    X.g = D.g;
    X.r0 = (int)((long long)X.k * R.nc / X.g);
    X.r1 = (int)((long long)(X.k + 1) * R.nc / X.g);
    X.up = (X.k + 1) % X.g;
    X.down = (X.k + X.g - 1) % X.g;
    X.last = (int)((long long)(X.down + 1) * R.nc / X.g) - (int)((long long)X.down * R.nc / X.g) > 1;
    X.par = 0;
    X.seq = 0;
    if constexpr (CL) {   // every CTA runs: its shared memory may be written
        __shared__ unsigned s_box[2 * SLAB_CLUSTER];
        X.box = s_box;
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    SlabPar<T> P;
    P.h = rd<T>(R.h, R.hf);
    P.rc2 = rd<T>(R.rc2, R.rc2f);
    P.eps24 = T(24) * rd<T>(R.eps, R.epsf);
    P.sig2 = rd<T>(R.sig2, R.sig2f);
    P.hk = rd<T>(R.hk, R.hkf);
    P.dt = rd<T>(R.dt, R.dtf);
    P.vscale = (float)(R.dt / R.half_skin);
    P.rc2f = R.rc2f + R.hf * R.hf * 0x1p-18f;   // as the lists' test
    for (int e = tid; e < S.n_lg * per_lg; e += nt) sh_hist[e] = 0;
    if (tid < S.n_lg) {   // first t = n_equil + m lg_every, m >= 0, after step0
        const long long t = step0 + 1 - S.n_equil, v = S.lg_every[tid];
        s_next[tid] = S.n_equil + (t <= 0 ? 0 : (t + v - 1) / v * v);
    }
    double disp = S.disp_rep[0];
    if (X.k == 0 && tid == 0) C->n_rebuilds += D.counted;
    bool ok = true;
    // ---- load: the slab's slots are contiguous, in the order of the cells'
    // sort or as a slab launch left them
    int first = 0, n;
    if (slab_order) {
        for (int j = 0; j < X.k; ++j) first += D.slab_n[j];
        first += R.pbase;
        n = D.slab_n[X.k];
    } else {
        const int32_t *cs = S.cell_start + R.cbase;
        first = cs[X.r0 * R.nc];
        n = cs[X.r1 * R.nc] - first;
    }
    bool fits = n <= D.p_cap;
    X.p = fits ? n : 0;
    {
        const V *pos = static_cast<const V *>(S.pos[set][gcur]);
        const V *vel = static_cast<const V *>(S.vel[set]);
        for (int i = tid; i < X.p; i += nt) {
            M.put_off(i, pos[first + i]);
            M.vel()[i] = vel[first + i];
            M.cell()[i] = S.cell[set][first + i];
            M.id()[i] = S.pid[set][first + i];
        }
    }
    __syncthreads();
    if (!CL && S.dbg_leave_cta == X.k) return;   // the self-test: one CTA never posts
    fits = slab_publish_rows<T>(D, M, X) && fits;
    unsigned over = slab_sync<CL>(S, D, X, !fits, ok);
    if (!ok) return;
    if (!over) {
        slab_read_rows<T>(D, M, X);
        // (lists between two rebuilds: the limit nbr_max is one of rebuilds)
        over = slab_sync<CL>(S, D, X, !slab_lists<T>(R, D, M, X, RES_MAXLIST, s_w), ok);
        if (!ok) return;
    }
    if (over) {   // nothing was changed: all steps are left
        if (X.k == 0 && tid == 0) {
            *D.left = nsteps;
            C->slab_ends += 1;
        }
        return;
    }
    long long it = 0;
    bool early = false;   // a slab outgrew its room
    int extra = 0;        // leavers still counted here when the launch ends early
    for (; it < nsteps; ++it) {
        const long long s = step0 + it;
        if (tid == nt - 32) {
            unsigned due = 0;
            for (int k = 0; k < S.n_lg; ++k) {
                if (s + 1 == s_next[k]) {
                    due |= 1u << k;
                    s_win[k] = (s_next[k] - S.n_equil) / S.lg_every[k] - 1;
                    s_next[k] += S.lg_every[k];
                }
            }
            s_due[it & 1] = due;
        }
        // ---- forces and kick, then drift
        float vm = 0.0f;
        bool bad = false;
        slab_forces(S, M, X, P, it == 0 && phase_half == 0, S.dbg_fx && it == nsteps - 1, vm, bad);
        const unsigned vb = __reduce_max_sync(0xffffffffu, __float_as_uint(vm));   // non-negative floats order as uints
        if (lane == 0) s_vm[tid >> 5] = vb;
        if (bad) atomicOr(&C->status, (int)DS_NONFINITE);
        __syncthreads();
        {
            const int npar = X.par ^ 1;
            V *pub = static_cast<V *>(D.halo_off) + ((size_t)X.k * 4 + npar) * D.h_cap;   // side 0; side 1: + 2 h_cap
            for (int i = tid; i < X.p; i += nt) {
                V o = M.off()[i];
                const V v = M.vel()[i];
                o.x = axpyT(o.x, P.dt, v.x);
                o.y = axpyT(o.y, P.dt, v.y);
                M.put_off(i, o);
                if (X.g > 1) {
                    const uint16_t b = M.bpos()[i];
                    if (b != RES_NOB) pub[(b >> 15 ? 2 * (size_t)D.h_cap : 0) + (b & 0x7fffu)] = o;
                }
            }
            X.par = npar;
        }
        unsigned vmax = 0;
        if (tid == 0)
            for (int w = 0; w < nw; ++w) vmax = max(vmax, s_vm[w]);
        vmax = slab_sync<CL>(S, D, X, vmax, ok);
        if (!ok) return;
        slab_read_offsets<T>(D, M, X);
        disp += (double)__uint_as_float(vmax) * 1.0000001;
        // ---- sampling pass (Eq. n_i), the arithmetic of the global engine
        const unsigned due = s_due[it & 1];
        if (due) {
            for (int k = 0; k < S.n_lg; ++k) {
                if (!(due >> k & 1u)) continue;
                const bool bin = s_win[k] >= 0;
                DD a2{0.0, 0.0}, a4{0.0, 0.0};
                for (int base = 0; base < X.p; base += nt) {
                    const int i = base + tid;
                    int bins[MD_MAX_DX] = {-1, -1, -1, -1};
                    double m2 = 0.0, m4 = 0.0;
                    if (i < X.p)
                        sample_particle<T>(S, R, 0, k, bin, M.id()[i], M.cell()[i], M.off()[i], bins, m2, m4);
                    if (bin) {
                        for (int d = 0; d < S.n_dx; ++d)
                            warp_hist_add(sh_hist + k * per_lg + d * S.nb, bins[d], lane);
                        dd_add(a2, m2, 0.0);
                        dd_add(a4, m4, 0.0);
                    }
                }
                if (!bin) continue;
                for (int o = 16; o > 0; o >>= 1) {
                    const double h2 = __shfl_xor_sync(0xffffffffu, a2.hi, o), l2 = __shfl_xor_sync(0xffffffffu, a2.lo, o);
                    const double h4 = __shfl_xor_sync(0xffffffffu, a4.hi, o), l4 = __shfl_xor_sync(0xffffffffu, a4.lo, o);
                    dd_add(a2, h2, l2);
                    dd_add(a4, h4, l4);
                }
                __syncthreads();
                if (lane == 0) {
                    s_dd[0][tid >> 5] = a2.hi;
                    s_dd[1][tid >> 5] = a2.lo;
                    s_dd[2][tid >> 5] = a4.hi;
                    s_dd[3][tid >> 5] = a4.lo;
                }
                __syncthreads();
                if (tid < 2) {
                    DD t{0.0, 0.0};
                    for (int w = 0; w < nw; ++w) dd_add(t, s_dd[2 * tid][w], s_dd[2 * tid + 1][w]);
                    S.mom[((long long)(R.pbase / 32 + X.k) * S.n_lg + k) * 2 + tid] += t.hi;
                }
            }
            __syncthreads();
            flush_hist(S, sh_hist, 0, due, s_win);
            __syncthreads();   // s_win is rewritten
        }
        if (disp < 1.0) continue;
        __syncthreads();
        // ---- rebuild: canonical cells, migration, boundary rows, lists
        disp = 0.0;
        if (X.k == 0 && tid == 0) C->n_rebuilds += 1;
        const T h = P.h;
        for (int i = tid; i < X.p; i += nt) {
            V o = M.off()[i];
            const uint32_t cpk = M.cell()[i];
            const int sx = o.x >= h ? 1 : (o.x < T(0) ? -1 : 0);
            const int sy = o.y >= h ? 1 : (o.y < T(0) ? -1 : 0);
            o.x -= (T)sx * h;
            o.y -= (T)sy * h;
            M.put_off(i, o);
            M.cell()[i] = (uint32_t)wrap1((int)(cpk & 0xffffu) + sx, R.nc) |
                          ((uint32_t)wrap1((int)(cpk >> 16) + sy, R.nc) << 16);
        }
        __syncthreads();
        if (X.g > 1) {
            // leaving through the top (row r1) -> direction 0, the bottom -> 1;
            // the leavers are copied out, then the stayers compacted in place
            // (every read of a round precedes its writes)
            const int top = X.r1 == R.nc ? 0 : X.r1;
            int nout[2] = {0, 0};
            const auto dir_of = [&](int i) {
                const int cy = (int)(M.cell()[i] >> 16);
                return cy >= X.r0 && cy < X.r1 ? -1 : (cy == top ? 0 : 1);
            };
            V *mo = static_cast<V *>(D.mig_off), *mv = static_cast<V *>(D.mig_vel);
            for (int base = 0; base < X.p; base += nt) {
                const int i = base + tid, dir = i < X.p ? dir_of(i) : -1;
                int tot;   // both directions' counts in one scan
                const int ex = block_excl_scan(dir == 0 ? 1 : (dir == 1 ? 1 << 16 : 0), s_w, &tot);
                const int t0 = tot & 0xffff, t1 = tot >> 16;
                const int at = dir == 0 ? nout[0] + (ex & 0xffff) : nout[1] + (ex >> 16);
                if (dir >= 0 && at < D.h_cap) {
                    const size_t gi = ((size_t)X.k * 2 + dir) * D.h_cap + at;
                    mo[gi] = M.off()[i];
                    mv[gi] = M.vel()[i];
                    D.mig_ci[gi] = make_uint2(M.cell()[i], (uint32_t)M.id()[i]);
                }
                nout[0] += t0;
                nout[1] += t1;
            }
            if (tid < 2) D.mig_n[X.k * 2 + tid] = nout[tid];
            over = slab_sync<CL>(S, D, X, nout[0] > D.h_cap || nout[1] > D.h_cap, ok);
            if (!ok) return;
            if (over) {   // nobody has moved yet
                early = true;
                ++it;
                break;
            }
            int keep = 0;
            for (int base = 0; base < X.p; base += nt) {
                const int i = base + tid;
                V o{}, v{};
                uint32_t c = 0;
                int id = 0;
                const bool stay = i < X.p && dir_of(i) < 0;
                if (stay) {
                    o = M.off()[i];
                    v = M.vel()[i];
                    c = M.cell()[i];
                    id = M.id()[i];
                }
                int tot;
                const int at = keep + block_excl_scan(stay, s_w, &tot);
                if (stay) {
                    M.put_off(at, o);
                    M.vel()[at] = v;
                    M.cell()[at] = c;
                    M.id()[at] = id;
                }
                keep += tot;
                __syncthreads();
            }
            // arrivals: from the down neighbour's top, then the up one's bottom
            const int src[2] = {X.down, X.up};
            const int in0 = *(volatile int32_t *)&D.mig_n[src[0] * 2], in1 = *(volatile int32_t *)&D.mig_n[src[1] * 2 + 1];
            fits = keep + in0 + in1 <= D.p_cap;
            for (int t = tid; fits && t < in0 + in1; t += nt) {
                const size_t gi = t < in0 ? ((size_t)src[0] * 2) * D.h_cap + t : ((size_t)src[1] * 2 + 1) * D.h_cap + t - in0;
                const uint2 ci = __ldcg(&D.mig_ci[gi]);
                M.put_off(keep + t, __ldcg(&mo[gi]));
                M.vel()[keep + t] = __ldcg(&mv[gi]);
                M.cell()[keep + t] = ci.x;
                M.id()[keep + t] = (int32_t)ci.y;
            }
            X.p = fits ? keep + in0 + in1 : keep;
            __syncthreads();
            fits = slab_publish_rows<T>(D, M, X) && fits;
            over = slab_sync<CL>(S, D, X, !fits, ok);
            if (!ok) return;
            if (over) {   // every slab writes its stayers and its own leavers
                X.p = keep;
                extra = nout[0] + nout[1];
                early = true;
                ++it;
                break;
            }
            slab_read_rows<T>(D, M, X);
        }
        over = slab_sync<CL>(S, D, X, !slab_lists<T>(R, D, M, X, min(S.K, RES_MAXLIST), s_w), ok);
        if (!ok) return;
        if (over) {
            early = true;
            ++it;
            break;
        }
    }
    // ---- write back into the other set, slab after slab
    const int own = X.p + extra;
    slab_sync<CL>(S, D, X, (unsigned)own, ok);
    if (!ok) return;
    if (tid == 0) s_before = slab_before<CL>(D, X);
    __syncthreads();
    {
        V *pos = static_cast<V *>(S.pos[nset][0]);
        V *vel = static_cast<V *>(S.vel[nset]);
        const int b = R.pbase + s_before;
        for (int i = tid; i < X.p; i += nt) {
            pos[b + i] = M.off()[i];
            vel[b + i] = M.vel()[i];
            S.cell[nset][b + i] = M.cell()[i];
            S.pid[nset][b + i] = M.id()[i];
        }
        if (extra) {
            const V *mo = static_cast<const V *>(D.mig_off), *mv = static_cast<const V *>(D.mig_vel);
            const int n0 = D.mig_n[X.k * 2];
            for (int t = tid; t < extra; t += nt) {
                const size_t gi = t < n0 ? ((size_t)X.k * 2) * D.h_cap + t : ((size_t)X.k * 2 + 1) * D.h_cap + t - n0;
                pos[b + X.p + t] = mo[gi];
                vel[b + X.p + t] = mv[gi];
                S.cell[nset][b + X.p + t] = D.mig_ci[gi].x;
                S.pid[nset][b + X.p + t] = (int32_t)D.mig_ci[gi].y;
            }
        }
        if (tid == 0) D.slab_n[X.k] = own;
    }
    // every CTA has read the set index (it passed an exchange since)
    if (X.k == 0 && tid == 0) {
        C->set = nset;
        C->cur = 0;
        // a state left early is sorted by the global engine, which then runs
        // the steps left (possibly none)
        C->slab_order = !early;
        C->slab_ends += early;
        *D.left = nsteps - it;
        S.disp_rep[0] = disp;
    }
}

}  // namespace mdlg
