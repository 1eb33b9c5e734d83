// resample.cu -- population set-up, resampling, gather and observables.
//
// PAMD scheme, step 1 (init), step 2 (resampling with relative Boltzmann
// weights, velocity rescaling) and step 4 (population averages with
// family-binned errors).  Everything here is O(R) work between the
// propagate launches; the gather is the one HBM-bound kernel.
#include <cooperative_groups.h>
#include <math.h>

#include "pamd_device.cuh"
#include "pamd_internal.h"

namespace pamd {

constexpr int kScanBlock = 1024;  // elements per scan block (256 threads x 4)
constexpr int kScanThreads = 256;

// ------------------------------------------------------------------ helpers

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T n = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += n;
    }
    return v;
}

// Inclusive scan of the 4 values held by each of the 256 threads (1024
// consecutive elements); returns the block total.
template <typename T>
__device__ __forceinline__ T block_scan4(T (&v)[4], T* sh /* [8] */) {
    v[1] += v[0];
    v[2] += v[1];
    v[3] += v[2];
    const T tsum = v[3];
    const T incl = warp_incl_scan(tsum);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 31) sh[w] = incl;
    __syncthreads();
    T wpre = 0, total = 0;
#pragma unroll
    for (int i = 0; i < kScanThreads / 32; ++i) {
        if (i < w) wpre += sh[i];
        total += sh[i];
    }
    const T pre = wpre + incl - tsum;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] += pre;
    __syncthreads();
    return total;
}

// Sum in a fixed tree order (deterministic for a given launch shape).
__device__ __forceinline__ double block_sum_d(double v, double* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) sh[w] = v;
    __syncthreads();
    double s = 0.0;
    for (int i = 0; i < nw; ++i) s += sh[i];
    __syncthreads();
    return s;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ------------------------------------------------------------------ init

// Step 1: x = recentred start geometry, v ~ Maxwell-Boltzmann(T0) from
// Philox(seed; atom, slot, 0, INIT | mol << 8), family = slot.
__global__ void init_kernel(float* state, double* E, int32_t* fam, const float* x0,
                            const float* masses, long long R, int N, int Np, float kT0,
                            unsigned long long seed, uint32_t purpose) {
    const long long total = R * (long long)Np;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long k = t / Np;
        const int i = (int)(t - k * Np);
        float* st = state + (size_t)k * 6 * Np;
        if (i < N) {
            const float3 z = normal3(seed, (uint32_t)i, (uint32_t)k, 0u, purpose);
            const float sdv = sqrtf(kT0 / masses[i]);
            st[i] = x0[i];
            st[Np + i] = x0[Np + i];
            st[2 * Np + i] = x0[2 * Np + i];
            st[3 * Np + i] = sdv * z.x;
            st[4 * Np + i] = sdv * z.y;
            st[5 * Np + i] = sdv * z.z;
        } else {
#pragma unroll
            for (int c = 0; c < 6; ++c) st[c * Np + i] = 0.0f;
        }
        if (i == 0) {
            fam[k] = (int32_t)k;
            E[k] = 0.0;
        }
    }
}

__global__ void reset_scalars_kernel(DevScalars* s) {
    s->m = 0.0;
    s->S = 0.0;
    s->lnQ = 0.0;
    s->sum_lnQ = 0.0;
    s->C_total = 0ull;
    s->max_copies = 1;
    s->status = 0;
    s->bad_replica = -1;
}

__global__ void set_counters_kernel(uint32_t* ctr, uint32_t step, uint32_t ridx) {
    ctr[0] = step;
    ctr[1] = ridx;
}

// Population size of a context with a variable population (device counter
// word 2, read by every kernel that loops over the population).
__global__ void set_live_kernel(uint32_t* ctr, uint32_t live) { ctr[2] = live; }

// Live population size: *live when the population size varies, else R.
__device__ __forceinline__ long long live_size(const uint32_t* live, long long R) {
    return live ? (long long)*live : R;
}

// ------------------------------------------------------------------ weights

// Order-preserving map of a double's bits to a signed 64-bit key (no NaN):
// the maximum then runs on the integer units.  Its own inverse.
__device__ __forceinline__ long long order_key(double v) {
    const long long b = __double_as_longlong(v);
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double key_value(long long k) {
    return __longlong_as_double(k >= 0 ? k : (k ^ 0x7fffffffffffffffLL));
}

// Maximum over the block of integer keys; thread 0 has it.
__device__ __forceinline__ long long block_max_key(long long k, long long* sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = k;
    __syncthreads();
    if (threadIdx.x < 32) {
        k = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : order_key(-INFINITY);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) k = max(k, __shfl_xor_sync(0xffffffffu, k, o));
    }
    return k;
}

// a_j = -(beta_next - beta_prev) E_j ; block maxima.  On integer keys: FP64
// comparisons and conversions of every warp were most of these two kernels'
// time (2^20 replicas: 16 + 14 us, now 7.7 + 3.0).
__global__ void amax_kernel(const double* E, long long R, double dbeta, double* blk_max,
                            const uint32_t* live) {
    __shared__ long long sh[32];
    R = live_size(live, R);
    const long long base = (long long)blockIdx.x * kScanBlock;
    long long k = order_key(-INFINITY);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        if (j < R && isfinite(E[j])) k = max(k, order_key(__dmul_rn(-dbeta, E[j])));
    }
    k = block_max_key(k, sh);
    if (threadIdx.x == 0) blk_max[blockIdx.x] = key_value(k);
}

__global__ void max_top_kernel(const double* blk_max, int nblk, DevScalars* s) {
    __shared__ long long sh[32];
    long long k = order_key(-INFINITY);
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) k = max(k, order_key(blk_max[b]));
    k = block_max_key(k, sh);
    if (threadIdx.x == 0) s->m = key_value(k);
}

// W_j = floor(2^s exp_det(a_j - m)); block sums of W (exact) and of the
// exponentials (for Q).
__global__ void weights_kernel(const double* E, long long R, double dbeta, double two_s,
                               DevScalars* s, ExpCoef cf, unsigned long long* W,
                               unsigned long long* blk_w, double* blk_e, const uint32_t* live) {
    __shared__ double sh[32];
    __shared__ unsigned long long shw[8];
    if (live) {  // 2^s with s = 63 - ceil(log2 R) of the live population
        R = (long long)*live;
        const int bits = (R > 1) ? 64 - __clzll((unsigned long long)(R - 1)) : 0;
        two_s = ldexp(1.0, 63 - bits);
    }
    const long long base = (long long)blockIdx.x * kScanBlock;
    const double m = s->m;
    unsigned long long w[4];
    double es = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        w[q] = 0ull;
        if (j < R) {
            const double Ej = E[j];
            double e = 0.0;
            if (isfinite(Ej)) {
                const double a = __dmul_rn(-dbeta, Ej);
                e = exp_det(__dsub_rn(a, m), cf);
                w[q] = __double2ull_rz(__dmul_rn(two_s, e));
            } else if (atomicCAS(&s->status, 0, PAMD_ENONFINITE) == 0) {
                s->bad_replica = (int)j;  // a non-finite energy gets weight 0
            }
            W[j] = w[q];
            es += e;
        }
    }
    const double bs = block_sum_d(es, sh);
    const unsigned long long tot = block_scan4(w, shw);
    if (threadIdx.x == 0) {
        blk_w[blockIdx.x] = tot;
        blk_e[blockIdx.x] = bs;
    }
}

// Exclusive scan of the block sums of W (in place), C_total, ln Q.
__global__ void weights_top_kernel(unsigned long long* blk_w, const double* blk_e, int nblk,
                                   long long R, DevScalars* s, const uint32_t* live) {
    R = live_size(live, R);
    __shared__ unsigned long long shw[8];
    __shared__ unsigned long long carry;
    if (threadIdx.x == 0) carry = 0ull;
    __syncthreads();
    for (int b0 = 0; b0 < nblk; b0 += kScanBlock) {
        unsigned long long v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = b0 + threadIdx.x * 4 + q;
            v[q] = (b < nblk) ? blk_w[b] : 0ull;
        }
        unsigned long long orig[4] = {v[0], v[1], v[2], v[3]};
        const unsigned long long tot = block_scan4(v, shw);
        const unsigned long long c = carry;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = b0 + threadIdx.x * 4 + q;
            if (b < nblk) blk_w[b] = c + v[q] - orig[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) carry = c + tot;
        __syncthreads();
    }
    // S = sum of the block sums in a fixed order: each thread a contiguous
    // chunk, then a fixed shuffle tree per warp, then the warps in order
    __shared__ double wsum[32];
    double part = 0.0;
    {
        const int per = (nblk + blockDim.x - 1) / blockDim.x;
        const int lo = threadIdx.x * per, hi = min(lo + per, nblk);
        for (int b = lo; b < hi; ++b) part += blk_e[b];
    }
    for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double S = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) S += wsum[w];
        s->S = S;
        s->C_total = carry;
        const double lnq = s->m + (log(S) - log((double)R));
        s->lnQ = lnq;
        s->sum_lnQ += lnq;
    }
}

// C_j = block offset + inclusive scan of W inside the block.
__global__ void scan_local_u64_kernel(unsigned long long* W, long long R,
                                      const unsigned long long* blk_off, unsigned long long* C,
                                      const uint32_t* live) {
    __shared__ unsigned long long shw[8];
    R = live_size(live, R);
    const long long base = (long long)blockIdx.x * kScanBlock;
    unsigned long long v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        v[q] = (j < R) ? W[j] : 0ull;
    }
    block_scan4(v, shw);
    const unsigned long long off = blk_off[blockIdx.x];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        if (j < R) C[j] = off + v[q];
    }
}

// ------------------------------------------------------------------ counts

// Target of draw k.  Multinomial (rule 1): u_k from Philox(seed; k, resampling
// index, 0, RESAMPLE | mol << 8), t = floor(u_k C_total / 2^64).  Systematic
// (rule 2): t_k = floor((k C + V) / R), V = floor(u_0 C / 2^64), by long
// division in 32-bit digits (the numerator is below 2^84 and the quotient
// below C).
__device__ __forceinline__ unsigned long long draw_target(long long k, long long R, unsigned long long total, int rule,
                                                          unsigned long long seed, uint32_t ridx, uint32_t purpose) {
    const uint4 o = philox4x32_10(make_uint4(rule == 2 ? 0u : (uint32_t)k, ridx, 0u, purpose), seed_key(seed));
    const unsigned long long u = (unsigned long long)o.x | ((unsigned long long)o.y << 32);
    const unsigned long long V = __umul64hi(u, total);
    if (rule != 2) return V;
    const unsigned long long plo = (unsigned long long)k * total;  // low 64 bits of k C
    unsigned long long phi = __umul64hi((unsigned long long)k, total);
    const unsigned long long lo64 = plo + V;
    phi += (lo64 < plo) ? 1ull : 0ull;
    const unsigned long long r64 = (unsigned long long)R;
    unsigned long long rem = phi % r64;  // phi < R: the quotient's high word is zero
    unsigned long long cur = (rem << 32) | (lo64 >> 32);
    const unsigned long long q1 = cur / r64;
    rem = cur % r64;
    cur = (rem << 32) | (lo64 & 0xffffffffull);
    const unsigned long long q0 = cur / r64;
    return (q1 << 32) | q0;
}

// Draw k: ancestor = first j with C_j > target.
__global__ void counts_kernel(const unsigned long long* C, long long R, const DevScalars* s,
                              unsigned long long seed, const uint32_t* dev_counters,
                              uint32_t ridx_off, uint32_t purpose, int do_resample,
                              int32_t* cnt, const uint32_t* live) {
    R = live_size(live, R);
    const uint32_t ridx = (dev_counters ? dev_counters[1] : 0u) + ridx_off;
    const unsigned long long total = s->C_total;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < R;
         k += (long long)gridDim.x * blockDim.x) {
        if (!do_resample) {
            cnt[k] = 1;
            continue;
        }
        const unsigned long long t = draw_target(k, R, total, do_resample, seed, ridx, purpose);
        long long lo = 0, hi = R;
        while (lo < hi) {
            const long long mid = lo + ((hi - lo) >> 1);
            if (C[mid] > t) hi = mid;
            else lo = mid + 1;
        }
        // t < C_total whenever C_total > 0, so lo < R; the clamp only guards
        // a population whose weights are all zero (all energies non-finite)
        atomicAdd(&cnt[lo < R ? lo : R - 1], 1);
    }
}

// ------------------------------------------------------------------ one launch
//
// Weights, prefix sums, draws, copy counts and ancestors of a population of up
// to kClusterMaxR replicas in one launch: a cluster of up to eight CTAs, each
// with a chunk of the population in shared memory, exchanging maxima, totals,
// search probes and count increments through distributed shared memory.  Same
// integer weights, targets and ancestors as the kernels above, bit for bit;
// only the sum behind ln Q is taken in another order.
// Bound by latency: six cluster barriers, one binary search and, per element,
// one FP64 exponential (maxima run on integer keys and block sums in one warp:
// an FP64 instruction of all 16 warps costs 256 cycles).  12 us at R = 256 and
// 33 us at R = 8192; the separate kernels and a cleared count array take 42
// and 64 us and eight more launches.  A chunk of more than 2048 would spend
// longer on its exponentials (5.5 us per 1024) than the launches saved, and
// eight CTAs are the portable cluster size: above 16384 replicas the separate
// kernels, spread over all SMs, are used.
constexpr int kClusterThreads = 512, kClusterCtas = 8, kClusterMaxPer = 4;
constexpr long long kClusterMaxR = (long long)kClusterThreads * kClusterCtas * kClusterMaxPer;

struct ClusterArgs {
    const double* E;
    long long R;
    double dbeta, two_s;
    DevScalars* s;
    ExpCoef cf;
    unsigned long long seed;
    const uint32_t* dev_counters;
    uint32_t ridx_off, purpose;
    int rule;                // 0: every copy once, 1 multinomial, 2 systematic
    int32_t *cnt, *incl, *anc;
};

// inclusive scan over the block of PER consecutive values per thread; returns the total
template <typename T, int PER>
__device__ __forceinline__ T block_scan(T (&v)[PER], T* sh) {
#pragma unroll
    for (int q = 1; q < PER; ++q) v[q] += v[q - 1];
    const T mine = v[PER - 1];
    const T incl = warp_incl_scan(mine);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 31) sh[w] = incl;
    __syncthreads();
    T pre = incl - mine, total = 0;
#pragma unroll
    for (int i = 0; i < kClusterThreads / 32; ++i) {
        const T x = sh[i];
        if (i < w) pre += x;
        total += x;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) v[q] += pre;
    __syncthreads();
    return total;
}

template <int PER>
__global__ void __launch_bounds__(kClusterThreads) resample_cluster_kernel(const ClusterArgs g) {
    namespace cg = cooperative_groups;
    constexpr int kChunk = kClusterThreads * PER;
    __shared__ unsigned long long sC[kChunk];
    __shared__ int32_t sN[kChunk];
    __shared__ unsigned long long shw[kClusterThreads / 32];
    __shared__ double shd[kClusterThreads / 32];
    __shared__ long long shk[kClusterThreads / 32];
    __shared__ int32_t shi[kClusterThreads / 32], sht[kClusterThreads / 32];
    // this CTA's contributions, read by the others
    __shared__ long long x_max;
    __shared__ double x_sum;
    __shared__ unsigned long long x_w;
    __shared__ int32_t x_n, x_top;
    __shared__ unsigned long long w_end[kClusterCtas];  // inclusive sums of the CTAs' totals
    __shared__ int32_t n_end[kClusterCtas];
    constexpr int kWarps = kClusterThreads / 32;
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    const long long j0 = (long long)rank * kChunk + (long long)threadIdx.x * PER;
    // a_j and the maximum
    double a[PER];
    long long mk = order_key(-INFINITY);
    bool ok[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const bool in = j0 + q < g.R;
        const double e = in ? g.E[j0 + q] : 0.0;
        ok[q] = in && isfinite(e);
        if (in && !ok[q] && atomicCAS(&g.s->status, 0, PAMD_ENONFINITE) == 0)
            g.s->bad_replica = (int)(j0 + q);  // a non-finite energy gets weight 0
        a[q] = ok[q] ? __dmul_rn(-g.dbeta, e) : 0.0;
        if (ok[q]) mk = max(mk, order_key(a[q]));
        sN[threadIdx.x * PER + q] = 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mk = max(mk, __shfl_xor_sync(0xffffffffu, mk, o));
    if (lane == 0) shk[wp] = mk;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kWarps; ++i) mk = max(mk, shk[i]);
        x_max = mk;
    }
    cl.sync();
    mk = order_key(-INFINITY);
    for (int r = 0; r < ctas; ++r) mk = max(mk, *cl.map_shared_rank(&x_max, r));
    const double m = key_value(mk);
    // integer weights and their prefix sums
    unsigned long long w[PER];
    double es = 0.0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        double e = 0.0;
        w[q] = 0ull;
        if (ok[q]) {
            e = exp_det(__dsub_rn(a[q], m), g.cf);
            w[q] = __double2ull_rz(__dmul_rn(g.two_s, e));
        }
        es = q ? es + e : e;
    }
    es = warp_sum_d(es);
    if (lane == 0) shd[wp] = es;
    const unsigned long long wt = block_scan(w, shw);  // orders the writes of shd as well
    if (threadIdx.x == 0) {
        for (int i = 1; i < kWarps; ++i) es += shd[i];
        x_sum = es;
        x_w = wt;
    }
    cl.sync();
    if (threadIdx.x == 0) {
        unsigned long long c = 0;
        for (int r = 0; r < ctas; ++r) w_end[r] = c += *cl.map_shared_rank(&x_w, r);
    }
    __syncthreads();
    const unsigned long long total = w_end[ctas - 1], woff = rank ? w_end[rank - 1] : 0ull;
#pragma unroll
    for (int q = 0; q < PER; ++q) sC[threadIdx.x * PER + q] = woff + w[q];
    cl.sync();
    // the last warp forms ln Q while the others search
    if (rank == 0 && threadIdx.x == kClusterThreads - 1) {
        double S = 0.0;
        for (int r = 0; r < ctas; ++r) S += *cl.map_shared_rank(&x_sum, r);
        const double lnq = m + (log(S) - log((double)g.R));
        g.s->m = m;
        g.s->S = S;
        g.s->C_total = total;
        g.s->lnQ = lnq;
        g.s->sum_lnQ += lnq;
    }
    // draws: the CTA that holds the ancestor, then a search of its chunk, all
    // of a thread's draws side by side
    const uint32_t ridx = (g.dev_counters ? g.dev_counters[1] : 0u) + g.ridx_off;
    if (!g.rule) {
#pragma unroll
        for (int q = 0; q < PER; ++q)
            if (j0 + q < g.R) sN[threadIdx.x * PER + q] = 1;
    } else {
        unsigned long long t[PER];
        const unsigned long long* chunk[PER];
        int rr[PER], at[PER];
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            t[q] = draw_target(j0 + q, g.R, total, g.rule, g.seed, ridx, g.purpose);
            int r = 0;
            while (r < ctas - 1 && w_end[r] <= t[q]) ++r;
            rr[q] = r;
            chunk[q] = cl.map_shared_rank(sC, r);
            at[q] = 0;  // elements known to be <= t
        }
#pragma unroll
        for (int h = kChunk / 2; h > 0; h >>= 1)
#pragma unroll
            for (int q = 0; q < PER; ++q)
                if (chunk[q][at[q] + h - 1] <= t[q]) at[q] += h;
#pragma unroll
        for (int q = 0; q < PER; ++q) {
            if (j0 + q >= g.R) continue;
            if (chunk[q][at[q]] <= t[q]) ++at[q];
            long long j = (long long)rr[q] * kChunk + at[q];
            // only a population whose weights are all zero reaches the clamp
            if (j >= g.R) j = g.R - 1;
            const int r = (int)(j / kChunk);
            atomicAdd(cl.map_shared_rank(sN, r) + (j - (long long)r * kChunk), 1);
        }
    }
    cl.sync();
    // copy counts and their prefix sums
    int32_t n[PER], cnt[PER], top = 0;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        cnt[q] = n[q] = sN[threadIdx.x * PER + q];
        top = max(top, n[q]);
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) sht[wp] = top;
    const int32_t nt = block_scan(n, shi);
    if (threadIdx.x == 0) {
        for (int i = 1; i < kWarps; ++i) top = max(top, sht[i]);
        x_n = nt;
        x_top = top;
    }
    cl.sync();
    if (threadIdx.x == 0) {
        int32_t c = 0, t = 0;
        for (int r = 0; r < ctas; ++r) {
            n_end[r] = c += *cl.map_shared_rank(&x_n, r);
            t = max(t, *cl.map_shared_rank(&x_top, r));
        }
        if (rank == 0) {
            g.s->max_copies = t;
            g.s->R_new = c;  // size of the new population (sum of the copy counts)
        }
    }
    __syncthreads();
    const int32_t noff = rank ? n_end[rank - 1] : 0;
    // ancestors of the new slots: each ancestor fills its own, the whole warp
    // those of an ancestor with many copies
#pragma unroll
    for (int q = 0; q < PER; ++q) {
        const int32_t end = noff + n[q], c = cnt[q];
        if (j0 + q < g.R) {
            g.cnt[j0 + q] = c;
            g.incl[j0 + q] = end;
        }
        if (c <= 4)
            for (int i = 0; i < c; ++i) g.anc[end - c + i] = (int32_t)(j0 + q);
        unsigned many = __ballot_sync(0xffffffffu, c > 4);
        while (many) {
            const int l = __ffs(many) - 1;
            many &= many - 1;
            const int32_t lc = __shfl_sync(0xffffffffu, c, l), le = __shfl_sync(0xffffffffu, end, l);
            const int32_t lj = (int32_t)__shfl_sync(0xffffffffu, j0 + q, l);
            for (int i = lane; i < lc; i += 32) g.anc[le - lc + i] = lj;
        }
    }
    cl.sync();  // no CTA leaves while another reads its shared memory
}

cudaError_t launch_resample_cluster(const ClusterArgs& g, cudaStream_t s) {
    int ctas = 1;
    while (ctas < kClusterCtas && (long long)ctas * kClusterThreads < g.R) ctas *= 2;
    const long long per = (g.R + (long long)ctas * kClusterThreads - 1) / ((long long)ctas * kClusterThreads);
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kClusterThreads);
    cfg.stream = s;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (per <= 1) return cudaLaunchKernelEx(&cfg, resample_cluster_kernel<1>, g);
    if (per <= 2) return cudaLaunchKernelEx(&cfg, resample_cluster_kernel<2>, g);
    return cudaLaunchKernelEx(&cfg, resample_cluster_kernel<4>, g);
}

// ------------------------------------------------------------------ copy numbers
// of the rules that let the population size vary around a target R_t

// q = floor(a b / c), r = a b - q c exactly, for a < 2^32, b <= c, c >= 1:
// an FP64 estimate corrected in 128-bit integer arithmetic.
__device__ __forceinline__ void muldiv_exact(unsigned long long a, unsigned long long b,
                                             unsigned long long c, unsigned long long& q,
                                             unsigned long long& r) {
    const unsigned long long plo = a * b, phi = __umul64hi(a, b);
    unsigned long long qq = (unsigned long long)__ddiv_rn(
        __dmul_rn(__ull2double_rn(a), __ull2double_rn(b)), __ull2double_rn(c));
    for (int it = 0; it < 8; ++it) {
        const unsigned long long tlo = qq * c, thi = __umul64hi(qq, c);
        if (thi > phi || (thi == phi && tlo > plo)) {  // qq c > a b
            --qq;
            continue;
        }
        const unsigned long long rlo = plo - tlo;
        const unsigned long long rhi = phi - thi - (plo < tlo ? 1ull : 0ull);
        if (rhi == 0ull && rlo < c) {
            q = qq;
            r = rlo;
            return;
        }
        ++qq;
    }
    q = qq;  // not reached: the estimate is within one of the quotient
    r = 0ull;
}

// Smallest n with F(n) >= u for the Poisson CDF F of mean lam, summed as
// p_0 = e^-lam, p_n = (p_{n-1} lam) / n (every operation rounded to FP64 as
// written); at most floor(lam + 20 sqrt(lam)) + 50.
__device__ __forceinline__ long long poisson_inverse(double lam, double u, const ExpCoef& cf) {
    const long long n_max = (long long)floor(__dadd_rn(lam, __dmul_rn(20.0, __dsqrt_rn(lam)))) + 50;
    double p = exp_det(-lam, cf);
    double F = p;
    long long n = 0;
    while (u > F && n < n_max) {
        ++n;
        p = __ddiv_rn(__dmul_rn(p, lam), (double)n);
        F = __dadd_rn(F, p);
    }
    return n;
}

// Copy numbers of ancestor j with E[n_j] = tau_j = R_t W_j / C (C = sum of
// the integer weights W of the live population): rule 3 nearest integer
// (floor(tau_j) plus a Bernoulli draw of the fractional part), rule 4
// Poisson (CDF inversion, in chunks of at most 500 of the mean).
__global__ void varsize_counts_kernel(const unsigned long long* W, long long R, const DevScalars* s,
                                      long long R_target, unsigned long long seed,
                                      const uint32_t* dev_counters, uint32_t ridx_off,
                                      uint32_t purpose, int rule, ExpCoef cf, int32_t* cnt,
                                      const uint32_t* live) {
    R = live_size(live, R);
    const uint32_t ridx = (dev_counters ? dev_counters[1] : 0u) + ridx_off;
    const unsigned long long C = s->C_total;
    for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < R;
         j += (long long)gridDim.x * blockDim.x) {
        long long n = 0;
        if (C > 0ull && rule == 3) {
            unsigned long long q, r;
            muldiv_exact((unsigned long long)R_target, W[j], C, q, r);
            const uint4 o = philox4x32_10(make_uint4((uint32_t)j, ridx, 0u, purpose), seed_key(seed));
            const unsigned long long u = (unsigned long long)o.x | ((unsigned long long)o.y << 32);
            n = (long long)q + ((__umul64hi(u, C) < r) ? 1 : 0);
        } else if (C > 0ull) {
            const double lam = __ddiv_rn(__dmul_rn((double)R_target, __ull2double_rn(W[j])),
                                         __ull2double_rn(C));
            int m = (int)ceil(__ddiv_rn(lam, 500.0));
            m = m < 1 ? 1 : m;
            const double chunk = __ddiv_rn(lam, (double)m);
            for (int c = 0; c < m; ++c) {
                const uint4 o = philox4x32_10(make_uint4((uint32_t)j, ridx, (uint32_t)c, purpose),
                                              seed_key(seed));
                const unsigned long long u64 = (unsigned long long)o.x | ((unsigned long long)o.y << 32);
                const double u = __dmul_rn(__dadd_rn(__ull2double_rn(u64 >> 11), 0.5), 0x1p-53);
                n += poisson_inverse(chunk, u, cf);
            }
        }
        cnt[j] = (int32_t)n;
    }
}

// After the gather: the new population size becomes the live size (at most
// the capacity R); an empty or overflowing population is reported.
__global__ void commit_size_kernel(DevScalars* s, uint32_t* ctr, long long R) {
    const long long n = s->R_new;
    if ((n == 0 || n > R) && atomicCAS(&s->status, 0, PAMD_EPOPSIZE) == 0) s->bad_replica = -1;
    ctr[2] = (uint32_t)(n < R ? n : R);
}

__global__ void cnt_block_kernel(const int32_t* cnt, long long R, int32_t* blk_sum,
                                 int32_t* blk_max, const uint32_t* live) {
    R = live_size(live, R);
    __shared__ int32_t shs[8];
    __shared__ int32_t shm[8];
    const long long base = (long long)blockIdx.x * kScanBlock;
    int32_t v[4], mx = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        v[q] = (j < R) ? cnt[j] : 0;
        mx = max(mx, v[q]);
    }
    const int32_t tot = block_scan4(v, shs);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t m = 0;
        for (int i = 0; i < kScanThreads / 32; ++i) m = max(m, shm[i]);
        blk_sum[blockIdx.x] = tot;
        blk_max[blockIdx.x] = m;
    }
}

__global__ void cnt_top_kernel(int32_t* blk_sum, const int32_t* blk_max, int nblk, DevScalars* s) {
    __shared__ int32_t shs[8];
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int b0 = 0; b0 < nblk; b0 += kScanBlock) {
        int32_t v[4], orig[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = b0 + threadIdx.x * 4 + q;
            v[q] = orig[q] = (b < nblk) ? blk_sum[b] : 0;
        }
        const int32_t tot = block_scan4(v, shs);
        const int32_t c = carry;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int b = b0 + threadIdx.x * 4 + q;
            if (b < nblk) blk_sum[b] = c + v[q] - orig[q];
        }
        __syncthreads();
        if (threadIdx.x == 0) carry = c + tot;
        __syncthreads();
    }
    // largest count: an integer max, the same in any order
    __shared__ int32_t wmax[32];
    int32_t mloc = 0;
    for (int b = threadIdx.x; b < nblk; b += blockDim.x) mloc = max(mloc, blk_max[b]);
    for (int o = 16; o > 0; o >>= 1) mloc = max(mloc, __shfl_down_sync(0xffffffffu, mloc, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mloc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t m = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m = max(m, wmax[w]);
        s->max_copies = m;
        s->R_new = carry;  // size of the new population (sum of the copy counts)
    }
}

__global__ void cnt_local_kernel(const int32_t* cnt, long long R, const int32_t* blk_off,
                                 int32_t* incl, const uint32_t* live) {
    __shared__ int32_t shs[8];
    R = live_size(live, R);
    const long long base = (long long)blockIdx.x * kScanBlock;
    int32_t v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        v[q] = (j < R) ? cnt[j] : 0;
    }
    block_scan4(v, shs);
    const int32_t off = blk_off[blockIdx.x];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const long long j = base + threadIdx.x * 4 + q;
        if (j < R) incl[j] = off + v[q];
    }
}

// ------------------------------------------------------------------ gather

// Ancestor of every new slot: anc[k] = first j with incl_j > k (copies of j
// fill slots incl_{j-1} .. incl_j - 1).  One thread per slot.
// With a variable population (live != null) the ancestors are the live
// population and the new slots number min(R_new, R), R the capacity.
__global__ void ancestor_kernel(const int32_t* __restrict__ incl, long long R, int32_t* anc,
                                const uint32_t* live, const DevScalars* s) {
    long long n_new = R;
    if (live) {
        n_new = s->R_new < R ? s->R_new : R;
        R = (long long)*live;
    }
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n_new;
         k += (long long)gridDim.x * blockDim.x) {
        long long lo = 0, hi = R;
        while (lo < hi) {
            const long long mid = lo + ((hi - lo) >> 1);
            if (incl[mid] > k) hi = mid;
            else lo = mid + 1;
        }
        anc[k] = (int32_t)(lo < R ? lo : R - 1);
    }
}

// One warp per new slot k copies the ancestor's state (6 Np floats, Np % 4 ==
// 0) as P float4s per lane: positions shifted to the centre of mass,
// velocities scaled by vscale, and the new replica's kinetic energy and
// radius of gyration recomputed from the moved state (FP32 sums: GB300's FP64
// rate is a small fraction of its FP32 rate, and every propagate launch
// recomputes these values in FP64).
//
// The copy is HBM work, but the arithmetic around it decides: at 692
// instructions per slot (75 atoms) the issue slots were the bottleneck (66 %
// busy, DRAM 45 %).  What does not change between slots, each float4's
// coordinate, masses and padding, is worked out once per lane; a float4
// column that holds no positions (or no velocities) in any lane skips that
// half by a uniform branch; values of one coordinate are picked by bit masks;
// and the sums of several values share shuffles: after the first butterfly
// step both halves of the warp hold the same sum, so the halves go on with
// different values (the same additions in the same order).  75 atoms, R = 2^20
// (3.83 GB): 638 us, 88 % of the measured copy bandwidth; before, 883 us.
// Bulk copies through shared memory (4 records in flight per warp) took 991 us
// at 2^20: fewer warps for the same instructions.
// The roundings are written out, so that every P (and every change around
// them) gives the same bits.
__device__ __forceinline__ float dot4(const float4 a, const float4 b) {
    return __fmaf_rn(a.w, b.w, __fmaf_rn(a.z, b.z, __fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y))));
}
__device__ __forceinline__ float mass_square(const float4 m, const float4 w) {
    return __fmaf_rn(__fmul_rn(m.w, w.w), w.w,
                     __fmaf_rn(__fmul_rn(m.z, w.z), w.z,
                               __fmaf_rn(__fmul_rn(m.y, w.y), w.y, __fmul_rn(__fmul_rn(m.x, w.x), w.x))));
}

template <int P>
__global__ void __launch_bounds__(256, P <= 4 ? 4 : P <= 8 ? 3 : 2) gather_kernel(
    const float* __restrict__ st_in, float* __restrict__ st_out, const double* E_in,
    double* E_out, const int32_t* fam_in, int32_t* fam_out, double* ke_out, double* rg_out,
    const int32_t* __restrict__ anc, const float* __restrict__ masses, long long R, int N, int Np,
    float vscale, float inv_mtot, const uint32_t* live, const DevScalars* sc) {
    constexpr bool kHoldMasses = P <= 4;  // registers
    const int lane = threadIdx.x & 31;
    if (live) R = sc->R_new < R ? sc->R_new : R;  // new slots of a variable population
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    const int q4 = Np / 4;          // float4s per component
    const int nq = 6 * q4;          // float4s per replica
    const float4* m4 = reinterpret_cast<const float4*>(masses);
    // per float4 of this lane: its coordinate (0..2 positions, 3.. velocities,
    // 6 beyond the record), its index among the masses, the masses
    int comp[P], mi[P];
    float4 mh[kHoldMasses ? P : 1];
#pragma unroll
    for (int r = 0; r < P; ++r) {
        const int q = lane + 32 * r;
        comp[r] = q < nq ? q / q4 : 6;
        mi[r] = q < nq ? q - comp[r] * q4 : 0;
        if (kHoldMasses) mh[r] = m4[mi[r]];
    }
    for (long long k = warp; k < R; k += nwarps) {
        const long long j = anc[k];
        const float4* src = reinterpret_cast<const float4*>(st_in + (size_t)j * 6 * Np);
        float4* dst = reinterpret_cast<float4*>(st_out + (size_t)k * 6 * Np);
        float4 v[P];
#pragma unroll
        for (int r = 0; r < P; ++r)
            if (comp[r] < 6) v[r] = __ldcs(src + lane + 32 * r);  // read once: streaming load
        double Ej = 0.0;
        int32_t fj = 0;
        if (lane == 0) {
            Ej = E_in[j];
            fj = fam_in[j];
        }
        float sx = 0.f, sy = 0.f, sz = 0.f;
#pragma unroll
        for (int r = 0; r < P; ++r) {
            if (32 * r >= 3 * q4) break;  // no positions in this column or later ones
            if (comp[r] < 3) {
                const float4 m = kHoldMasses ? mh[r] : m4[mi[r]];
                const float s = dot4(m, v[r]);
                sx += comp[r] == 0 ? s : 0.f;
                sy += comp[r] == 1 ? s : 0.f;
                sz += comp[r] == 2 ? s : 0.f;
            }
        }
        float cx, cy, cz;
        {  // butterfly sums of three values, halves and quarters sharing steps
            const float a = sx + __shfl_xor_sync(0xffffffffu, sx, 16), b = sy + __shfl_xor_sync(0xffffffffu, sy, 16),
                        c = sz + __shfl_xor_sync(0xffffffffu, sz, 16);
            float ab = lane < 16 ? a : b, t = c;
            ab += __shfl_xor_sync(0xffffffffu, ab, 8);
            t += __shfl_xor_sync(0xffffffffu, t, 8);
            float u = (lane & 8) ? t : ab;  // lanes 0..7 x, 16..23 y, 8..15 and 24..31 z
            u += __shfl_xor_sync(0xffffffffu, u, 4);
            u += __shfl_xor_sync(0xffffffffu, u, 2);
            u += __shfl_xor_sync(0xffffffffu, u, 1);
            cx = __shfl_sync(0xffffffffu, u, 0);
            cy = __shfl_sync(0xffffffffu, u, 16);
            cz = __shfl_sync(0xffffffffu, u, 8);
        }
        float mv2 = 0.f, ux = 0.f, uy = 0.f, uz = 0.f, u2 = 0.f;
#pragma unroll
        for (int r = 0; r < P; ++r) {
            float4 w = v[r];
            if (32 * r < 3 * q4 && comp[r] < 3) {
                const float c = (comp[r] == 0) ? cx : (comp[r] == 1) ? cy : cz;  // sum of m x
                w.x = __fmaf_rn(-c, inv_mtot, w.x);
                w.y = __fmaf_rn(-c, inv_mtot, w.y);
                w.z = __fmaf_rn(-c, inv_mtot, w.z);
                w.w = __fmaf_rn(-c, inv_mtot, w.w);
                float4 z = w;  // padding atoms (>= N) are kept out of the sums
                if (Np != N) {
                    const int left = N - 4 * mi[r];
                    z.y = left > 1 ? z.y : 0.f;
                    z.z = left > 2 ? z.z : 0.f;
                    z.w = left > 3 ? z.w : 0.f;
                }
                const float s1 = z.x + z.y + z.z + z.w;
                u2 += dot4(z, w);
                ux += comp[r] == 0 ? s1 : 0.f;
                uy += comp[r] == 1 ? s1 : 0.f;
                uz += comp[r] == 2 ? s1 : 0.f;
            }
            if (32 * r + 31 >= 3 * q4 && comp[r] >= 3) {
                const float4 m = kHoldMasses ? mh[r] : m4[mi[r]];  // 0 for padding atoms
                w.x *= vscale; w.y *= vscale; w.z *= vscale; w.w *= vscale;
                if (comp[r] < 6) mv2 += mass_square(m, w);
            }
            if (comp[r] < 6) __stcs(dst + lane + 32 * r, w);  // written once: streaming store
        }
        // five butterfly sums: u2, ux, uy, uz end in lanes 0, 8, 16, 24, mv2 in lane 4
        ux += __shfl_xor_sync(0xffffffffu, ux, 16);
        uy += __shfl_xor_sync(0xffffffffu, uy, 16);
        uz += __shfl_xor_sync(0xffffffffu, uz, 16);
        u2 += __shfl_xor_sync(0xffffffffu, u2, 16);
        mv2 += __shfl_xor_sync(0xffffffffu, mv2, 16);
        float a = lane < 16 ? u2 : uy, b = lane < 16 ? ux : uz;
        a += __shfl_xor_sync(0xffffffffu, a, 8);
        b += __shfl_xor_sync(0xffffffffu, b, 8);
        mv2 += __shfl_xor_sync(0xffffffffu, mv2, 8);
        a = (lane & 8) ? b : a;  // 0..7 u2, 8..15 ux, 16..23 uy, 24..31 uz
        a += __shfl_xor_sync(0xffffffffu, a, 4);
        mv2 += __shfl_xor_sync(0xffffffffu, mv2, 4);
        a = (lane & 28) == 4 ? mv2 : a;
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        if (lane == 4) ke_out[k] = 0.5 * (double)a;
        const float mean = a / N;  // each of the four sums in its lane
        const float mx = __shfl_sync(0xffffffffu, mean, 8), my = __shfl_sync(0xffffffffu, mean, 16),
                    mz = __shfl_sync(0xffffffffu, mean, 24);
        if (lane == 0) {
            E_out[k] = Ej;
            fam_out[k] = fj;
            rg_out[k] = (double)sqrtf(fmaxf(mean - (mx * mx + my * my + mz * mz), 0.f));
        }
    }
}

// ------------------------------------------------------------------ observables

// One observation is one launch for populations of up to kObsFusedRows chunks
// of 1024 replicas: every block writes its chunk's sums per family bin and
// the block that finishes last adds the rows and forms the jackknife errors.
// Larger populations add the rows in a second launch and finish in a third.
// Everything is bound by latency, and by FP64 issue (one warp instruction in
// 16 cycles per SM), so the sums run over short segments side by side and the
// four jackknife errors in four warps.  R = 256: 15 us; R = 2^20: 40 + 4 + 11
// us.  Before, with a cleared flag array, a marking pass, one thread per bin
// walking its replicas and one thread doing the four errors in turn: 2 + 3 +
// 13 + 87 us at R = 4096 and 5 + 43 + 407 us at R = 2^20.

constexpr int kObsVals = 5;  // count, E, E_kin, R_g, R_g^2
constexpr int kObsStride = kNumBins * kObsVals;
constexpr int kObsSeg = 8;   // replicas a thread adds in a row
constexpr int kObsFusedRows = 64;
constexpr int kObsSlices = 16;

// Device state of the observations of one context (zero at the start):
// stamp[f] is the number of the last observation that saw family f, so that
// no flag array is cleared between observations.
struct ObsCtl {
    uint32_t epoch;   // observations so far
    uint32_t done;    // blocks that have finished this one
    uint32_t families;
    uint32_t pad;
};

// Per-bin partial sums of one 1024-replica chunk into out[kObsStride], and
// the families this chunk is the first to see.  The replicas are ordered by
// bin with a stable counting sort (ranks within 32-replica pieces from
// __match_any_sync, prefix counts over the pieces), each bin's segment is cut
// into pieces of at most kObsSeg, one thread each, and one thread per bin
// adds its pieces in order.  A family id is counted by the first atomic
// exchange that finds an older stamp; a run of equal ids (copies stand side
// by side) needs one exchange.
__device__ __forceinline__ void obs_chunk(const int32_t* fam, const double* E, const double* ke, const double* rg,
                                          uint32_t* stamp, uint32_t epoch, ObsCtl* ctl, long long base, long long n,
                                          long long R, double* out) {
    constexpr int kPieces = kScanBlock / 32;
    constexpr int kPerWarp = kPieces / (kScanThreads / 32);
    constexpr int kSegs = kNumBins + kScanBlock / kObsSeg;  // at most
    static_assert(kPieces % (kScanThreads / 32) == 0, "pieces per warp");
    static_assert(kSegs <= kScanThreads, "one thread per segment");
    __shared__ int32_t sf[kScanBlock];
    __shared__ double se[kScanBlock], sk[kScanBlock], sr[kScanBlock];
    __shared__ int32_t pcount[kPieces][kNumBins];  // per piece and bin: count, then prefix
    __shared__ int32_t bstart[kNumBins + 1], sstart[kNumBins + 1];
    __shared__ int16_t order[kScanBlock];          // chunk entries sorted by bin (stable)
    __shared__ double seg[4][kSegs];
    int fresh = 0;
    for (int t = threadIdx.x; t < kScanBlock; t += kScanThreads) {
        const long long k = base + t;
        int32_t bin = -1;
        if (k < n) {
            const int32_t f = fam[k];
            bin = f & (kNumBins - 1);
            se[t] = E[k];
            sk[t] = ke[k];
            sr[t] = rg[k];
            if (f >= 0 && f < R && (k == 0 || fam[k - 1] != f) && atomicExch(&stamp[f], epoch) != epoch) ++fresh;
        }
        sf[t] = bin;
    }
    for (int i = threadIdx.x; i < kPieces * kNumBins; i += kScanThreads) (&pcount[0][0])[i] = 0;
    fresh = __reduce_add_sync(0xffffffffu, fresh);
    if ((threadIdx.x & 31) == 0 && fresh) atomicAdd(&ctl->families, (uint32_t)fresh);
    __syncthreads();
    // ranks within each piece, and the pieces' counts per bin
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int rank[kPerWarp];
#pragma unroll
    for (int q = 0; q < kPerWarp; ++q) {
        const int c = w + q * (kScanThreads / 32);
        const int bin = sf[32 * c + lane];
        const unsigned peers = __match_any_sync(0xffffffffu, bin);
        rank[q] = __popc(peers & ((1u << lane) - 1u));
        if (bin >= 0 && rank[q] == 0) pcount[c][bin] = __popc(peers);
    }
    __syncthreads();
    if (threadIdx.x < kNumBins) {  // prefix over the pieces, per bin
        int s = 0;
#pragma unroll 8
        for (int c = 0; c < kPieces; ++c) {
            const int x = pcount[c][threadIdx.x];
            pcount[c][threadIdx.x] = s;
            s += x;
        }
        bstart[threadIdx.x + 1] = s;  // the bin's size, turned into starts below
    }
    __syncthreads();
    if (w == 0) {  // starts of the bins and of their segments: two bins per lane
        const int c0 = bstart[2 * lane + 1], c1 = bstart[2 * lane + 2];
        const int s0 = (c0 + kObsSeg - 1) / kObsSeg, s1 = (c1 + kObsSeg - 1) / kObsSeg;
        const int bi = warp_incl_scan(c0 + c1), si = warp_incl_scan(s0 + s1);
        __syncwarp();
        bstart[2 * lane + 1] = bi - c1;
        bstart[2 * lane + 2] = bi;
        sstart[2 * lane + 1] = si - s1;
        sstart[2 * lane + 2] = si;
        if (lane == 0) bstart[0] = sstart[0] = 0;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPerWarp; ++q) {
        const int c = w + q * (kScanThreads / 32);
        const int t = 32 * c + lane;
        const int bin = sf[t];
        if (bin >= 0) order[bstart[bin] + pcount[c][bin] + rank[q]] = (int16_t)t;
    }
    __syncthreads();
    if ((int)threadIdx.x < sstart[kNumBins]) {
        int b = 0;  // the bin of this segment
#pragma unroll
        for (int h = kNumBins / 2; h > 0; h >>= 1)
            if (sstart[b + h] <= (int)threadIdx.x) b += h;
        const int i0 = bstart[b] + ((int)threadIdx.x - sstart[b]) * kObsSeg, i1 = min(i0 + kObsSeg, bstart[b + 1]);
        double e = 0, k2 = 0, r = 0, r2 = 0;
        for (int i = i0; i < i1; ++i) {
            const int t = order[i];
            e += se[t];
            k2 += sk[t];
            r += sr[t];
            r2 += sr[t] * sr[t];
        }
        seg[0][threadIdx.x] = e;
        seg[1][threadIdx.x] = k2;
        seg[2][threadIdx.x] = r;
        seg[3][threadIdx.x] = r2;
    }
    __syncthreads();
    {  // one thread per bin and value
        const int b = threadIdx.x & (kNumBins - 1), v = threadIdx.x / kNumBins;
        double s = 0;
        for (int i = sstart[b]; i < sstart[b + 1]; ++i) s += seg[v][i];
        out[b * kObsVals + 1 + v] = s;
        if (v == 0) out[b * kObsVals] = (double)(bstart[b + 1] - bstart[b]);
    }
}
static_assert(kScanThreads == 4 * kNumBins, "one thread per bin and value");

// Averages and jackknife standard errors over the family bins from `rows`
// rows of per-bin sums (whole block, kScanThreads threads).  Warp v takes
// value v + 1, two bins per lane; bins that are empty or hold the whole
// population are left out.
__device__ __forceinline__ void obs_finish(const double* part, int rows, long long R, int N, double T,
                                           const DevScalars* s, ObsCtl* ctl, pamd_obs* dst) {
    __shared__ double bins[kObsStride];
    __shared__ double mean[4], err[4];
    for (int c = threadIdx.x; c < kObsStride; c += kScanThreads) {
        double acc = 0.0;
#pragma unroll 8
        for (int r = 0; r < rows; ++r) acc += __ldcg(part + (size_t)r * kObsStride + c);
        bins[c] = acc;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, v = threadIdx.x >> 5;
    const double Rd = (double)R;
    if (v < 4) {
        const double x0 = bins[lane * kObsVals + 1 + v], x1 = bins[(lane + 32) * kObsVals + 1 + v];
        const double n0 = bins[lane * kObsVals], n1 = bins[(lane + 32) * kObsVals];
        const double tot = warp_sum_d(x0 + x1);
        const bool k0 = n0 != 0.0 && n0 != Rd, k1 = n1 != 0.0 && n1 != Rd;
        // leave-one-bin-out means
        const double j0 = k0 ? (tot - x0) / (Rd - n0) : 0.0, j1 = k1 ? (tot - x1) / (Rd - n1) : 0.0;
        const int nb = __popc(__ballot_sync(0xffffffffu, k0)) + __popc(__ballot_sync(0xffffffffu, k1));
        const double jm = warp_sum_d(j0 + j1) / (double)(nb > 0 ? nb : 1);
        const double d0 = k0 ? j0 - jm : 0.0, d1 = k1 ? j1 - jm : 0.0;
        const double ss = warp_sum_d(d0 * d0 + d1 * d1);
        if (lane == 0) {
            mean[v] = tot / Rd;
            err[v] = nb < 2 ? 0.0 : sqrt((double)(nb - 1) / nb * ss);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        pamd_obs o;
        o.T = T;
        o.lnQ = s->lnQ;
        o.sum_lnQ = s->sum_lnQ;
        o.e_pot = mean[0];
        o.e_pot_se = err[0];
        o.e_kin = mean[1];
        o.e_kin_se = err[1];
        o.t_meas = 2.0 * o.e_kin / (3.0 * N * kBoltzmann);
        o.rg = mean[2];
        o.rg_se = err[2];
        o.rg2 = mean[3];
        o.rg2_se = err[3];
        o.n_families = (int64_t)__ldcg(&ctl->families);
        o.max_copies = s->max_copies;
        o.pad_ = s->status;
        o.R_live = R;
        *dst = o;
        // ready for the next observation
        ctl->epoch += 1;
        ctl->families = 0;
        ctl->done = 0;
    }
}

struct ObsArgs {
    const int32_t* fam;
    const double *E, *ke, *rg;
    uint32_t* stamp;
    ObsCtl* ctl;
    double* part;          // [blocks][kObsStride], then [kObsSlices][kObsStride]
    long long R;
    const uint32_t* live;
    int N, nblk;
    double T;
    const DevScalars* s;
    pamd_obs* dst;
};

template <bool FUSED>
__global__ void __launch_bounds__(kScanThreads) obs_kernel(const ObsArgs g) {
    __shared__ int last;
    const long long n = live_size(g.live, g.R);
    obs_chunk(g.fam, g.E, g.ke, g.rg, g.stamp, g.ctl->epoch + 1, g.ctl, (long long)blockIdx.x * kScanBlock, n, g.R,
              g.part + (size_t)blockIdx.x * kObsStride);
    if (!FUSED) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&g.ctl->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    obs_finish(g.part, g.nblk, n, g.N, g.T, g.s, g.ctl, g.dst);
}

// Rows of slice blockIdx.y added: 32 columns per block, eight row groups.
__global__ void __launch_bounds__(kScanThreads) obs_rows_kernel(const double* part, int nblk, double* out) {
    __shared__ double sh[kScanThreads];
    const int c = blockIdx.x * 32 + (threadIdx.x & 31), q = threadIdx.x >> 5;
    const int per = (nblk + kObsSlices - 1) / kObsSlices;
    const int r0 = blockIdx.y * per, r1 = min(r0 + per, nblk);
    double s = 0.0;
#pragma unroll 4
    for (int r = r0 + q; r < r1; r += kScanThreads / 32) s += part[(size_t)r * kObsStride + c];
    sh[threadIdx.x] = s;
    __syncthreads();
    if (q) return;
    for (int i = 1; i < kScanThreads / 32; ++i) s += sh[threadIdx.x + 32 * i];
    out[(size_t)blockIdx.y * kObsStride + c] = s;
}
static_assert(kObsStride % 32 == 0, "whole column groups");

__global__ void __launch_bounds__(kScanThreads) obs_final_kernel(const ObsArgs g) {
    obs_finish(g.part + (size_t)g.nblk * kObsStride, kObsSlices, live_size(g.live, g.R), g.N, g.T, g.s, g.ctl, g.dst);
}

// ------------------------------------------------------------------ host side

static int grid_for(long long n, int threads, int cap) {
    long long b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > cap) b = cap;
    return (int)b;
}

cudaError_t launch_init(pamd_ctx* c, double T0) {
    if (c->precision == PAMD_PREC_FP64) {
        const cudaError_t e = launch_init_f64(c, T0);
        if (e != cudaSuccess) return e;
        reset_scalars_kernel<<<1, 1, 0, c->stream>>>(c->b.scal);
        c->launches += 1;
        return cudaGetLastError();
    }
    const long long total = c->R * c->Np;
    init_kernel<<<grid_for(total, 256, c->num_sms * 16), 256, 0, c->stream>>>(
        c->b.state, c->b.E, c->b.fam, c->b.x0, c->b.masses, c->R, c->N, c->Np,
        (float)(kBoltzmann * T0), c->seed, kPurposeInit | ((uint32_t)c->mol << 8));
    reset_scalars_kernel<<<1, 1, 0, c->stream>>>(c->b.scal);
    c->launches += 2;
    if (c->variable) {  // the population starts at its target size
        set_live_kernel<<<1, 1, 0, c->stream>>>(c->b.counters, (uint32_t)c->R_target);
        c->launches += 1;
    }
    return cudaGetLastError();
}

cudaError_t launch_set_counters(pamd_ctx* c, uint32_t step, uint32_t ridx) {
    set_counters_kernel<<<1, 1, 0, c->stream>>>(c->b.counters, step, ridx);
    c->launches += 1;
    return cudaGetLastError();
}

static ExpCoef exp_coefficients() {
    ExpCoef cf;
    double f = 1.0;
    for (int n = 0; n < 14; ++n) {
        if (n > 0) f *= (double)n;
        cf.c[n] = 1.0 / f;
    }
    return cf;
}

cudaError_t launch_resample(pamd_ctx* c, double T_prev, double T_next, int do_resample,
                            const uint32_t* dev_counters, uint32_t resample_offset) {
    // R: slots of the population buffers (the capacity of a variable
    // population, whose live size the kernels read from counter word 2)
    const long long R = c->R;
    const uint32_t* live = c->variable ? c->b.counters + 2 : nullptr;
    const int nblk = c->n_blk;
    cudaStream_t s = c->stream;
    const double dbeta = 1.0 / (kBoltzmann * T_next) - 1.0 / (kBoltzmann * T_prev);
    int bits = 0;
    while ((1LL << bits) < R) ++bits;
    const double two_s = ldexp(1.0, 63 - bits);
    static const ExpCoef cf = exp_coefficients();

    // energies of the current population (the ping-pong buffers alternate)
    const double* Ecur = c->cur_is_alt ? c->b.E_alt : c->b.E;
    const int rule = !do_resample ? 0 : (c->resample_rule == PAMD_RESAMPLE_SYSTEMATIC ? 2 : 1);
    const uint32_t purpose = kPurposeResample | ((uint32_t)c->mol << 8);
    // ancestors of the new slots (into the weight buffer)
    int32_t* anc = reinterpret_cast<int32_t*>(c->b.W);
    if (!c->variable && R <= kClusterMaxR) {
        const ClusterArgs g{Ecur, R, dbeta, two_s, c->b.scal, cf, c->seed, dev_counters, resample_offset, purpose, rule,
                            c->b.cnt, c->b.cnt_incl, anc};
        const cudaError_t e = launch_resample_cluster(g, s);
        if (e != cudaSuccess) return e;
        c->launches += 1;
    } else {
        amax_kernel<<<nblk, kScanThreads, 0, s>>>(Ecur, R, dbeta, c->b.blk_f64, live);
        max_top_kernel<<<1, 1024, 0, s>>>(c->b.blk_f64, nblk, c->b.scal);
        weights_kernel<<<nblk, kScanThreads, 0, s>>>(Ecur, R, dbeta, two_s, c->b.scal, cf, c->b.W,
                                                     c->b.blk_u64, c->b.blk_f64, live);
        weights_top_kernel<<<1, kScanThreads, 0, s>>>(c->b.blk_u64, c->b.blk_f64, nblk, R, c->b.scal, live);
        scan_local_u64_kernel<<<nblk, kScanThreads, 0, s>>>(c->b.W, R, c->b.blk_u64, c->b.C, live);
        const cudaError_t e = cudaMemsetAsync(c->b.cnt, 0, sizeof(int32_t) * (size_t)R, s);
        if (e != cudaSuccess) return e;
        if (c->variable && do_resample)
            varsize_counts_kernel<<<grid_for(R, 256, c->num_sms * 16), 256, 0, s>>>(
                c->b.W, R, c->b.scal, c->R_target, c->seed, dev_counters, resample_offset, purpose,
                c->resample_rule == PAMD_RESAMPLE_NEAREST ? 3 : 4, cf, c->b.cnt, live);
        else
            counts_kernel<<<grid_for(R, 256, c->num_sms * 16), 256, 0, s>>>(
                c->b.C, R, c->b.scal, c->seed, dev_counters, resample_offset, purpose, rule, c->b.cnt, live);
        cnt_block_kernel<<<nblk, kScanThreads, 0, s>>>(c->b.cnt, R, c->b.blk_i32, c->b.blk_i32 + nblk, live);
        cnt_top_kernel<<<1, kScanThreads, 0, s>>>(c->b.blk_i32, c->b.blk_i32 + nblk, nblk, c->b.scal);
        cnt_local_kernel<<<nblk, kScanThreads, 0, s>>>(c->b.cnt, R, c->b.blk_i32, c->b.cnt_incl, live);
        c->launches += 9;
        if (c->precision != PAMD_PREC_FP64) {
            ancestor_kernel<<<grid_for(R, 256, c->num_sms * 16), 256, 0, s>>>(c->b.cnt_incl, R, anc, live, c->b.scal);
            c->launches += 1;
        }
    }
    double mt = 0.0;
    for (double m : c->host_mass) mt += m;
    const float* src = c->cur_is_alt ? c->b.state_alt : c->b.state;
    float* dst = c->cur_is_alt ? c->b.state : c->b.state_alt;
    const double* Ein = c->cur_is_alt ? c->b.E_alt : c->b.E;
    double* Eout = c->cur_is_alt ? c->b.E : c->b.E_alt;
    const int32_t* fin = c->cur_is_alt ? c->b.fam_alt : c->b.fam;
    int32_t* fout = c->cur_is_alt ? c->b.fam : c->b.fam_alt;
    if (c->precision == PAMD_PREC_FP64) {
        const cudaError_t e = launch_gather_f64(
            c, reinterpret_cast<const double*>(src), reinterpret_cast<double*>(dst), Ein, Eout, fin,
            fout, sqrt(T_next / T_prev));
        return e != cudaSuccess ? e : cudaGetLastError();
    }
    const float vs = (float)sqrt(T_next / T_prev), imt = (float)(1.0 / mt);
    const int gridg = grid_for(R * 32, 256, c->num_sms * 64);
    switch ((6 * (c->Np / 4) + 31) / 32) {
#define PAMD_GATHER_CASE(P)                                                                     \
    case P:                                                                                     \
        gather_kernel<P><<<gridg, 256, 0, s>>>(src, dst, Ein, Eout, fin, fout, c->b.ke, c->b.rg, \
                                               anc, c->b.masses, R, c->N, c->Np, vs, imt, live, \
                                               c->b.scal);                                      \
        break;
        PAMD_GATHER_CASE(1) PAMD_GATHER_CASE(2) PAMD_GATHER_CASE(3) PAMD_GATHER_CASE(4)
        PAMD_GATHER_CASE(5) PAMD_GATHER_CASE(6) PAMD_GATHER_CASE(7) PAMD_GATHER_CASE(8)
        PAMD_GATHER_CASE(9) PAMD_GATHER_CASE(10) PAMD_GATHER_CASE(11) PAMD_GATHER_CASE(12)
#undef PAMD_GATHER_CASE
        default: return cudaErrorInvalidValue;
    }
    c->launches += 1;
    if (c->variable) {
        commit_size_kernel<<<1, 1, 0, s>>>(c->b.scal, c->b.counters, R);
        c->launches += 1;
    }
    return cudaGetLastError();
}

size_t obs_part_bytes(int nblk) { return sizeof(double) * kObsStride * ((size_t)nblk + kObsSlices); }
size_t obs_ctl_bytes() { return sizeof(ObsCtl); }

cudaError_t launch_observe(pamd_ctx* c, double T, pamd_obs* dst) {
    cudaStream_t s = c->stream;
    ObsArgs g{};
    g.fam = c->cur_is_alt ? c->b.fam_alt : c->b.fam;
    g.E = c->cur_is_alt ? c->b.E_alt : c->b.E;
    g.ke = c->b.ke;
    g.rg = c->b.rg;
    g.stamp = c->b.fam_stamp;
    g.ctl = reinterpret_cast<ObsCtl*>(c->b.obs_ctl);
    g.part = c->b.obs_part;
    g.R = c->R;
    g.live = c->variable ? c->b.counters + 2 : nullptr;
    g.N = c->N;
    g.nblk = c->n_blk;
    g.T = T;
    g.s = c->b.scal;
    g.dst = dst;
    if (g.nblk <= kObsFusedRows) {
        obs_kernel<true><<<g.nblk, kScanThreads, 0, s>>>(g);
        c->launches += 1;
    } else {
        obs_kernel<false><<<g.nblk, kScanThreads, 0, s>>>(g);
        obs_rows_kernel<<<dim3(kObsStride / 32, kObsSlices), kScanThreads, 0, s>>>(
            g.part, g.nblk, g.part + (size_t)g.nblk * kObsStride);
        obs_final_kernel<<<1, kScanThreads, 0, s>>>(g);
        c->launches += 3;
    }
    return cudaGetLastError();
}

}  // namespace pamd
