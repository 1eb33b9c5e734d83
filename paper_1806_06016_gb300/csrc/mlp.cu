// mlp.cu -- the MLP energy surrogate: parameters, features, forces, the
// force-matching loss and its gradient, Adam, and the C-ABI of pamd_mlp.h.
//
// Dense layers are BF16 tensor-core GEMMs (mlp_gemm.cu) whose epilogues apply
// the bias, the SiLU and its derivative and write the BF16 operands of the
// next product; the weight gradients contract over the samples of the same
// row-major operands.
// Everything between the products (features, the pair Jacobian and its
// transpose, second-derivative terms, column sums) is FP32 here; energies and
// loss sums are FP64.
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "mlp_device.cuh"
#include "pamd_device.cuh"

namespace pamd {

constexpr uint32_t kPurposeMlpInit = 3u;

namespace {

int mfail(int code, const std::string& msg) {
    set_last_error(msg);
    return code;
}

int mcuda(pamd_mlp* m, cudaError_t e, const char* what) {
    if (m) m->broken = true;
    return mfail(PAMD_ECUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

#define MLP_CU(m, call)                                       \
    do {                                                      \
        const cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return mcuda((m), e_, #call);  \
    } while (0)

int grid_for(long long n, int threads, int cap = 152 * 16) {
    long long g = (n + threads - 1) / threads;
    if (g > cap) g = cap;
    return (int)(g < 1 ? 1 : g);
}

__device__ __forceinline__ float sig(float z) { return 1.0f / (1.0f + __expf(-z)); }
// second derivative of silu(z) = z s(z): s (1 - s) (2 + z (1 - 2 s))
__device__ __forceinline__ float d2silu(float z) {
    const float s = sig(z);
    return s * (1.0f - s) * (2.0f + z * (1.0f - 2.0f * s));
}

// ---------------------------------------------------------------- parameters

__global__ void mlp_init_kernel(float* params, size_t oW1, size_t oW2, size_t ow3, int H, int P,
                                int Pp, unsigned long long seed) {
    const long long n1 = (long long)H * Pp, n2 = (long long)H * H, n3 = H;
    const long long n = n1 + n2 + n3;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        uint32_t region;
        long long local;
        size_t dst;
        float scale;
        bool zero = false;
        if (e < n1) {
            region = 1;
            local = e;
            zero = (int)(e % Pp) >= P;
            scale = rsqrtf((float)P);
            dst = oW1 + (size_t)local;
        } else if (e < n1 + n2) {
            region = 2;
            local = e - n1;
            scale = rsqrtf((float)H);
            dst = oW2 + (size_t)local;
        } else {
            region = 3;
            local = e - n1 - n2;
            scale = rsqrtf((float)H);
            dst = ow3 + (size_t)local;
        }
        float v = 0.0f;
        if (!zero) {
            const uint4 o = philox4x32_10(
                make_uint4((uint32_t)local, (uint32_t)(local >> 32), region, kPurposeMlpInit),
                make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
            const float u0 = ((float)(o.x >> 9) + 0.5f) * 1.1920928955078125e-07f;
            const float u1 = ((float)(o.y >> 9) + 0.5f) * 1.1920928955078125e-07f;
            v = sqrtf(-2.0f * logf(u0)) * cospif(2.0f * u1) * scale;  // Box-Muller
        }
        params[dst] = v;
    }
}

// The BF16 copies of W1 and W2 the tensor cores read: same layout, rounded.
struct WeightCopies {
    size_t oW1, nW1, oW2, nW2;  // offsets and sizes in the parameter block
    __nv_bfloat16 *W1b, *W2b;
    __device__ __forceinline__ void put(size_t e, float p) const {
        if (e - oW1 < nW1) W1b[e - oW1] = __float2bfloat16(p);
        else if (e - oW2 < nW2) W2b[e - oW2] = __float2bfloat16(p);
    }
};

__global__ void mlp_pack_kernel(const float* __restrict__ params, long long n, const WeightCopies w) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x)
        w.put((size_t)e, params[e]);
}

// Adam and, from the new value in hand, the BF16 copies: HBM/L2-bound, 28
// bytes read and written per parameter.  75 atoms, H = 512 (1.7 M
// parameters): 11.9 us; an update and a pass that also wrote transposed
// copies in 2-byte stores took 11.5 + 16.7 us.
__global__ void mlp_adam_kernel(float* p, const float* __restrict__ g, float* m, float* v,
                                long long n, float lr, float b1, float b2, float eps, float bc1,
                                float bc2, const WeightCopies w) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n;
         e += (long long)gridDim.x * blockDim.x) {
        const float gi = g[e];
        const float mi = b1 * m[e] + (1.0f - b1) * gi;
        const float vi = b2 * v[e] + (1.0f - b2) * gi * gi;
        m[e] = mi;
        v[e] = vi;
        const float pn = p[e] - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
        p[e] = pn;
        w.put((size_t)e, pn);
    }
}

// ------------------------------------------------------------- normalisation

// Mean and sum of squared deviations of every feature g_p = 1 / r over n
// configurations (and of the energies), merged from slices of the data.
//
// GB300's FP64 units do a 64th of the FP32 rate, and a reciprocal square root
// per sample and pair is all the work there is.  So a sample's g is formed in
// pairs of FP32 numbers (TwoSum: Knuth 1969; exact products by fma):
// coordinate differences are exact, r^2 carries its rounding errors, and one
// Newton step on the hardware reciprocal square root leaves g = y0 + corr
// within 2^-44 of its value.  Deviations from the slice's first sample
// (exactly zero for an equal one, so that a constant feature has no spurious
// deviation) are pairs as well; they and their squares are added in
// compensated FP32 over kStatHold samples or a tile, then in FP64.  Slices become
// (mean, M2) in FP64 and are merged by Chan, Golub & LeVeque's (1979) formula.
// A spread below 2^-16 of the mean, of which 2^-44 of g would be 2^-28 or more,
// and a distance outside [1e-10, 1e10] nm (coincident atoms, non-finite input;
// its pair is marked with a NaN) are left to the merge kernel, which does that
// pair in plain FP64.  mu and sd are then the FP32 roundings of values within
// 2^-40 and 2^-28 of the 64-bit ones (a slice whose first sample lies far from
// the rest loses log2 of its length of these bits).
//
// One thread per pair, the positions of a tile of configurations in shared
// memory as float4 (consecutive pairs read consecutive atoms: no bank
// conflicts), the data cut into as many slices as fill the chip.
// 65536 configurations of 75 atoms: 624 + 31 us, bound by instruction issue
// (about 100 per sample and pair, 83 % of the slots; 661 us with a subnormal-safe
// reciprocal square root and a TwoSum for the squares).  Deviations rounded to
// FP32 took 611 us and lost up to half the last bit of sd; one thread per pair
// looping twice over all configurations in FP64 (22 blocks) took 151.0 ms.
// Against 64-bit torch, 27 sets of 9..75 atoms x 100..65536 samples: mu and sd
// are as far from it as that FP64 loop's, to five digits.
constexpr int kStatThreads = 256;
constexpr int kStatTileBytes = 24 * 1024;
constexpr int kStatHold = 64;  // samples added in FP32 pairs before they join the FP64 sums
// block columns (the last one for the energies), and slices that give every SM six blocks
int stat_columns(int P) { return (P + kStatThreads - 1) / kStatThreads + 1; }
int stat_slices(int P, int sms) { return (6 * sms + stat_columns(P) - 1) / stat_columns(P); }

// a + b = s + e exactly
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
    const float s = __fadd_rn(a, b);
    const float bp = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
    return s;
}
// (s, e) with s^2 and its error including 2 s e
__device__ __forceinline__ float square_err(float s, float e, float& err) {
    const float p = __fmul_rn(s, s);
    err = __fmaf_rn(__fadd_rn(s, s), e, __fmaf_rn(s, s, -p));
    return p;
}
// (mean, M2) of na + nb values from those of the parts
__device__ __forceinline__ void merge_moments(double& na, double& ma, double& qa, double nb, double mb, double qb) {
    if (nb == 0.0) return;
    if (na == 0.0) {
        na = nb; ma = mb; qa = qb;
        return;
    }
    const double n = na + nb, d = mb - ma;
    ma += d * (nb / n);
    qa += qb + d * d * (na * (nb / n));
    na = n;
}

// part[blockIdx.y][p]: (mean, M2) of slice blockIdx.y; the last block column
// does the energies, entry P.
__global__ void __launch_bounds__(kStatThreads) mlp_moments_kernel(const float* __restrict__ x,
                                                                   const double* __restrict__ E, long long n,
                                                                   long long per, int N, int P, int tile,
                                                                   const ushort2* __restrict__ pairs,
                                                                   double2* __restrict__ part) {
    extern __shared__ float4 sx[];
    __shared__ double red[32];
    const long long m0 = blockIdx.y * per, m1 = m0 + per < n ? m0 + per : n;
    double2* out = part + (size_t)blockIdx.y * (P + 1);
    if (blockIdx.x == gridDim.x - 1) {
        double s = 0.0;
        for (long long m = m0 + threadIdx.x; m < m1; m += kStatThreads) s += E[m];
        const double mean = block_sum(s, red) / (double)(m1 - m0);
        double q = 0.0;
        for (long long m = m0 + threadIdx.x; m < m1; m += kStatThreads) {
            const double d = E[m] - mean;
            q += d * d;
        }
        q = block_sum(q, red);
        if (threadIdx.x == 0) out[P] = make_double2(mean, q);
        return;
    }
    const int p = blockIdx.x * kStatThreads + threadIdx.x;
    const ushort2 ij = pairs[p < P ? p : 0];
    float g0 = 0.0f, c0 = 0.0f;
    double S = 0.0, Q = 0.0;  // of the deviations from g0 + c0
    float s = 0.0f, sl = 0.0f, q = 0.0f, ql = 0.0f;
    int held = 0;  // samples in the FP32 sums
    float h_min = 1.0f, h_max = 1.0f;  // squared distances (a NaN reaches the sums)
    // g = y + corr of sample c of the tile
    auto feature = [&](int c, float& y, float& corr) {
        const float4 a = sx[c * N + ij.x], b = sx[c * N + ij.y];
        float ex, ey, ez, l1, l2;
        const float dx = two_sum(a.x, -b.x, ex), dy = two_sum(a.y, -b.y, ey), dz = two_sum(a.z, -b.z, ez);
        const float px = __fmul_rn(dx, dx), py = __fmul_rn(dy, dy), pz = __fmul_rn(dz, dz);
        const float h = two_sum(two_sum(px, py, l1), pz, l2);
        // the squares' errors and the cross terms 2 d e
        const float qe = __fadd_rn(__fmaf_rn(dx, dx, -px), __fadd_rn(__fmaf_rn(dy, dy, -py), __fmaf_rn(dz, dz, -pz)));
        const float qc = __fmaf_rn(dx, ex, __fmaf_rn(dy, ey, __fmul_rn(dz, ez)));
        const float lo = __fadd_rn(__fadd_rn(l1, l2), __fmaf_rn(2.0f, qc, qe));
        h_min = fminf(h_min, h);
        h_max = fmaxf(h_max, h);
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(h));  // no subnormal h comes into the sums
        // e = 1 - r^2 y^2
        const float u = __fmul_rn(h, y), ue = __fmaf_rn(h, y, -u);
        float e = __fmaf_rn(-u, y, 1.0f);
        e = __fmaf_rn(-ue, y, e);
        e = __fmaf_rn(-__fmul_rn(lo, y), y, e);
        corr = __fmul_rn(__fmul_rn(y, e), __fmaf_rn(0.375f, e, 0.5f));
    };
    for (long long t0 = m0; t0 < m1; t0 += tile) {
        const int nt = (int)(m1 - t0 < tile ? m1 - t0 : tile);
        __syncthreads();
        const float* src = x + (size_t)t0 * 3 * N;
        for (int a = threadIdx.x; a < nt * N; a += kStatThreads)
            sx[a] = make_float4(src[3 * a], src[3 * a + 1], src[3 * a + 2], 0.0f);
        __syncthreads();
        if (t0 == m0) feature(0, g0, c0);
#pragma unroll 4
        for (int c = 0; c < nt; ++c) {
            float y, corr, ey0, dl, err;
            feature(c, y, corr);
            const float dy0 = two_sum(y, -g0, ey0);
            const float dc = __fadd_rn(__fsub_rn(corr, c0), ey0);
            const float d = __fadd_rn(dy0, dc);
            dl = __fsub_rn(dc, __fsub_rn(d, dy0));  // dy0 is 0 or at least an ulp of g, dc a few: lost are 2^-22 of these
            s = two_sum(s, d, err);
            sl = __fadd_rn(sl, __fadd_rn(err, dl));
            float e2;
            const float d2 = square_err(d, dl, e2);
            const float big = fmaxf(q, d2), small = fminf(q, d2);  // neither is negative
            q = __fadd_rn(big, small);
            ql = __fadd_rn(ql, __fadd_rn(__fsub_rn(small, __fsub_rn(q, big)), e2));
        }
        held += nt;
        if (held >= kStatHold || t0 + tile >= m1) {
            S += (double)s + (double)sl;
            Q += (double)q + (double)ql;
            s = sl = q = ql = 0.0f;
            held = 0;
        }
    }
    if (p < P) {
        const double cnt = (double)(m1 - m0);
        const double m2 = Q - S * (S / cnt);
        const bool bad = !(h_min > 1e-20f && h_max < 1e20f);
        out[p] = bad ? make_double2(NAN, NAN) : make_double2(((double)g0 + (double)c0) + S / cnt, m2 > 0.0 ? m2 : 0.0);
    }
}

// One warp per feature merges the slices in a fixed order; warp P the
// energies (out[0] mean, out[1] standard deviation).
__global__ void __launch_bounds__(128) mlp_moments_merge_kernel(const float* __restrict__ x, long long n,
                                                                long long per, int slices, int N, int P,
                                                                const ushort2* __restrict__ pairs,
                                                                const double2* __restrict__ part, float* mu,
                                                                float* sd, float* inv_sd, double* out) {
    const int p = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (p > P) return;
    double cn = 0.0, mean = 0.0, m2 = 0.0;
    for (int y = lane; y < slices; y += 32) {
        const long long m0 = y * per, m1 = m0 + per < n ? m0 + per : n;
        const double2 v = part[(size_t)y * (P + 1) + p];
        merge_moments(cn, mean, m2, (double)(m1 - m0), v.x, v.y);
    }
    for (int o = 1; o < 32; o <<= 1) {
        const double bn = __shfl_down_sync(0xffffffffu, cn, o), bm = __shfl_down_sync(0xffffffffu, mean, o),
                     bq = __shfl_down_sync(0xffffffffu, m2, o);
        merge_moments(cn, mean, m2, bn, bm, bq);
    }
    mean = __shfl_sync(0xffffffffu, mean, 0);
    m2 = __shfl_sync(0xffffffffu, m2, 0);
    if (p == P) {
        if (lane == 0) {
            out[0] = mean;
            out[1] = sqrt(m2 / (double)n);
        }
        return;
    }
    // a distance out of the fast path's range, or a spread too small for its bits: this pair in FP64
    if (isnan(mean) || (m2 > 0.0 && m2 < 0x1p-32 * (double)n * mean * mean)) {
        const ushort2 ij = pairs[p];
        auto g_of = [&](long long m) {
            const float* c = x + m * 3 * N;
            const double dx = (double)c[3 * ij.x] - c[3 * ij.y];
            const double dy = (double)c[3 * ij.x + 1] - c[3 * ij.y + 1];
            const double dz = (double)c[3 * ij.x + 2] - c[3 * ij.y + 2];
            return 1.0 / sqrt(dx * dx + dy * dy + dz * dz);
        };
        double s = 0.0;
        for (long long m = lane; m < n; m += 32) s += g_of(m);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        mean = s / (double)n;
        double q = 0.0;
        for (long long m = lane; m < n; m += 32) {
            const double d = g_of(m) - mean;
            q += d * d;
        }
        for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
        m2 = q;
    }
    if (lane == 0) {
        double dev = sqrt(m2 / (double)n);
        if (!(dev > 0.0)) dev = 1.0;
        mu[p] = (float)mean;
        sd[p] = (float)dev;
        inv_sd[p] = (float)(1.0 / dev);
    }
}

// ------------------------------------------------------- features and forces

// Features of 2 DUOS configurations per block, one after another from one read
// of the pair's tables.  Bound by shared-memory reads (4 wavefronts a pair
// and 32 configurations' lanes) and issue; the BF16 rows it writes are 5.5 KB a
// configuration of 75 atoms.
// 65536 configurations of 75 atoms, DUOS = 4: 165 us (a block per configuration
// that read six words and three table entries a pair: 342), shared-memory
// pipe 84 % busy.
constexpr int kFeatThreads = 256;

template <int DUOS>
__global__ void __launch_bounds__(kFeatThreads) mlp_features_kernel(const FeatArgs f) {
    extern __shared__ __align__(16) unsigned char qsm[];
    const int N = f.N, n3 = 3 * N, m0 = blockIdx.x * 2 * DUOS;
    for (int t = threadIdx.x; t < 2 * DUOS * n3; t += kFeatThreads) {
        const int g = t / n3;
        int i, c;
        config_element(f.cv, t - g * n3, N, i, c);
        const int m = m0 + g < f.M ? m0 + g : f.M - 1;
        duo_pos(qsm + (g >> 1) * duo_pos_bytes(N), N).put(g & 1, i, c, config_value(f.cv, m, i, c));
    }
    __syncthreads();
#pragma unroll 2
    for (int p = threadIdx.x; p < f.Pp; p += kFeatThreads) {
        const bool in = p < f.P;
        const ushort2 ij = in ? f.pairs[p] : make_ushort2(0, 0);
        const float mu = in ? f.mu[p] : 0.0f, isd = in ? f.inv_sd[p] : 0.0f;
        __nv_bfloat16* a = f.a + (size_t)m0 * f.Pp + p;
#pragma unroll
        for (int u = 0; u < DUOS; ++u, a += 2 * f.Pp) {
            const float2 v = duo_feature(duo_pos(qsm + u * duo_pos_bytes(N), N), ij, mu, isd);
            if (m0 + 2 * u < f.M) a[0] = __float2bfloat16(in ? v.x : 0.0f);
            if (m0 + 2 * u + 1 < f.M) a[f.Pp] = __float2bfloat16(in ? v.y : 0.0f);
        }
    }
}

// Energies, and the forces of molecules with gamma_matrix(N): two
// configurations at a time per block.  One pass over the pairs fills the
// matrix c_ij, one over its rows sums c_kj (x_k - x_j) with each row split
// over several threads; meanwhile the next two de/da rows arrive by
// cp.async and their positions in registers.  Bound by shared-memory
// wavefronts (8 per 32 pairs and configuration in the first pass, 2 per 32
// elements in the second) and by the barriers between the passes.
// 65536 configurations of 75 atoms: 431 us (one configuration at a time, 75 of
// 128 threads in the second pass: 796); shared-memory pipe three quarters busy.
// byte offsets: matrix, de/da rows, positions, partial force sums [part][2][N][3]
struct DuoSmem {
    size_t ga, pos, part, total;
};
__host__ __device__ __forceinline__ DuoSmem duo_smem(int N, int Pp) {
    auto up = [](size_t b) { return (b + 15) & ~size_t(15); };
    DuoSmem L{};
    L.ga = up(duo_gamma_bytes(N));
    L.pos = L.ga + 4 * (size_t)Pp;
    L.part = L.pos + duo_pos_bytes(N);
    L.total = L.part + 24 * (size_t)N * duo_parts(N);
    return L;
}

__device__ __forceinline__ void duo_fetch_pos(const ConfigView& cv, int m0, int m1, int N, float (&v)[kDuoElems]) {
#pragma unroll
    for (int u = 0; u < kDuoElems; ++u) {
        const int t = threadIdx.x + u * blockDim.x, b = t >= 3 * N;
        int i, c;
        config_element(cv, t - 3 * N * b, N, i, c);
        v[u] = t < 6 * N ? config_value(cv, b ? m1 : m0, i, c) : 0.0f;
    }
}
__device__ __forceinline__ void duo_store_pos(const ConfigView& cv, int N, const float (&v)[kDuoElems], const DuoPos& q) {
#pragma unroll
    for (int u = 0; u < kDuoElems; ++u) {
        const int t = threadIdx.x + u * blockDim.x, b = t >= 3 * N;
        int i, c;
        config_element(cv, t - 3 * N * b, N, i, c);
        if (t < 6 * N) q.put(b, i, c, v[u]);
    }
}

__device__ __forceinline__ void energies(const ForceArgs& f) {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < f.M; m += gridDim.x * blockDim.x)
        f.E[m] = f.sigma_E * head_energy(f.part, f.nparts, m, f.b3) + f.mu_E;
}

template <int T>
__global__ void __launch_bounds__(T, duo_blocks(T)) mlp_forces_duo_kernel(const ForceArgs f) {
    extern __shared__ __align__(16) unsigned char dsm[];
    const int N = f.N, D = (f.M + 1) / 2;
    const DuoSmem L = duo_smem(N, f.Pp);
    float2* gam = reinterpret_cast<float2*>(dsm);
    const __nv_bfloat16* ga = reinterpret_cast<const __nv_bfloat16*>(dsm + L.ga);
    const DuoPos q = duo_pos(dsm + L.pos, N);
    float* part = reinterpret_cast<float*>(dsm + L.part);
    if (f.E) energies(f);
    if (!f.F) return;
    const float sE = (float)f.sigma_E;
    auto second = [&](int d) { return 2 * d + 1 < f.M ? 2 * d + 1 : 2 * d; };
    float v[kDuoElems];
    int d = blockIdx.x;
    if (d < D) {
        duo_fetch_rows(f.ga, 2 * d, second(d), f.Pp, dsm + L.ga);
        duo_fetch_pos(f.cv, 2 * d, second(d), N, v);
    }
    for (int k = threadIdx.x; k < N; k += T) gam[k * gamma_stride(N) + k] = make_float2(0.0f, 0.0f);
    for (; d < D; d += gridDim.x) {
        duo_store_pos(f.cv, N, v, q);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        duo_gamma(q, ga, f.pairs, f.inv_sd, f.P, f.Pp, N, gam);
        __syncthreads();
        const int nd = d + gridDim.x;
        if (nd < D) {
            duo_fetch_rows(f.ga, 2 * nd, second(nd), f.Pp, dsm + L.ga);
            duo_fetch_pos(f.cv, 2 * nd, second(nd), N, v);
        }
        duo_force_parts(q, gam, N, duo_parts(N), part);
        __syncthreads();
        const int n = 2 * d + 1 < f.M ? 6 * N : 3 * N;
        float* Fo = f.F + (size_t)d * 6 * N;
        for (int t = threadIdx.x; t < n; t += T) Fo[t] = sE * duo_force_sum(part, N, duo_parts(N), t);
    }
}

using ForceKernel = void (*)(const ForceArgs);
ForceKernel forces_duo_kernel(int N) {
    const int t = duo_threads(N);
    return t == 64    ? mlp_forces_duo_kernel<64>
           : t == 128 ? mlp_forces_duo_kernel<128>
           : t == 256 ? mlp_forces_duo_kernel<256>
                      : mlp_forces_duo_kernel<384>;
}

// The same for molecules past gamma_matrix(N), whose matrix does not fit.
__global__ void __launch_bounds__(kMlpThreads) mlp_forces_kernel(const ForceArgs f) {
    extern __shared__ float fsm[];
    float* xs = fsm;
    float* gam = fsm + 3 * kXs;
    if (f.E) energies(f);
    if (!f.F) return;
    const float sE = (float)f.sigma_E;
    for (int m = blockIdx.x; m < f.M; m += gridDim.x) {
        __syncthreads();
        load_config(f.cv, m, f.N, xs);
        __syncthreads();
        load_gamma(f.ga + (size_t)m * f.Pp, f.inv_sd, f.P, gam);
        __syncthreads();
        float* Fo = f.F + (size_t)m * 3 * f.N;
        for (int k = threadIdx.x; k < f.N; k += blockDim.x) {
            const float3 a = atom_force(k, xs, gam, f.N);
            Fo[3 * k] = sE * a.x;
            Fo[3 * k + 1] = sE * a.y;
            Fo[3 * k + 2] = sE * a.z;
        }
    }
}

// Force-matching loss of one sample and the direction of the tangent pass:
// f = sum_p gam_p dg_p/dx (normalised forces), u = dL/df, and
// nu_a = dL/d(de/da) = (J u) / sd with (J u)_p = (x_i - x_j).(u_i - u_j) / r^3.
// Two samples at a time like the force kernel, with a second pass over the
// pairs for J u; bound likewise by shared-memory wavefronts and barriers.
// 2048 samples of 75 atoms: 44 us (one at a time, 75 of 128 threads at the
// force rows: 70).
// Shared memory: that of the force kernel with dL/df in the place of the partial sums.
__host__ __device__ __forceinline__ size_t loss_duo_smem(int N, int Pp) {
    return ((duo_smem(N, Pp).part + 15) & ~size_t(15)) + duo_pos_bytes(N);
}

template <int T>
__global__ void __launch_bounds__(T, T == 384 ? 3 : duo_blocks(T)) mlp_loss_duo_kernel(const LossArgs A) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ double red[32];
    const int N = A.N, D = (A.M + 1) / 2;
    const DuoSmem L = duo_smem(N, A.Pp);
    float2* gam = reinterpret_cast<float2*>(dsm);
    const __nv_bfloat16* ga = reinterpret_cast<const __nv_bfloat16*>(dsm + L.ga);
    const DuoPos q = duo_pos(dsm + L.pos, N), us = duo_pos(dsm + ((L.part + 15) & ~size_t(15)), N);
    const float2* xs = reinterpret_cast<const float2*>(q.xy);  // x of atom i at 2 i, y at 2 i + 1
    const double inv_sE = 1.0 / A.sigma_E;
    const float cu = (float)(2.0 * A.lam / (3.0 * N * (double)A.M));
    auto second = [&](int d) { return 2 * d + 1 < A.M ? 2 * d + 1 : 2 * d; };
    float v[kDuoElems];
    int d = blockIdx.x;
    if (d < D) {
        duo_fetch_rows(A.ga, 2 * d, second(d), A.Pp, dsm + L.ga);
        duo_fetch_pos(A.cv, 2 * d, second(d), N, v);
    }
    for (int k = threadIdx.x; k < N; k += T) gam[k * gamma_stride(N) + k] = make_float2(0.0f, 0.0f);
    for (; d < D; d += gridDim.x) {
        const int m0 = 2 * d, m1 = second(d);
        duo_store_pos(A.cv, N, v, q);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        const long long src0 = config_index(A.cv, m0), src1 = config_index(A.cv, m1);
        duo_gamma(q, ga, A.pairs, A.inv_sd, A.P, A.Pp, N, gam);
        __syncthreads();
        const int nd = d + gridDim.x;
        if (nd < D) {
            duo_fetch_rows(A.ga, 2 * nd, second(nd), A.Pp, dsm + L.ga);
            duo_fetch_pos(A.cv, 2 * nd, second(nd), N, v);
        }
        // One thread per atom and coordinate sums a whole row in order: the BF16
        // rounding of nu_a turns a different order into flips of a bit.
        double sq0 = 0.0, sq1 = 0.0;
        if (threadIdx.x < 3 * N) {
            const int c = threadIdx.x / N, k = threadIdx.x - c * N;
            const float2* xc = c == 0 ? xs : c == 1 ? xs + 1 : q.z;
            const int sx = c < 2 ? 2 : 1;
            const float2 xk = xc[sx * k], m1 = make_float2(-1.0f, -1.0f);
            const float2* row = gam + k * gamma_stride(N);
            float2 f = make_float2(0.0f, 0.0f);
#pragma unroll 5
            for (int j = 0; j < N; ++j) f = __ffma2_rn(row[j], __ffma2_rn(m1, xc[sx * j], xk), f);
            const float d0 = f.x - (float)(A.F_ref[src0 * 3 * N + 3 * k + c] * inv_sE);
            const float d1 = f.y - (float)(A.F_ref[src1 * 3 * N + 3 * k + c] * inv_sE);
            us.put(0, k, c, cu * d0);
            us.put(1, k, c, cu * d1);
            sq0 = (double)d0 * d0;
            sq1 = (double)d1 * d1;
        }
        // the two sums of squares: half a warp each, then one thread each adds the
        // warps' (FP64 instructions cost 20 clocks of the SM: block-wide sums in
        // every warp were half of this kernel)
        const int lane = threadIdx.x & 31, nw = (3 * N + 31) / 32;
        if ((int)(threadIdx.x >> 5) < nw) {
            const bool hi = lane & 16;
            double t = (hi ? sq1 : sq0) + __shfl_xor_sync(0xffffffffu, hi ? sq0 : sq1, 16);
            for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            if ((lane & 15) == 0) red[lane + (threadIdx.x >> 5)] = t;
        }
        __syncthreads();  // also orders the writes of us before the reads below
        if ((threadIdx.x & 31) == 0 && threadIdx.x < 64 && (threadIdx.x == 0 || m1 != m0)) {
            const int m = threadIdx.x ? m1 : m0;
            double sq = 0.0;
            for (int w = 0; w < nw; ++w) sq += red[(threadIdx.x ? 16 : 0) + w];
            const double e = head_energy(A.part, A.nparts, m, A.b3);
            const double de = e - (A.E_ref[threadIdx.x ? src1 : src0] - A.mu_E) * inv_sE;
            A.ebar[m] = (float)(2.0 * de / (double)A.M);
            A.loss_part[m] = de * de + A.lam / (3.0 * N) * sq;
        }
        __nv_bfloat16* nrow = A.nu_a + (size_t)m0 * A.Pp;
#pragma unroll 2
        for (int p = threadIdx.x; p < A.Pp; p += T) {
            float2 w = make_float2(0.0f, 0.0f);
            if (p < A.P) {
                const ushort2 ij = A.pairs[p];
                const float isd = A.inv_sd[p];
                const Duo3 dx = duo_diff(q.xy[ij.x], q.z[ij.x], q.xy[ij.y], q.z[ij.y]);
                const Duo3 du = duo_diff(us.xy[ij.x], us.z[ij.x], us.xy[ij.y], us.z[ij.y]);
                const float2 r2 = __ffma2_rn(dx.z, dx.z, __ffma2_rn(dx.x, dx.x, __fmul2_rn(dx.y, dx.y)));
                const float2 ir = make_float2(rsqrtf(r2.x), rsqrtf(r2.y));
                w = __ffma2_rn(dx.z, du.z, __ffma2_rn(dx.x, du.x, __fmul2_rn(dx.y, du.y)));
                w = __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(w, ir), ir), ir), make_float2(isd, isd));
            }
            nrow[p] = __float2bfloat16(w.x);
            if (m1 != m0) nrow[A.Pp + p] = __float2bfloat16(w.y);
        }
        __syncthreads();  // q and us are read until here
    }
}

using LossKernel = void (*)(const LossArgs);
LossKernel loss_duo_kernel(int N) {
    const int t = duo_threads_wide(N);
    return t == 64 ? mlp_loss_duo_kernel<64> : t == 128 ? mlp_loss_duo_kernel<128> : mlp_loss_duo_kernel<384>;
}

// The same for molecules past gamma_matrix(N).
__global__ void __launch_bounds__(kMlpThreads) mlp_loss_kernel(const LossArgs L) {
    extern __shared__ float lsm[];
    __shared__ double red[32];
    float* xs = lsm;
    float* us = lsm + 3 * kXs;
    float* gam = lsm + 6 * kXs;
    const double inv_sE = 1.0 / L.sigma_E;
    const float cu = (float)(2.0 * L.lam / (3.0 * L.N * (double)L.M));
    for (int m = blockIdx.x; m < L.M; m += gridDim.x) {
        __syncthreads();
        load_config(L.cv, m, L.N, xs);
        __syncthreads();
        load_gamma(L.ga + (size_t)m * L.Pp, L.inv_sd, L.P, gam);
        __syncthreads();
        const long long src = config_index(L.cv, m);
        const float* Fr = L.F_ref + src * 3 * L.N;
        double sq = 0.0;
        for (int k = threadIdx.x; k < L.N; k += blockDim.x) {
            const float3 a = atom_force(k, xs, gam, L.N);
            const float dfx = a.x - (float)(Fr[3 * k] * inv_sE);
            const float dfy = a.y - (float)(Fr[3 * k + 1] * inv_sE);
            const float dfz = a.z - (float)(Fr[3 * k + 2] * inv_sE);
            us[k] = cu * dfx;
            us[kXs + k] = cu * dfy;
            us[2 * kXs + k] = cu * dfz;
            sq += (double)dfx * dfx + (double)dfy * dfy + (double)dfz * dfz;
        }
        sq = block_sum(sq, red);  // also orders the writes of us before the reads below
        __nv_bfloat16* nrow = L.nu_a + (size_t)m * L.Pp;
        for (int p = threadIdx.x; p < L.Pp; p += blockDim.x) {
            float v = 0.0f;
            if (p < L.P) {
                const ushort2 ij = L.pairs[p];
                const int i = ij.x, j = ij.y;
                const float dx = xs[i] - xs[j], dy = xs[kXs + i] - xs[kXs + j],
                            dz = xs[2 * kXs + i] - xs[2 * kXs + j];
                const float ir = rsqrtf(dx * dx + dy * dy + dz * dz);
                const float jn = (dx * (us[i] - us[j]) + dy * (us[kXs + i] - us[kXs + j]) +
                                  dz * (us[2 * kXs + i] - us[2 * kXs + j])) *
                                 ir * ir * ir;
                v = jn * L.inv_sd[p];
            }
            nrow[p] = __float2bfloat16(v);
        }
        if (threadIdx.x == 0) {
            const double e = head_energy(L.part, L.nparts, m, L.b3);
            const double de = e - (L.E_ref[src] - L.mu_E) * inv_sE;
            L.ebar[m] = (float)(2.0 * de / (double)L.M);
            L.loss_part[m] = de * de + L.lam / (3.0 * L.N) * sq;
        }
    }
}

// Reverse pass through the two hidden layers.  Tiles of kBarRows samples m by
// kBarCols hidden units h, 256 threads: a thread keeps one column h and walks
// the tile's rows four apart, reads and writes are coalesced along h, and the
// bias and w3 gradients' sums over the samples start here, in FP64 in
// registers, so that their per-sample terms never go to memory.  Each tile
// leaves one partial per column; mlp_sums_kernel adds those.
// Bound by the FP64 conversions and additions (two per element and sum on
// units that do a 64th of the FP32 rate) and the latency of one tile.  At 2048
// samples and H = 512: layer 2 13.9 us, layer 1 10.0 us, sums 5.3 us (tiles of
// 64 rows: 15.9, 14.7, 5.3); with element-wise kernels that stored the terms
// and column sums of four blocks, each thread walking all samples in one
// serial FP64 chain, 14.8 + 14.1 + 3 x 249 + 167 us.
constexpr int kBarRows = 32, kBarCols = 64, kBarThreads = 256;

struct BarArgs {
    int M, H;
    const float* ebar;       // [M]
    const float* z;          // pre-activations of the layer
    const float* s;          // silu'(z)
    const float* zd;         // tangent of z
    const float* up;         // layer 1: dL/dh1; layer 2: unused
    const float* w2d2;       // layer 1: W2^T d2
    const float* w3;         // layer 2
    __nv_bfloat16* zb;       // dL/dz
    double* part_b;          // [tiles][H] partial sums of dL/dz
    double* part_w3;         // layer 2: [tiles][H] partial sums of the w3 gradient
};

// LAYER 2: dL/dz2 = ebar d2 + w3 zd2 silu''(z2), d2 = w3 silu'(z2)
// LAYER 1: dL/dz1 = h1_bar silu'(z1) + (W2^T d2) zd1 silu''(z1)
template <int LAYER>
__global__ void __launch_bounds__(kBarThreads) mlp_zbar_kernel(const BarArgs g) {
    __shared__ double sb[kBarThreads], sw[kBarThreads];
    constexpr int kGroups = kBarThreads / kBarCols, kPer = kBarRows / kGroups;
    const int hl = threadIdx.x % kBarCols, r0 = threadIdx.x / kBarCols;
    const int h = blockIdx.x * kBarCols + hl, m0 = blockIdx.y * kBarRows;
    const bool col = h < g.H;
    const float w = (LAYER == 2 && col) ? g.w3[h] : 0.0f;
    float z[kPer], ds[kPer], td[kPer], u0[kPer], u1[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {  // every load of the tile in flight
        const int m = m0 + r0 + q * kGroups;
        const bool ok = col && m < g.M;
        const size_t e = (size_t)m * g.H + h;
        z[q] = ok ? g.z[e] : 0.0f;
        ds[q] = ok ? g.s[e] : 0.0f;
        td[q] = ok ? g.zd[e] : 0.0f;
        u0[q] = !ok ? 0.0f : LAYER == 2 ? g.ebar[m] : g.up[e];
        u1[q] = (LAYER == 1 && ok) ? g.w2d2[e] : 0.0f;
    }
    double ab = 0.0, aw = 0.0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
        const int m = m0 + r0 + q * kGroups;
        if (!col || m >= g.M) continue;
        float zb;
        if (LAYER == 2) {
            zb = u0[q] * (w * ds[q]) + w * td[q] * d2silu(z[q]);
            aw += (double)(u0[q] * (z[q] * sig(z[q])) + td[q] * ds[q]);
        } else {
            zb = u0[q] * ds[q] + u1[q] * td[q] * d2silu(z[q]);
        }
        ab += (double)zb;
        g.zb[(size_t)m * g.H + h] = __float2bfloat16(zb);
    }
    sb[threadIdx.x] = ab;
    if (LAYER == 2) sw[threadIdx.x] = aw;
    __syncthreads();
    if (r0 == 0 && col) {  // the row groups in order
        double tb = sb[hl], tw = sw[hl];
        for (int q = 1; q < kGroups; ++q) {
            tb += sb[hl + q * kBarCols];
            if (LAYER == 2) tw += sw[hl + q * kBarCols];
        }
        g.part_b[(size_t)blockIdx.y * g.H + h] = tb;
        if (LAYER == 2) g.part_w3[(size_t)blockIdx.y * g.H + h] = tw;
    }
}

// Sums over the samples, in a fixed order and in FP64.  blockIdx.y 0..2: the
// b1, b2 and w3 gradients from their tile partials, 32 columns a block, eight
// threads a column; 3: the b3 gradient; 4: the loss (mean).
struct SumArgs {
    int M, H, tiles;
    const double* part[3];
    float* out[3];
    const float* ebar;
    float* out_b3;
    const double* loss_part;
    double* out_loss;
};
__global__ void __launch_bounds__(256) mlp_sums_kernel(const SumArgs g) {
    __shared__ double red[256];
    if (blockIdx.y < 3) {
        const int c = threadIdx.x & 31, q = threadIdx.x >> 5, h = blockIdx.x * 32 + c;
        const double* p = g.part[blockIdx.y];
        double s = 0.0;
        for (int t = q; t < g.tiles; t += 8) s += p[(size_t)t * g.H + h];  // H is a multiple of 32
        red[threadIdx.x] = s;
        __syncthreads();
        if (q == 0) {
            for (int u = 1; u < 8; ++u) s += red[c + 32 * u];
            g.out[blockIdx.y][h] = (float)s;
        }
        return;
    }
    if (blockIdx.x) return;
    double s = 0.0;
    if (blockIdx.y == 3)
        for (int m = threadIdx.x; m < g.M; m += 256) s += (double)g.ebar[m];
    else
        for (int m = threadIdx.x; m < g.M; m += 256) s += g.loss_part[m];
    s = block_sum(s, red);
    if (threadIdx.x) return;
    if (blockIdx.y == 3) *g.out_b3 = (float)s;
    else *g.out_loss = s / (double)g.M;
}

// ------------------------------------------------------------------ helpers

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

int launch_check(pamd_mlp* m, const char* what) {
    m->launches += 1;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return mcuda(m, e, what);
    return PAMD_OK;
}

int gemm(pamd_mlp* m, GemmArgs g, cudaStream_t s, int* status = nullptr) {
    g.status = status ? status : m->status;
    const cudaError_t e = launch_gemm_bf16(g, s);
    m->launches += 1;
    if (e != cudaSuccess) return mcuda(m, e, "tensor-core GEMM launch");
    return PAMD_OK;
}

int check_model(pamd_mlp* m) {
    if (!m) return mfail(PAMD_EINVAL, "null model");
    if (m->broken) return mfail(PAMD_ESTATE, "model unusable after an earlier CUDA error");
    return PAMD_OK;
}

int read_model_status(pamd_mlp* m) {
    int st = 0;
    MLP_CU(m, cudaMemcpyAsync(&st, m->status, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
    MLP_CU(m, cudaStreamSynchronize(m->stream));
    if (st) {
        m->broken = true;
        return mfail(st, "tensor-core pipeline timed out");
    }
    return PAMD_OK;
}

WeightCopies weight_copies(const pamd_mlp* m) {
    return {m->oW1, (size_t)m->H * m->Pp, m->oW2, (size_t)m->H * m->H, m->W1b, m->W2b};
}

int pack(pamd_mlp* m) {
    const long long n = (long long)m->ob2;  // W1, b1 and W2 come first
    mlp_pack_kernel<<<grid_for(n, 256), 256, 0, m->stream>>>(m->params, n, weight_copies(m));
    return launch_check(m, "weight pack");
}

size_t forces_smem(const pamd_mlp* m) { return sizeof(float) * (3 * kXs + (size_t)m->Pp); }
size_t loss_smem(const pamd_mlp* m) { return sizeof(float) * (6 * kXs + (size_t)m->Pp); }

// The dynamic shared-memory limits of the force and loss kernels on the
// current device, raised to what this model needs.
int set_smem_attrs(const pamd_mlp* m) {
    cudaError_t e = gamma_matrix(m->N) ? ensure_dyn_smem((const void*)forces_duo_kernel(m->N), duo_smem(m->N, m->Pp).total)
                                       : ensure_dyn_smem((const void*)mlp_forces_kernel, forces_smem(m));
    if (e == cudaSuccess)
        e = gamma_matrix(m->N) ? ensure_dyn_smem((const void*)loss_duo_kernel(m->N), loss_duo_smem(m->N, m->Pp))
                               : ensure_dyn_smem((const void*)mlp_loss_kernel, loss_smem(m));
    return e == cudaSuccess ? PAMD_OK : mfail(PAMD_ECUDA, std::string("kernel attributes: ") + cudaGetErrorString(e));
}

int features(pamd_mlp* m, const ConfigView& cv, int M, __nv_bfloat16* a) {
    FeatArgs f{};
    f.cv = cv;
    f.M = M;
    f.N = m->N;
    f.P = m->P;
    f.Pp = m->Pp;
    f.pairs = m->pairs;
    f.mu = m->mu;
    f.inv_sd = m->inv_sd;
    f.a = a;
    // Eight configurations a block read the tables least; two keep enough
    // blocks in flight below four waves of the chip.  Whole energy call, 75
    // atoms, eight / two, us: M 64 41.9 / 36.8, 1024 43.9 / 41.9, 4096 52.1 /
    // 51.1, 8192 62.4 / 64.5, 65536 290 / 334.
    if (M >= 8 * 152 * 4)
        mlp_features_kernel<4><<<(M + 7) / 8, kFeatThreads, 4 * duo_pos_bytes(m->N), m->stream>>>(f);
    else
        mlp_features_kernel<1><<<(M + 1) / 2, kFeatThreads, duo_pos_bytes(m->N), m->stream>>>(f);
    return launch_check(m, "features");
}

}  // namespace

// Workspace of cap >= M configurations (grows only; training buffers once
// requested stay).
int mlp_ensure_work(pamd_mlp* m, long long M, bool train) {
    MlpWork& w = m->w;
    if (M <= w.cap && (!train || w.train)) return PAMD_OK;
    const long long cap = M > w.cap ? ((M + 127) / 128) * 128 : w.cap;
    const bool tr = train || w.train;
    const size_t H = (size_t)m->H, Pp = (size_t)m->Pp, C = (size_t)cap;
    std::vector<size_t> sizes;
    // order: a h1 d2 d1 s1 ga part | z1 z2 s2 w2d2 zd1 zd2 h1b A1 B1 A2 B2 ebar loss sums
    sizes = {2 * C * Pp, 2 * C * H, 2 * C * H, 2 * C * H, 4 * C * H, 2 * C * Pp, 4 * C * (size_t)m->nparts};
    if (tr) {
        for (int i = 0; i < 7; ++i) sizes.push_back(4 * C * H);
        sizes.push_back(2 * H * 2 * C);
        sizes.push_back(2 * Pp * 2 * C);
        sizes.push_back(2 * H * 2 * C);
        sizes.push_back(2 * H * 2 * C);
        sizes.push_back(4 * C);
        sizes.push_back(8 * C);
        sizes.push_back(3 * 8 * H * ((C + kBarRows - 1) / kBarRows));
    }
    size_t total = 0;
    for (size_t s : sizes) total += align256(s);
    void* base = nullptr;
    if (cudaMalloc(&base, total) != cudaSuccess) {
        cudaGetLastError();
        return mfail(PAMD_ENOMEM, "surrogate workspace: cudaMalloc failed");
    }
    if (w.base) {
        cudaStreamSynchronize(m->stream);
        cudaFree(w.base);
    }
    // graphs captured over another workspace are stale: also one of a model
    // that was destroyed and whose address this one took
    static std::atomic<long long> generations{0};
    m->work_gen = ++generations;
    MlpWork nw;
    nw.cap = cap;
    nw.train = tr;
    nw.base = base;
    char* p = static_cast<char*>(base);
    size_t k = 0;
    auto take = [&]() {
        char* r = p;
        p += align256(sizes[k++]);
        return r;
    };
    nw.a = reinterpret_cast<__nv_bfloat16*>(take());
    nw.h1 = reinterpret_cast<__nv_bfloat16*>(take());
    nw.d2 = reinterpret_cast<__nv_bfloat16*>(take());
    nw.d1 = reinterpret_cast<__nv_bfloat16*>(take());
    nw.s1 = reinterpret_cast<float*>(take());
    nw.ga = reinterpret_cast<__nv_bfloat16*>(take());
    nw.part = reinterpret_cast<float*>(take());
    if (tr) {
        float** f32[7] = {&nw.z1, &nw.z2, &nw.s2, &nw.w2d2, &nw.zd1, &nw.zd2, &nw.h1b};
        for (auto q : f32) *q = reinterpret_cast<float*>(take());
        nw.A1 = reinterpret_cast<__nv_bfloat16*>(take());
        nw.B1 = reinterpret_cast<__nv_bfloat16*>(take());
        nw.A2 = reinterpret_cast<__nv_bfloat16*>(take());
        nw.B2 = reinterpret_cast<__nv_bfloat16*>(take());
        nw.ebar = reinterpret_cast<float*>(take());
        nw.loss_part = reinterpret_cast<double*>(take());
        nw.sum_part = reinterpret_cast<double*>(take());
    }
    w = nw;
    return PAMD_OK;
}

int mlp_prepare_capture(pamd_mlp* m) {
    if (!m->loop_ctr && cudaMalloc(&m->loop_ctr, sizeof(int)) != cudaSuccess) {
        m->loop_ctr = nullptr;
        cudaGetLastError();
        return mfail(PAMD_ENOMEM, "surrogate loop counter");
    }
    if (!m->body_stream && cudaStreamCreateWithFlags(&m->body_stream, cudaStreamNonBlocking) != cudaSuccess) {
        m->body_stream = nullptr;
        cudaGetLastError();
        return mfail(PAMD_ECUDA, "surrogate capture stream");
    }
    const cudaError_t e = gemm_prepare_device();
    if (e != cudaSuccess) return mcuda(m, e, "tensor-core GEMM set-up");
    return PAMD_OK;
}

int mlp_gemms(pamd_mlp* m, int M, bool forces, cudaStream_t s, int* status) {
    const MlpWork& w = m->w;
    const int H = m->H, Pp = m->Pp;
    int rc;
    GemmArgs g{};
    // layer 1: h1 = silu(a W1^T + b1), s1 = silu'(.)
    g.A = w.a; g.B = m->W1b; g.M = M; g.N = H; g.K = Pp; g.lda = Pp; g.ldb = Pp;
    g.bias = m->params + m->ob1; g.epi = kEpiSilu;
    g.Cs = w.s1; g.ldc = H; g.Cb = w.h1; g.ldcb = H;
    if ((rc = gemm(m, g, s, status))) return rc;
    // layer 2 and head: d2 = w3 silu'(z2), partial sums of w3 . silu(z2)
    g = GemmArgs{};
    g.A = w.h1; g.B = m->W2b; g.M = M; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.bias = m->params + m->ob2; g.epi = kEpiHead; g.vec = m->params + m->ow3;
    g.Cb = w.d2; g.ldcb = H; g.ldc = H; g.part = w.part;
    if ((rc = gemm(m, g, s, status))) return rc;
    if (!forces) return PAMD_OK;
    // d1 = (d2 W2) * s1
    g = GemmArgs{};
    g.mode = kGemmNN; g.A = w.d2; g.B = m->W2b; g.M = M; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.epi = kEpiMul; g.mul = w.s1; g.ldc = H; g.Cb = w.d1; g.ldcb = H;
    if ((rc = gemm(m, g, s, status))) return rc;
    // de/da = d1 W1
    g = GemmArgs{};
    g.mode = kGemmNN; g.A = w.d1; g.B = m->W1b; g.M = M; g.N = Pp; g.K = H; g.lda = H; g.ldb = Pp;
    g.epi = kEpiStore; g.Cb = w.ga; g.ldcb = Pp; g.ldc = Pp;
    return gemm(m, g, s, status);
}

}  // namespace pamd

using namespace pamd;

extern "C" {

int pamd_mlp_create(pamd_mlp** out, int32_t n_atoms, int32_t hidden, uint64_t seed, void* stream) {
    if (!out) return mfail(PAMD_EINVAL, "pamd_mlp_create: null output");
    *out = nullptr;
    if (n_atoms < 2 || n_atoms > PAMD_MAX_ATOMS)
        return mfail(PAMD_EINVAL, "pamd_mlp_create: n_atoms must be in 2.." + std::to_string(PAMD_MAX_ATOMS));
    if (hidden < 32 || hidden > 1024 || hidden % 32)
        return mfail(PAMD_EINVAL, "pamd_mlp_create: hidden must be 32..1024, a multiple of 32");
    pamd_mlp* m = new pamd_mlp;
    m->N = n_atoms;
    m->P = n_atoms * (n_atoms - 1) / 2;
    m->Pp = (m->P + 7) / 8 * 8;
    m->H = hidden;
    m->nparts = gemm_head_parts(hidden);
    const size_t H = (size_t)hidden, Pp = (size_t)m->Pp;
    m->oW1 = 0;
    m->ob1 = H * Pp;
    m->oW2 = m->ob1 + H;
    m->ob2 = m->oW2 + H * H;
    m->ow3 = m->ob2 + H;
    m->ob3 = m->ow3 + H;
    m->n_params = m->ob3 + 4;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        delete m;
        return mfail(PAMD_ECUDA, "pamd_mlp_create: no CUDA device");
    }
    m->max_slices = stat_slices(m->P, sms);
    const size_t pbytes = align256(4 * m->n_params);
    const size_t sizes[] = {pbytes, pbytes, pbytes, pbytes, align256(4 * Pp), align256(4 * Pp),
                            align256(4 * Pp), align256(2 * H * Pp), align256(2 * H * H), align256(4 * Pp),
                            align256(sizeof(int)), align256(8 * 4),
                            align256(sizeof(double2) * (size_t)m->max_slices * (m->P + 1))};
    size_t total = 0;
    for (size_t s : sizes) total += s;
    if (stream) {
        m->stream = static_cast<cudaStream_t>(stream);
    } else {
        if (cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking) != cudaSuccess) {
            delete m;
            return mfail(PAMD_ECUDA, "pamd_mlp_create: stream creation failed");
        }
        m->own_stream = true;
    }
    if (cudaMalloc(&m->base, total) != cudaSuccess) {
        cudaGetLastError();
        pamd_mlp_destroy(m);
        return mfail(PAMD_ENOMEM, "pamd_mlp_create: cudaMalloc failed");
    }
    char* p = static_cast<char*>(m->base);
    int k = 0;
    auto take = [&]() {
        char* r = p;
        p += sizes[k++];
        return r;
    };
    m->params = reinterpret_cast<float*>(take());
    m->grads = reinterpret_cast<float*>(take());
    m->adam_m = reinterpret_cast<float*>(take());
    m->adam_v = reinterpret_cast<float*>(take());
    m->mu = reinterpret_cast<float*>(take());
    m->sd = reinterpret_cast<float*>(take());
    m->inv_sd = reinterpret_cast<float*>(take());
    m->W1b = reinterpret_cast<__nv_bfloat16*>(take());
    m->W2b = reinterpret_cast<__nv_bfloat16*>(take());
    m->pairs = reinterpret_cast<ushort2*>(take());
    m->status = reinterpret_cast<int*>(take());
    m->scratch = reinterpret_cast<double*>(take());
    m->moments = reinterpret_cast<double2*>(take());
    // pair table, identity normalisation, zero moments
    std::vector<ushort2> pr(Pp, make_ushort2(0, 0));
    for (int i = 0, q = 0; i < n_atoms; ++i)
        for (int j = i + 1; j < n_atoms; ++j, ++q) pr[q] = make_ushort2((unsigned short)i, (unsigned short)j);
    std::vector<float> zeros(Pp, 0.0f), ones(Pp, 1.0f);
    cudaStream_t s = m->stream;
    int rc = PAMD_OK;
    if (cudaMemcpyAsync(m->pairs, pr.data(), 4 * Pp, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(m->mu, zeros.data(), 4 * Pp, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(m->sd, ones.data(), 4 * Pp, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(m->inv_sd, ones.data(), 4 * Pp, cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemsetAsync(m->params, 0, 4 * pbytes, s) != cudaSuccess ||
        cudaMemsetAsync(m->status, 0, sizeof(int), s) != cudaSuccess)
        rc = mcuda(m, cudaGetLastError(), "pamd_mlp_create: initial copies");
    if (!rc) {
        const long long n = (long long)H * Pp + (long long)H * H + (long long)H;
        mlp_init_kernel<<<grid_for(n, 256), 256, 0, s>>>(m->params, m->oW1, m->oW2, m->ow3, m->H,
                                                         m->P, m->Pp, seed);
        rc = launch_check(m, "weight init");
    }
    if (!rc) rc = pack(m);
    if (!rc) rc = set_smem_attrs(m);
    if (!rc && cudaStreamSynchronize(s) != cudaSuccess) rc = mcuda(m, cudaGetLastError(), "pamd_mlp_create");
    if (rc) {
        const std::string msg = pamd_last_error();
        pamd_mlp_destroy(m);
        return mfail(rc, msg);
    }
    *out = m;
    return PAMD_OK;
}

int pamd_mlp_info(pamd_mlp* m, int32_t* n_atoms, int32_t* n_pairs, int32_t* hidden) {
    if (!m) return mfail(PAMD_EINVAL, "null model");
    if (n_atoms) *n_atoms = m->N;
    if (n_pairs) *n_pairs = m->P;
    if (hidden) *hidden = m->H;
    return PAMD_OK;
}

int pamd_mlp_set_params(pamd_mlp* m, const pamd_mlp_params* hp) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!hp) return mfail(PAMD_EINVAL, "pamd_mlp_set_params: null parameters");
    if (hp->sd)
        for (int p = 0; p < m->P; ++p)
            if (!(hp->sd[p] > 0.0f) || !std::isfinite(hp->sd[p]))
                return mfail(PAMD_EINVAL, "pamd_mlp_set_params: sd must be positive and finite");
    if (!(hp->sigma_E > 0.0) || !std::isfinite(hp->sigma_E) || !std::isfinite(hp->mu_E) ||
        !std::isfinite(hp->b3))
        return mfail(PAMD_EINVAL, "pamd_mlp_set_params: sigma_E > 0, mu_E and b3 finite");
    const int H = m->H, P = m->P, Pp = m->Pp;
    std::vector<float> buf((size_t)m->n_params);
    MLP_CU(m, cudaMemcpy(buf.data(), m->params, 4 * m->n_params, cudaMemcpyDeviceToHost));
    if (hp->W1)
        for (int h = 0; h < H; ++h)
            std::memcpy(&buf[m->oW1 + (size_t)h * Pp], hp->W1 + (size_t)h * P, 4 * (size_t)P);
    if (hp->b1) std::memcpy(&buf[m->ob1], hp->b1, 4 * (size_t)H);
    if (hp->W2) std::memcpy(&buf[m->oW2], hp->W2, 4 * (size_t)H * H);
    if (hp->b2) std::memcpy(&buf[m->ob2], hp->b2, 4 * (size_t)H);
    if (hp->w3) std::memcpy(&buf[m->ow3], hp->w3, 4 * (size_t)H);
    buf[m->ob3] = (float)hp->b3;
    MLP_CU(m, cudaMemcpy(m->params, buf.data(), 4 * m->n_params, cudaMemcpyHostToDevice));
    if (hp->mu || hp->sd) {
        std::vector<float> mu(Pp, 0.0f), sd(Pp, 1.0f), isd(Pp, 1.0f);
        MLP_CU(m, cudaMemcpy(mu.data(), m->mu, 4 * (size_t)Pp, cudaMemcpyDeviceToHost));
        MLP_CU(m, cudaMemcpy(sd.data(), m->sd, 4 * (size_t)Pp, cudaMemcpyDeviceToHost));
        if (hp->mu) std::memcpy(mu.data(), hp->mu, 4 * (size_t)P);
        if (hp->sd) std::memcpy(sd.data(), hp->sd, 4 * (size_t)P);
        for (int p = 0; p < Pp; ++p) isd[p] = (float)(1.0 / (double)sd[p]);
        MLP_CU(m, cudaMemcpy(m->mu, mu.data(), 4 * (size_t)Pp, cudaMemcpyHostToDevice));
        MLP_CU(m, cudaMemcpy(m->sd, sd.data(), 4 * (size_t)Pp, cudaMemcpyHostToDevice));
        MLP_CU(m, cudaMemcpy(m->inv_sd, isd.data(), 4 * (size_t)Pp, cudaMemcpyHostToDevice));
    }
    m->mu_E = hp->mu_E;
    m->sigma_E = hp->sigma_E;
    MLP_CU(m, cudaMemsetAsync(m->adam_m, 0, 4 * m->n_params, m->stream));
    MLP_CU(m, cudaMemsetAsync(m->adam_v, 0, 4 * m->n_params, m->stream));
    m->adam_t = 0;
    if ((rc = pack(m))) return rc;
    MLP_CU(m, cudaStreamSynchronize(m->stream));
    return PAMD_OK;
}

static int copy_out(pamd_mlp* m, const float* src, pamd_mlp_params* hp, bool with_norm) {
    const int H = m->H, P = m->P, Pp = m->Pp;
    std::vector<float> buf((size_t)m->n_params);
    MLP_CU(m, cudaStreamSynchronize(m->stream));
    MLP_CU(m, cudaMemcpy(buf.data(), src, 4 * m->n_params, cudaMemcpyDeviceToHost));
    if (hp->W1)
        for (int h = 0; h < H; ++h)
            std::memcpy(hp->W1 + (size_t)h * P, &buf[m->oW1 + (size_t)h * Pp], 4 * (size_t)P);
    if (hp->b1) std::memcpy(hp->b1, &buf[m->ob1], 4 * (size_t)H);
    if (hp->W2) std::memcpy(hp->W2, &buf[m->oW2], 4 * (size_t)H * H);
    if (hp->b2) std::memcpy(hp->b2, &buf[m->ob2], 4 * (size_t)H);
    if (hp->w3) std::memcpy(hp->w3, &buf[m->ow3], 4 * (size_t)H);
    hp->b3 = buf[m->ob3];
    if (with_norm) {
        if (hp->mu) MLP_CU(m, cudaMemcpy(hp->mu, m->mu, 4 * (size_t)P, cudaMemcpyDeviceToHost));
        if (hp->sd) MLP_CU(m, cudaMemcpy(hp->sd, m->sd, 4 * (size_t)P, cudaMemcpyDeviceToHost));
        hp->mu_E = m->mu_E;
        hp->sigma_E = m->sigma_E;
    }
    return PAMD_OK;
}

int pamd_mlp_get_params(pamd_mlp* m, pamd_mlp_params* hp) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!hp) return mfail(PAMD_EINVAL, "pamd_mlp_get_params: null output");
    return copy_out(m, m->params, hp, true);
}

int pamd_mlp_get_grads(pamd_mlp* m, pamd_mlp_params* hp) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!hp) return mfail(PAMD_EINVAL, "pamd_mlp_get_grads: null output");
    if ((rc = read_model_status(m))) return rc;
    return copy_out(m, m->grads, hp, false);
}

int pamd_mlp_fit_normalization(pamd_mlp* m, const float* x_dev, const double* E_dev, int64_t n) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!x_dev || !E_dev || n < 2) return mfail(PAMD_EINVAL, "pamd_mlp_fit_normalization: null pointer or n < 2");
    const int cols = stat_columns(m->P);
    const int tile = kStatTileBytes / (16 * m->N) > 0 ? kStatTileBytes / (16 * m->N) : 1;
    long long slices = (n + tile - 1) / tile;  // a tile each at least
    if (slices > m->max_slices) slices = m->max_slices;
    const long long per = (n + slices - 1) / slices;
    slices = (n + per - 1) / per;  // no empty slice
    mlp_moments_kernel<<<dim3(cols, (unsigned)slices), kStatThreads, sizeof(float4) * (size_t)tile * m->N, m->stream>>>(
        x_dev, E_dev, n, per, m->N, m->P, tile, m->pairs, m->moments);
    if ((rc = launch_check(m, "feature statistics"))) return rc;
    mlp_moments_merge_kernel<<<(m->P + 4) / 4, 128, 0, m->stream>>>(x_dev, n, per, (int)slices, m->N, m->P, m->pairs,
                                                                    m->moments, m->mu, m->sd, m->inv_sd, m->scratch);
    if ((rc = launch_check(m, "feature statistics"))) return rc;
    double st[2];
    MLP_CU(m, cudaMemcpyAsync(st, m->scratch, sizeof(st), cudaMemcpyDeviceToHost, m->stream));
    MLP_CU(m, cudaStreamSynchronize(m->stream));
    if (!std::isfinite(st[0]) || !std::isfinite(st[1]))
        return mfail(PAMD_EINVAL, "pamd_mlp_fit_normalization: non-finite energies");
    m->mu_E = st[0];
    m->sigma_E = st[1] > 0.0 ? st[1] : 1.0;
    return PAMD_OK;
}

int pamd_mlp_energy_forces(pamd_mlp* m, const float* x_dev, int64_t M, double* E_dev, float* F_dev) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!x_dev || M < 1 || M > (1LL << 24)) return mfail(PAMD_EINVAL, "pamd_mlp_energy_forces: null x or M");
    if (!E_dev && !F_dev) return PAMD_OK;
    if ((rc = mlp_ensure_work(m, M, false))) return rc;
    const ConfigView cv{x_dev, 3LL * m->N, 3, 1, nullptr};
    if ((rc = features(m, cv, (int)M, m->w.a))) return rc;
    if ((rc = mlp_gemms(m, (int)M, F_dev != nullptr, m->stream, m->status))) return rc;
    ForceArgs f{};
    f.cv = cv;
    f.M = (int)M;
    f.N = m->N;
    f.P = m->P;
    f.Pp = m->Pp;
    f.nparts = m->nparts;
    f.ga = m->w.ga;
    f.pairs = m->pairs;
    f.part = m->w.part;
    f.inv_sd = m->inv_sd;
    f.b3 = m->params + m->ob3;
    f.sigma_E = m->sigma_E;
    f.mu_E = m->mu_E;
    f.E = E_dev;
    f.F = F_dev;
    if (gamma_matrix(m->N)) {
        const int t = duo_threads(m->N);
        const int grid = F_dev ? grid_for((M + 1) / 2 * t, t, 152 * duo_blocks(t)) : grid_for(M, t);
        forces_duo_kernel(m->N)<<<grid, t, duo_smem(m->N, m->Pp).total, m->stream>>>(f);
    } else {
        mlp_forces_kernel<<<F_dev ? grid_for(M * kMlpThreads, kMlpThreads, 152 * 16) : grid_for(M, kMlpThreads), kMlpThreads,
                            forces_smem(m), m->stream>>>(f);
    }
    return launch_check(m, "surrogate forces");
}

int pamd_mlp_loss_grads(pamd_mlp* m, const float* x_dev, const double* E_dev, const float* F_dev,
                        const int32_t* idx_dev, int64_t M, double lam, double* loss) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!x_dev || !E_dev || !F_dev) return mfail(PAMD_EINVAL, "pamd_mlp_loss_grads: null data pointer");
    if (M < 4 || M > 65536 || M % 4) return mfail(PAMD_EINVAL, "pamd_mlp_loss_grads: M must be 4..65536, a multiple of 4");
    if (!(lam >= 0.0) || !std::isfinite(lam)) return mfail(PAMD_EINVAL, "pamd_mlp_loss_grads: lam must be >= 0");
    if ((rc = mlp_ensure_work(m, M, true))) return rc;
    const MlpWork& w = m->w;
    const int H = m->H, Pp = m->Pp, Mi = (int)M;
    cudaStream_t s = m->stream;
    const ConfigView cv{x_dev, 3LL * m->N, 3, 1, idx_dev};
    // the operands of the weight gradients: M rows of the energy part, then M
    // of the force part (see MlpWork)
    const size_t MH = (size_t)Mi * H;
    __nv_bfloat16 *const a = w.B1, *const nu_a = w.B1 + (size_t)Mi * Pp, *const h1 = w.B2, *const hd1 = w.B2 + MH,
                  *const z1b = w.A1, *const d1 = w.A1 + MH, *const z2b = w.A2, *const d2 = w.A2 + MH;
    // forward, keeping what the gradient needs
    if ((rc = features(m, cv, Mi, a))) return rc;
    GemmArgs g{};
    g.A = a; g.B = m->W1b; g.M = Mi; g.N = H; g.K = Pp; g.lda = Pp; g.ldb = Pp;
    g.bias = m->params + m->ob1; g.epi = kEpiSilu;
    g.C = w.z1; g.Cs = w.s1; g.ldc = H; g.Cb = h1; g.ldcb = H;
    if ((rc = gemm(m, g, s))) return rc;
    g = GemmArgs{};
    g.A = h1; g.B = m->W2b; g.M = Mi; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.bias = m->params + m->ob2; g.epi = kEpiHead; g.vec = m->params + m->ow3;
    g.C = w.z2; g.Cs = w.s2; g.ldc = H; g.Cb = d2; g.ldcb = H;
    g.part = w.part;
    if ((rc = gemm(m, g, s))) return rc;
    g = GemmArgs{};
    g.mode = kGemmNN; g.A = d2; g.B = m->W2b; g.M = Mi; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.epi = kEpiMul; g.mul = w.s1; g.C = w.w2d2; g.ldc = H; g.Cb = d1; g.ldcb = H;
    if ((rc = gemm(m, g, s))) return rc;
    g = GemmArgs{};
    g.mode = kGemmNN; g.A = d1; g.B = m->W1b; g.M = Mi; g.N = Pp; g.K = H; g.lda = H; g.ldb = Pp;
    g.epi = kEpiStore; g.Cb = w.ga; g.ldcb = Pp; g.ldc = Pp;
    if ((rc = gemm(m, g, s))) return rc;
    // loss, energy cotangent and the tangent direction nu_a
    LossArgs L{};
    L.cv = cv;
    L.E_ref = E_dev;
    L.F_ref = F_dev;
    L.M = Mi;
    L.N = m->N;
    L.P = m->P;
    L.Pp = Pp;
    L.nparts = m->nparts;
    L.pairs = m->pairs;
    L.ga = w.ga;
    L.part = w.part;
    L.inv_sd = m->inv_sd;
    L.b3 = m->params + m->ob3;
    L.mu_E = m->mu_E;
    L.sigma_E = m->sigma_E;
    L.lam = lam;
    L.nu_a = nu_a;
    L.ebar = w.ebar;
    L.loss_part = w.loss_part;
    if (gamma_matrix(m->N)) {
        const int t = duo_threads_wide(m->N);
        loss_duo_kernel(m->N)<<<grid_for((M + 1) / 2 * t, t, 152 * (t == 384 ? 3 : duo_blocks(t))), t,
                                loss_duo_smem(m->N, m->Pp), s>>>(L);
    } else {
        mlp_loss_kernel<<<grid_for(M * kMlpThreads, kMlpThreads, 152 * 16), kMlpThreads, loss_smem(m), s>>>(L);
    }
    if ((rc = launch_check(m, "loss"))) return rc;
    // tangent pass: zd1 = W1 nu_a, hd1 = zd1 s1, zd2 = W2 hd1
    g = GemmArgs{};
    g.A = nu_a; g.B = m->W1b; g.M = Mi; g.N = H; g.K = Pp; g.lda = Pp; g.ldb = Pp;
    g.epi = kEpiMul; g.mul = w.s1; g.C = w.zd1; g.ldc = H; g.Cb = hd1; g.ldcb = H;
    if ((rc = gemm(m, g, s))) return rc;
    g = GemmArgs{};
    g.A = hd1; g.B = m->W2b; g.M = Mi; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.epi = kEpiStore; g.C = w.zd2; g.ldc = H;
    if ((rc = gemm(m, g, s))) return rc;
    // reverse: z2_bar, h1_bar = z2_bar W2, z1_bar
    const int tiles = (Mi + kBarRows - 1) / kBarRows;
    const size_t psz = (size_t)tiles * H;
    const dim3 bar_grid((H + kBarCols - 1) / kBarCols, tiles);
    BarArgs bar{};
    bar.M = Mi; bar.H = H; bar.ebar = w.ebar;
    bar.z = w.z2; bar.s = w.s2; bar.zd = w.zd2; bar.w3 = m->params + m->ow3;
    bar.zb = z2b; bar.part_b = w.sum_part + psz; bar.part_w3 = w.sum_part + 2 * psz;
    mlp_zbar_kernel<2><<<bar_grid, kBarThreads, 0, s>>>(bar);
    if ((rc = launch_check(m, "z2 cotangent"))) return rc;
    g = GemmArgs{};
    g.mode = kGemmNN; g.A = z2b; g.B = m->W2b; g.M = Mi; g.N = H; g.K = H; g.lda = H; g.ldb = H;
    g.epi = kEpiStore; g.C = w.h1b; g.ldc = H;
    if ((rc = gemm(m, g, s))) return rc;
    bar.z = w.z1; bar.s = w.s1; bar.zd = w.zd1; bar.up = w.h1b; bar.w2d2 = w.w2d2;
    bar.zb = z1b; bar.part_b = w.sum_part;
    mlp_zbar_kernel<1><<<bar_grid, kBarThreads, 0, s>>>(bar);
    if ((rc = launch_check(m, "z1 cotangent"))) return rc;
    // weight gradients: contractions over the 2M rows of the operands
    g = GemmArgs{};
    g.mode = kGemmTN;
    g.A = w.A1; g.B = w.B1; g.M = H; g.N = Pp; g.K = 2 * Mi; g.lda = H; g.ldb = Pp;
    g.epi = kEpiStore; g.C = m->grads + m->oW1; g.ldc = Pp;
    if ((rc = gemm(m, g, s))) return rc;
    g = GemmArgs{};
    g.mode = kGemmTN;
    g.A = w.A2; g.B = w.B2; g.M = H; g.N = H; g.K = 2 * Mi; g.lda = H; g.ldb = H;
    g.epi = kEpiStore; g.C = m->grads + m->oW2; g.ldc = H;
    if ((rc = gemm(m, g, s))) return rc;
    SumArgs sums{};
    sums.M = Mi; sums.H = H; sums.tiles = tiles;
    sums.part[0] = w.sum_part; sums.part[1] = w.sum_part + psz; sums.part[2] = w.sum_part + 2 * psz;
    sums.out[0] = m->grads + m->ob1; sums.out[1] = m->grads + m->ob2; sums.out[2] = m->grads + m->ow3;
    sums.ebar = w.ebar; sums.out_b3 = m->grads + m->ob3;
    sums.loss_part = w.loss_part; sums.out_loss = m->scratch;
    mlp_sums_kernel<<<dim3(H / 32, 5), 256, 0, s>>>(sums);
    if ((rc = launch_check(m, "sums over the samples"))) return rc;
    if (loss) {
        MLP_CU(m, cudaMemcpyAsync(loss, m->scratch, sizeof(double), cudaMemcpyDeviceToHost, s));
        if ((rc = read_model_status(m))) return rc;
    }
    return PAMD_OK;
}

int pamd_mlp_adam_step(pamd_mlp* m, double lr, double beta1, double beta2, double eps) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!(lr > 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
        return mfail(PAMD_EINVAL, "pamd_mlp_adam_step: lr > 0, 0 <= beta < 1, eps > 0");
    m->adam_t += 1;
    const float bc1 = (float)(1.0 - std::pow(beta1, (double)m->adam_t));
    const float bc2 = (float)(1.0 - std::pow(beta2, (double)m->adam_t));
    const long long n = (long long)m->ob3 + 1;
    mlp_adam_kernel<<<grid_for(n, 256), 256, 0, m->stream>>>(m->params, m->grads, m->adam_m, m->adam_v, n,
                                                             (float)lr, (float)beta1, (float)beta2,
                                                             (float)eps, bc1, bc2, weight_copies(m));
    return launch_check(m, "Adam");
}

// Model file: magic, {N, H}, the FP32 parameter block (W1 padded to Pp
// columns), mu and sd [Pp], mu_E, sigma_E, FNV-1a 64 checksum of all before.
static const char kMlpMagic[8] = {'P', 'A', 'M', 'D', 'M', 'L', 'P', '1'};

static uint64_t mlp_fnv(const void* d, size_t n, uint64_t h) {
    const unsigned char* b = static_cast<const unsigned char*>(d);
    for (size_t i = 0; i < n; ++i) {
        h ^= b[i];
        h *= 1099511628211ull;
    }
    return h;
}

int pamd_mlp_save(pamd_mlp* m, const char* path) {
    int rc = check_model(m);
    if (rc) return rc;
    if (!path) return mfail(PAMD_EINVAL, "pamd_mlp_save: null path");
    std::vector<float> prm(m->n_params), mu(m->Pp), sd(m->Pp);
    MLP_CU(m, cudaStreamSynchronize(m->stream));
    MLP_CU(m, cudaMemcpy(prm.data(), m->params, 4 * prm.size(), cudaMemcpyDeviceToHost));
    MLP_CU(m, cudaMemcpy(mu.data(), m->mu, 4 * mu.size(), cudaMemcpyDeviceToHost));
    MLP_CU(m, cudaMemcpy(sd.data(), m->sd, 4 * sd.size(), cudaMemcpyDeviceToHost));
    const int32_t shape[2] = {m->N, m->H};
    const double norm[2] = {m->mu_E, m->sigma_E};
    uint64_t h = mlp_fnv(kMlpMagic, 8, 1469598103934665603ull);
    h = mlp_fnv(shape, sizeof(shape), h);
    h = mlp_fnv(prm.data(), 4 * prm.size(), h);
    h = mlp_fnv(mu.data(), 4 * mu.size(), h);
    h = mlp_fnv(sd.data(), 4 * sd.size(), h);
    h = mlp_fnv(norm, sizeof(norm), h);
    const std::string tmp = std::string(path) + ".tmp";
    FILE* f = std::fopen(tmp.c_str(), "wb");
    if (!f) return mfail(PAMD_EINVAL, std::string("pamd_mlp_save: cannot write ") + tmp);
    bool ok = std::fwrite(kMlpMagic, 1, 8, f) == 8 && std::fwrite(shape, sizeof(shape), 1, f) == 1 &&
              std::fwrite(prm.data(), 4, prm.size(), f) == prm.size() &&
              std::fwrite(mu.data(), 4, mu.size(), f) == mu.size() &&
              std::fwrite(sd.data(), 4, sd.size(), f) == sd.size() &&
              std::fwrite(norm, sizeof(norm), 1, f) == 1 && std::fwrite(&h, sizeof(h), 1, f) == 1;
    ok = (std::fclose(f) == 0) && ok;
    if (!ok || std::rename(tmp.c_str(), path) != 0) {
        std::remove(tmp.c_str());
        return mfail(PAMD_EINVAL, std::string("pamd_mlp_save: cannot write ") + path);
    }
    return PAMD_OK;
}

int pamd_mlp_load(pamd_mlp** out, const char* path, void* stream) {
    if (!out || !path) return mfail(PAMD_EINVAL, "pamd_mlp_load: null output or path");
    *out = nullptr;
    FILE* f = std::fopen(path, "rb");
    if (!f) return mfail(PAMD_EINVAL, std::string("pamd_mlp_load: cannot read ") + path);
    char magic[8];
    int32_t shape[2] = {0, 0};
    if (std::fread(magic, 1, 8, f) != 8 || std::memcmp(magic, kMlpMagic, 8) != 0 ||
        std::fread(shape, sizeof(shape), 1, f) != 1) {
        std::fclose(f);
        return mfail(PAMD_EINVAL, std::string("pamd_mlp_load: ") + path + " is not a model file");
    }
    pamd_mlp* m = nullptr;
    int rc = pamd_mlp_create(&m, shape[0], shape[1], 0, stream);
    if (rc) {
        std::fclose(f);
        return rc;
    }
    std::vector<float> prm(m->n_params), mu(m->Pp), sd(m->Pp);
    double norm[2] = {0.0, 1.0};
    uint64_t h_file = 0;
    bool ok = std::fread(prm.data(), 4, prm.size(), f) == prm.size() &&
              std::fread(mu.data(), 4, mu.size(), f) == mu.size() &&
              std::fread(sd.data(), 4, sd.size(), f) == sd.size() &&
              std::fread(norm, sizeof(norm), 1, f) == 1 && std::fread(&h_file, sizeof(h_file), 1, f) == 1;
    std::fclose(f);
    uint64_t h = mlp_fnv(kMlpMagic, 8, 1469598103934665603ull);
    h = mlp_fnv(shape, sizeof(shape), h);
    h = mlp_fnv(prm.data(), 4 * prm.size(), h);
    h = mlp_fnv(mu.data(), 4 * mu.size(), h);
    h = mlp_fnv(sd.data(), 4 * sd.size(), h);
    h = mlp_fnv(norm, sizeof(norm), h);
    bool sane = ok && h == h_file && norm[1] > 0.0 && std::isfinite(norm[0]) && std::isfinite(norm[1]);
    for (size_t p = 0; sane && p < sd.size(); ++p) sane = sd[p] > 0.0f && std::isfinite(sd[p]);
    if (!sane) {
        pamd_mlp_destroy(m);
        return mfail(PAMD_EINVAL, std::string("pamd_mlp_load: ") + path + " is truncated or corrupt");
    }
    std::vector<float> isd(m->Pp);
    for (int p = 0; p < m->Pp; ++p) isd[p] = (float)(1.0 / (double)sd[p]);
    m->mu_E = norm[0];
    m->sigma_E = norm[1];
    cudaError_t e = cudaMemcpy(m->params, prm.data(), 4 * prm.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->mu, mu.data(), 4 * mu.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->sd, sd.data(), 4 * sd.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(m->inv_sd, isd.data(), 4 * isd.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        pamd_mlp_destroy(m);
        return mfail(PAMD_ECUDA, std::string("pamd_mlp_load: ") + cudaGetErrorString(e));
    }
    if ((rc = pack(m)) || (rc = read_model_status(m))) {
        pamd_mlp_destroy(m);
        return rc;
    }
    *out = m;
    return PAMD_OK;
}

int pamd_mlp_sync(pamd_mlp* m) {
    int rc = check_model(m);
    if (rc) return rc;
    return read_model_status(m);
}

int64_t pamd_mlp_launch_count(pamd_mlp* m) { return m ? m->launches : 0; }

void pamd_mlp_destroy(pamd_mlp* m) {
    if (!m) return;
    if (m->stream) cudaStreamSynchronize(m->stream);
    if (m->loop_ctr) cudaFree(m->loop_ctr);
    if (m->body_stream) cudaStreamDestroy(m->body_stream);
    if (m->w.base) cudaFree(m->w.base);
    if (m->base) cudaFree(m->base);
    if (m->own_stream && m->stream) cudaStreamDestroy(m->stream);
    delete m;
}

}  // extern "C"
