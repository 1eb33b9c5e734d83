// mlp_device.cuh -- block-level device helpers of the MLP energy surrogate:
// loading one configuration, its normalised inverse-distance features, and
// the force sum that maps de/dg back onto the atoms.
#pragma once

#include <cuda_bf16.h>

#include "mlp_internal.h"

namespace pamd {

constexpr int kXs = PAMD_MAX_ATOMS;  // stride of a coordinate row in shared memory

// index of pair (i, j), i < j, in row order
__device__ __forceinline__ int pair_id(int i, int j, int N) {
    return i * (2 * N - i - 1) / 2 + (j - i - 1);
}

__device__ __forceinline__ long long config_index(const ConfigView& cv, int m) {
    return cv.idx ? (long long)cv.idx[m] : (long long)m;
}

// xs[c * kXs + i] = coordinate c of atom i of configuration m (whole block)
__device__ __forceinline__ void load_config(const ConfigView& cv, int m, int N, float* xs) {
    const float* x = cv.x + config_index(cv, m) * cv.s_cfg;
    for (int t = threadIdx.x; t < 3 * N; t += blockDim.x) {
        int i, c;
        if (cv.s_coord == 1) {  // [N][3]: consecutive threads read consecutive floats
            i = t / 3;
            c = t - 3 * i;
        } else {
            c = t / N;
            i = t - c * N;
        }
        xs[c * kXs + i] = x[(long long)i * cv.s_atom + (long long)c * cv.s_coord];
    }
}

// ------------------------------------------------ two configurations at a time
// The pair passes are bound by shared-memory reads and instruction issue, not
// by HBM.  Two configurations side by side, (xA, xB, yA, yB) and (zA, zB) per
// atom, halve both: one 16- and one 8-byte read bring an atom of both, the
// packed FP32 instructions work on both, and the pair table is read once.
// Consecutive lanes take consecutive row-order pairs: the reads of atom j are
// free of bank conflicts, those of atom i are broadcasts.  Every element is
// rounded as it would be alone (a multiply by -1 is exact, so the fused
// difference rounds like the subtraction).
struct DuoPos {
    float4* xy;  // [N]
    float2* z;   // [N]
    __device__ __forceinline__ void put(int b, int i, int c, float v) const {
        if (c < 2) reinterpret_cast<float*>(xy)[4 * i + 2 * c + b] = v;
        else reinterpret_cast<float*>(z)[2 * i + b] = v;
    }
};

// a multiple of 16, so that one duo can follow another
__host__ __device__ __forceinline__ size_t duo_pos_bytes(int N) { return (24 * (size_t)N + 15) & ~size_t(15); }
__device__ __forceinline__ DuoPos duo_pos(unsigned char* sm, int N) {
    return DuoPos{reinterpret_cast<float4*>(sm), reinterpret_cast<float2*>(sm + 16 * (size_t)N)};
}

// element r < 3 N of a configuration in the order it lies in memory: atom i, coordinate c
__device__ __forceinline__ void config_element(const ConfigView& cv, int r, int N, int& i, int& c) {
    if (cv.s_coord == 1) {
        i = r / 3;
        c = r - 3 * i;
    } else {
        c = r / N;
        i = r - c * N;
    }
}
__device__ __forceinline__ float config_value(const ConfigView& cv, int m, int i, int c) {
    return cv.x[config_index(cv, m) * cv.s_cfg + (long long)i * cv.s_atom + (long long)c * cv.s_coord];
}

struct Duo3 {
    float2 x, y, z;
};

// x_i - x_j
__device__ __forceinline__ Duo3 duo_diff(const float4 a, const float2 az, const float4 b, const float2 bz) {
    const float2 m1 = make_float2(-1.0f, -1.0f);
    Duo3 d;
    d.x = __ffma2_rn(m1, make_float2(b.x, b.y), make_float2(a.x, a.y));
    d.y = __ffma2_rn(m1, make_float2(b.z, b.w), make_float2(a.z, a.w));
    d.z = __ffma2_rn(m1, bz, az);
    return d;
}

// 1 / |d|
__device__ __forceinline__ float2 duo_inv_norm(const Duo3& d) {
    const float2 s = __ffma2_rn(d.z, d.z, __ffma2_rn(d.y, d.y, __fmul2_rn(d.x, d.x)));
    return make_float2(rsqrtf(s.x), rsqrtf(s.y));
}

// (1 / r_ij - mu) / sd
__device__ __forceinline__ float2 duo_feature(const DuoPos& q, const ushort2 ij, float mu, float isd) {
    const float2 g = duo_inv_norm(duo_diff(q.xy[ij.x], q.z[ij.x], q.xy[ij.y], q.z[ij.y]));
    return __fmul2_rn(__fadd2_rn(g, make_float2(-mu, -mu)), make_float2(isd, isd));
}

// sum over j != k of gam_p(k,j) (x_k - x_j) / r_kj^3, i.e. minus the
// derivative of sum_p gam_p g_p with respect to x_k
__device__ __forceinline__ float3 atom_force(int k, const float* xs, const float* gam, int N) {
    const float xk = xs[k], yk = xs[kXs + k], zk = xs[2 * kXs + k];
    float fx = 0.0f, fy = 0.0f, fz = 0.0f;
    for (int j = 0; j < N; ++j) {
        if (j == k) continue;
        const int p = k < j ? pair_id(k, j, N) : pair_id(j, k, N);
        const float dx = xk - xs[j], dy = yk - xs[kXs + j], dz = zk - xs[2 * kXs + j];
        const float ir = rsqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
        const float c = gam[p] * ir * ir * ir;
        fx = fmaf(c, dx, fx);
        fy = fmaf(c, dy, fy);
        fz = fmaf(c, dz, fz);
    }
    return make_float3(fx, fy, fz);
}

// Molecules of up to kGammaMatrixMax atoms use a symmetric N x N shared-
// memory matrix c_ij = gam_ij / r_ij^3 per configuration, filled by one pass
// over the pairs (one rsqrt per pair), so that the force of atom k is the
// plain row sum F_k = sum_j c_kj (x_k - x_j).  Larger molecules keep gam per
// pair and use atom_force.
constexpr int kGammaMatrixMax = 128;

__host__ __device__ __forceinline__ bool gamma_matrix(int N) { return N <= kGammaMatrixMax; }
__host__ __device__ __forceinline__ int gamma_stride(int N) { return N | 1; }

// gam_p = de/dg_p of one configuration (whole block)
__device__ __forceinline__ void load_gamma(const __nv_bfloat16* __restrict__ ga_row, const float* __restrict__ inv_sd,
                                           int P, float* gam) {
    for (int p = threadIdx.x; p < P; p += blockDim.x) gam[p] = __bfloat162float(ga_row[p]) * inv_sd[p];
}

// The symmetric matrix c_ij = gam_ij / r_ij^3 of two configurations (odd row
// stride: rows of consecutive atoms start on distinct bank pairs), one 1/r per
// pair, from their de/da rows ga[0..P) and ga[Pp..Pp + P).
__host__ __device__ __forceinline__ size_t duo_gamma_bytes(int N) { return 8 * (size_t)N * gamma_stride(N); }

__device__ __forceinline__ void duo_gamma(const DuoPos& q, const __nv_bfloat16* ga, const ushort2* __restrict__ pairs,
                                          const float* __restrict__ inv_sd, int P, int Pp, int N, float2* gam) {
    const int S = gamma_stride(N);
#pragma unroll 4
    for (int p = threadIdx.x; p < P; p += blockDim.x) {
        const ushort2 ij = pairs[p];
        const float isd = inv_sd[p];
        const float2 g = make_float2(__bfloat162float(ga[p]), __bfloat162float(ga[Pp + p]));
        const float2 ir = duo_inv_norm(duo_diff(q.xy[ij.x], q.z[ij.x], q.xy[ij.y], q.z[ij.y]));
        const float2 c = __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(g, make_float2(isd, isd)), ir), ir), ir);
        gam[ij.x * S + ij.y] = c;
        gam[ij.y * S + ij.x] = c;
    }
}

// sum over j0 <= j < j1 of c_kj (x_k - x_j); lanes of consecutive k read x_j as broadcasts
__device__ __forceinline__ Duo3 duo_force(int k, const DuoPos& q, const float2* gam, int N, int j0, int j1) {
    const float4 kxy = q.xy[k];
    const float2 kz = q.z[k];
    const float2* row = gam + k * gamma_stride(N);
    const float2 zero = make_float2(0.0f, 0.0f);
    Duo3 f{zero, zero, zero};
#pragma unroll 5
    for (int j = j0; j < j1; ++j) {
        const float2 c = row[j];
        const Duo3 d = duo_diff(kxy, kz, q.xy[j], q.z[j]);
        f.x = __ffma2_rn(c, d.x, f.x);
        f.y = __ffma2_rn(c, d.y, f.y);
        f.z = __ffma2_rn(c, d.z, f.z);
    }
    return f;
}

// Block size and the blocks per SM it is compiled for: as many threads as a row
// split over up to eight keeps busy.  Small molecules in 384 threads leave
// most idle at the barriers (65536 configurations of 9 atoms, whole call: 210
// us, in 64 threads 131; 16384 of 22: 102 and, in 128, 87).  Three blocks' shared
// memory fits an SM up to 82 atoms; 256 threads with 85 registers then beat 384
// with 56 (75 atoms, 65536 configurations: forces 475 -> 432 us), and past it
// 384 at two blocks do (16384 of 97 atoms, whole call: 456 -> 391 us).
constexpr int kDuoPartsMax = 8;
constexpr int kDuoElems = 2;  // coordinates per thread: 6 N <= 2 threads

__host__ __device__ __forceinline__ int duo_threads(int N) { return N <= 21 ? 64 : N <= 42 ? 128 : N <= 82 ? 256 : 384; }
// The loss and MD step kernels run 384 from 43 atoms on: their work beside the
// pairs uses the warps (loss of 2048 samples of 75 atoms: 44 us in 384 threads,
// 49 in 256; a step of 16384 replicas of 75, H = 64: 286 and 294).
__host__ __device__ __forceinline__ int duo_threads_wide(int N) { return N <= 42 ? duo_threads(N) : 384; }
__host__ __device__ constexpr int duo_blocks(int threads) { return threads == 384 ? 2 : threads == 256 ? 3 : 1024 / threads; }
static_assert(6 * 21 <= kDuoElems * 64 && 6 * 42 <= kDuoElems * 128 && 6 * 82 <= kDuoElems * 256 &&
                  6 * kGammaMatrixMax <= kDuoElems * 384, "");
__host__ __device__ __forceinline__ int duo_parts(int N) {
    return duo_threads(N) / N < kDuoPartsMax ? duo_threads(N) / N : kDuoPartsMax;
}

// queue the copies of two rows of Pp BF16 values (16-byte multiples) to dst
__device__ __forceinline__ void duo_fetch_rows(const __nv_bfloat16* ga, int m0, int m1, int Pp, unsigned char* dst) {
    const int n = Pp / 8;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) {
        const __nv_bfloat16* src = ga + (size_t)(t < n ? m0 : m1) * Pp + 8 * (t < n ? t : t - n);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * t), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// the row sums of both configurations, each row in `parts` consecutive pieces:
// part[h][b][k][c], parts N <= blockDim.x
__device__ __forceinline__ void duo_force_parts(const DuoPos& q, const float2* gam, int N, int parts, float* part) {
    const int len = (N + parts - 1) / parts;
    const int h = threadIdx.x / N, k = threadIdx.x - h * N;
    if (h >= parts) return;
    const int j0 = min(h * len, N), j1 = min(N, j0 + len);
    const Duo3 s = duo_force(k, q, gam, N, j0, j1);
    float* o = part + (size_t)h * 6 * N + 3 * k;
    o[0] = s.x.x;
    o[1] = s.y.x;
    o[2] = s.z.x;
    o += 3 * N;
    o[0] = s.x.y;
    o[1] = s.y.y;
    o[2] = s.z.y;
}
__device__ __forceinline__ float duo_force_sum(const float* part, int N, int parts, int t) {
    float v = part[t];
    for (int h = 1; h < parts; ++h) v += part[h * 6 * N + t];
    return v;
}

// ------------------------------------------------ pair passes of the MD step kernel
// past gamma_matrix(N).  Positions sit in shared memory as float4 (x, y, z, 0).

__host__ __device__ __forceinline__ size_t step_pos_bytes(int N) { return 16 * (size_t)(N + 1); }

__device__ __forceinline__ float inv_dist4(const float4 a, const float4 b) {
    const float dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    return rsqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
}

// positions of one replica from the population layout [6][Np] (whole block)
__device__ __forceinline__ void load_pos4(const float* st, int N, int Np, float4* xs4) {
    for (int i = threadIdx.x; i < N; i += blockDim.x)
        xs4[i] = make_float4(st[i], st[Np + i], st[2 * Np + i], 0.0f);
}

// features of the configuration in xs4 (whole block)
__device__ __forceinline__ void pass_features(const float4* xs4, const ushort2* pij, int P, int Pp,
                                              const float* mu, const float* inv_sd, __nv_bfloat16* a_row) {
#pragma unroll 4
    for (int p = threadIdx.x; p < Pp; p += blockDim.x) {
        float v = 0.0f;
        if (p < P) {
            const ushort2 ij = pij[p];
            v = (inv_dist4(xs4[ij.x], xs4[ij.y]) - mu[p]) * inv_sd[p];
        }
        a_row[p] = __float2bfloat16(v);
    }
}

// sum over j != k of gam_kj (x_k - x_j) / r_kj^3 (atom_force on xs4)
__device__ __forceinline__ float3 atom_force4(int k, const float4* xs4, const float* gam, int N) {
    const float4 xk = xs4[k];
    float fx = 0.0f, fy = 0.0f, fz = 0.0f;
    for (int j = 0; j < N; ++j) {
        if (j == k) continue;
        const int p = k < j ? pair_id(k, j, N) : pair_id(j, k, N);
        const float4 xj = xs4[j];
        const float dx = xk.x - xj.x, dy = xk.y - xj.y, dz = xk.z - xj.z;
        const float ir = rsqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
        const float c = gam[p] * ir * ir * ir;
        fx = fmaf(c, dx, fx);
        fy = fmaf(c, dy, fy);
        fz = fmaf(c, dz, fz);
    }
    return make_float3(fx, fy, fz);
}

// normalised energy e = b3 + sum of the layer-2 partial sums
__device__ __forceinline__ double head_energy(const float* part, int nparts, int m, const float* b3) {
    double e = (double)*b3;
    for (int q = 0; q < nparts; ++q) e += (double)part[(size_t)m * nparts + q];
    return e;
}

// sum of v over the block (blockDim.x a multiple of 32, <= 1024); every
// thread receives the total.  red: >= 32 doubles of shared memory.
__device__ __forceinline__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[w] = v;
    __syncthreads();
    double t = 0.0;
    for (int i = 0; i < nw; ++i) t += red[i];
    return t;
}

}  // namespace pamd
