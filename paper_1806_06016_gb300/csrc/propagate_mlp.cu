// propagate_mlp.cu -- BAOAB Langevin steps of a population whose forces and
// energies come from the MLP energy surrogate.
//
// The exact-force propagate kernel keeps each replica in shared memory for
// all theta steps; here every force evaluation is a batch of tensor-core
// GEMMs over the whole population, so the state stays in global memory and
// one step is five launches: this kernel (finish the previous step with its
// closing half kick, then B A O A of the next one and the features of the new
// positions) and the four GEMMs.  Inside a graph capture (pamd_anneal) the
// theta steps become one WHILE node whose body is those five launches and a
// one-thread counter kernel.  The update arithmetic and the Philox noise
// stream are those of the exact propagate kernel (same key, counter and
// purpose), so that the two force fields can be compared on identical noise.
#include <map>
#include <mutex>
#include <tuple>

#include "mlp_device.cuh"
#include "pamd_device.cuh"

namespace pamd {

namespace {

constexpr int kStepThreads = 256;
static_assert(PAMD_MAX_ATOMS <= kStepThreads, "one atom per thread in the update");

// Pieces each atom's force sum is split into (consecutive parts of its row,
// added in order), up to three.
__host__ __device__ __forceinline__ int step_parts(int N) { return 3 * N <= 256 ? 3 : 2; }

// Byte offsets of the dynamic shared memory for two replicas at a time: the
// matrix c_ij, their de/da rows, positions, partial force sums and state rows.
struct StepSmem {
    size_t ga, pos, part, state, total;
};

__host__ __device__ __forceinline__ StepSmem step_smem(int N, int Np, int Pp) {
    auto up = [](size_t b) { return (b + 15) & ~size_t(15); };
    StepSmem L{};
    L.ga = up(duo_gamma_bytes(N));
    L.pos = L.ga + 4 * (size_t)Pp;
    L.part = L.pos + duo_pos_bytes(N);
    L.state = L.part + up(24 * (size_t)N * step_parts(N));
    L.total = L.state + 48 * (size_t)Np;
    return L;
}

// queue the copies of two replicas' states [6][Np] (16-byte multiples)
__device__ __forceinline__ void fetch_states(const float* state, long long k0, long long k1, int Np, unsigned char* dst) {
    const int n = 6 * Np / 4;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    for (int t = threadIdx.x; t < 2 * n; t += blockDim.x) {
        const float* src = state + (size_t)(t < n ? k0 : k1) * 6 * Np + 4 * (t < n ? t : t - n);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * t), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

struct StepAtom {
    float x, y, z, vx, vy, vz;
};

// mode 1 of one atom: closing B of the previous step (step_index > 0), B A O A
__device__ __forceinline__ void advance_atom(const MlpStepParams& p, int i, long long k, uint32_t step, bool close,
                                             const float3 f, StepAtom& s) {
    const float im = 1.0f / p.masses[i];
    if (close) {
        s.vx = fmaf(p.hdt * im, f.x, s.vx);
        s.vy = fmaf(p.hdt * im, f.y, s.vy);
        s.vz = fmaf(p.hdt * im, f.z, s.vz);
    }
    s.vx = fmaf(p.hdt * im, f.x, s.vx);  // B
    s.vy = fmaf(p.hdt * im, f.y, s.vy);
    s.vz = fmaf(p.hdt * im, f.z, s.vz);
    s.x = fmaf(p.hdt, s.vx, s.x);  // A
    s.y = fmaf(p.hdt, s.vy, s.y);
    s.z = fmaf(p.hdt, s.vz, s.z);
    const float sd = p.c2kT * sqrtf(im);  // O
    const float3 n = normal3_fast(p.seed, (uint32_t)i, (uint32_t)k, step, p.purpose_mol);
    s.vx = fmaf(p.c1, s.vx, sd * n.x);
    s.vy = fmaf(p.c1, s.vy, sd * n.y);
    s.vz = fmaf(p.c1, s.vz, sd * n.z);
    s.x = fmaf(p.hdt, s.vx, s.x);  // A
    s.y = fmaf(p.hdt, s.vy, s.y);
    s.z = fmaf(p.hdt, s.vz, s.z);
}

// mode 2 of one atom: closing B of the last step (theta > 0), forces out
__device__ __forceinline__ void finish_atom(const MlpStepParams& p, int i, long long k, const float3 f, StepAtom& s) {
    const float im = 1.0f / p.masses[i];
    if (p.theta > 0) {
        s.vx = fmaf(p.hdt * im, f.x, s.vx);
        s.vy = fmaf(p.hdt * im, f.y, s.vy);
        s.vz = fmaf(p.hdt * im, f.z, s.vz);
    }
    if (p.fout) {
        float* fo = p.fout + (size_t)k * 3 * p.Np;
        fo[i] = f.x;
        fo[p.Np + i] = f.y;
        fo[2 * p.Np + i] = f.z;
    }
}

// mode 2 of one replica by one warp: energy, kinetic energy and radius of
// gyration from its final state, row c < 6 of get(c, atom).  FP64 instructions
// bound it (a warp's takes 20 clocks of its SM however few lanes it has), so
// the four sums share their reduction, each in a quarter of the lanes, and
// the three divisions are one.
// 16384 replicas of 75 atoms, the whole launch: 234 us (five sums over the
// block, which every one of its warps adds up, for each replica: 1261).
template <typename F>
__device__ __forceinline__ void finish_replica(const MlpStepParams& p, long long k, F get) {
    const int N = p.N, lane = threadIdx.x & 31;
    const unsigned all = 0xffffffffu;
    double ek = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    for (int i = lane; i < N; i += 32) {
        sx += (double)get(0, i);
        sy += (double)get(1, i);
        sz += (double)get(2, i);
        const double vx = get(3, i), vy = get(4, i), vz = get(5, i);
        ek += 0.5 * (double)p.masses[i] * (vx * vx + vy * vy + vz * vz);
    }
    // lanes 0..7 end with ek, 8..15 sx, 16..23 sy, 24..31 sz
    const bool hi = lane & 16, mid = lane & 8;
    const double a0 = (hi ? sy : ek) + __shfl_xor_sync(all, hi ? ek : sy, 16);
    const double a1 = (hi ? sz : sx) + __shfl_xor_sync(all, hi ? sx : sz, 16);
    double v = (mid ? a1 : a0) + __shfl_xor_sync(all, mid ? a0 : a1, 8);
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(all, v, o);
    const double mean = v / N;
    const double cx = __shfl_sync(all, mean, 8), cy = __shfl_sync(all, mean, 16), cz = __shfl_sync(all, mean, 24);
    double r2 = 0.0;
    for (int i = lane; i < N; i += 32) {
        const double dx = (double)get(0, i) - cx, dy = (double)get(1, i) - cy, dz = (double)get(2, i) - cz;
        r2 += dx * dx + dy * dy + dz * dz;
    }
    for (int o = 16; o > 0; o >>= 1) r2 += __shfl_xor_sync(all, r2, o);
    if (lane == 0) {
        const double E = p.sigma_E * head_energy(p.part, p.nparts, (int)k, p.b3) + p.mu_E;
        p.E[k] = E;
        p.ke[k] = v;
        p.rg[k] = sqrt(r2 / N);
        if (!isfinite(E) && atomicCAS(&p.status[0], 0, PAMD_ENONFINITE) == 0) p.status[1] = (int)k;
    }
}

// Molecules with gamma_matrix(N): two replicas at a time per block, in the
// manner of the force kernel.  Both replicas' pair passes share each read and
// packed instruction; the next two de/da rows arrive while the rows are
// summed, the next states while the features are written.
// Bound by shared-memory wavefronts (67 % of the pipe's rate), reads of the pair
// tables, of which the first level cache holds a third beside three blocks'
// shared memory, and the barriers.  16384 replicas of 75 atoms: 188 us a step
// and 234 the last launch (one replica at a time with the tables in shared
// memory: 231 us a launch on average); 8192 of 97, whole step: 402 -> 344 us.
template <int T>
__global__ void __launch_bounds__(T, T == 384 ? 3 : 1024 / T) mlp_step_duo_kernel(const MlpStepParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int N = p.N, Np = p.Np, parts = step_parts(N);
    const StepSmem L = step_smem(N, Np, p.Pp);
    float2* gam = reinterpret_cast<float2*>(sm);
    const __nv_bfloat16* ga = reinterpret_cast<const __nv_bfloat16*>(sm + L.ga);
    const DuoPos q = duo_pos(sm + L.pos, N);
    float* part = reinterpret_cast<float*>(sm + L.part);
    float* ss = reinterpret_cast<float*>(sm + L.state);
    const int step_index = p.step_index_dev ? *p.step_index_dev : p.step_index;
    const uint32_t step = (p.dev_counters ? p.dev_counters[0] : 0u) + p.step0 + (uint32_t)step_index;
    const float sE = (float)p.sigma_E;
    const bool need_ga = p.mode != 0;
    const long long D = (p.R + 1) / 2;
    auto second = [&](long long d) { return 2 * d + 1 < p.R ? 2 * d + 1 : 2 * d; };
    long long d = blockIdx.x;
    if (d < D) {
        if (need_ga) duo_fetch_rows(p.ga, 2 * d, second(d), p.Pp, sm + L.ga);
        fetch_states(p.state, 2 * d, second(d), Np, sm + L.state);
    }
    for (int k = threadIdx.x; k < N; k += T) gam[k * gamma_stride(N) + k] = make_float2(0.0f, 0.0f);
    for (; d < D; d += gridDim.x) {
        const long long k0 = 2 * d, nd = d + gridDim.x;
        const bool two = k0 + 1 < p.R;
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncthreads();  // every thread's copies have landed; the last features have read q
        for (int t = threadIdx.x; t < 6 * N; t += T) {
            const int c = t / (2 * N), r = t - c * 2 * N, b = r >= N, i = r - N * b;
            q.put(b, i, c, ss[(6 * b + c) * Np + i]);
        }
        __syncthreads();
        const int b = threadIdx.x >= (unsigned)N, i = threadIdx.x - N * b;  // the update's replica and atom
        const bool mine = threadIdx.x < 2u * N && (b == 0 || two);
        if (need_ga) {
            duo_gamma(q, ga, p.pairs, p.inv_sd, p.P, p.Pp, N, gam);
            __syncthreads();
            if (nd < D) duo_fetch_rows(p.ga, 2 * nd, second(nd), p.Pp, sm + L.ga);
            duo_force_parts(q, gam, N, parts, part);
            __syncthreads();
            if (mine) {
                // F = -dE/dx of the current positions
                const float* o = part + 3 * N * b + 3 * i;
                float3 f = make_float3(o[0], o[1], o[2]);
                for (int h = 1; h < parts; ++h) {
                    f.x += o[6 * N * h];
                    f.y += o[6 * N * h + 1];
                    f.z += o[6 * N * h + 2];
                }
                f = make_float3(sE * f.x, sE * f.y, sE * f.z);
                float* sb = ss + 6 * b * Np;
                StepAtom s{sb[i], sb[Np + i], sb[2 * Np + i], sb[3 * Np + i], sb[4 * Np + i], sb[5 * Np + i]};
                float* st = p.state + (size_t)(k0 + b) * 6 * Np;
                if (p.mode == 1) {
                    advance_atom(p, i, k0 + b, step, step_index > 0, f, s);
                    q.put(b, i, 0, s.x);
                    q.put(b, i, 1, s.y);
                    q.put(b, i, 2, s.z);
                    st[i] = s.x;
                    st[Np + i] = s.y;
                    st[2 * Np + i] = s.z;
                } else {
                    finish_atom(p, i, k0 + b, f, s);
                    sb[3 * Np + i] = s.vx;
                    sb[4 * Np + i] = s.vy;
                    sb[5 * Np + i] = s.vz;
                }
                if (p.mode == 1 || p.theta > 0) {
                    st[3 * Np + i] = s.vx;
                    st[4 * Np + i] = s.vy;
                    st[5 * Np + i] = s.vz;
                }
            }
            __syncthreads();  // new positions complete in q, the states read
            if (p.mode == 2) {
                const int r = threadIdx.x >> 5;
                if (r <= (two ? 1 : 0)) finish_replica(p, k0 + r, [&](int c, int a) { return ss[(6 * r + c) * Np + a]; });
                __syncthreads();
            }
        }
        if (nd < D) fetch_states(p.state, 2 * nd, second(nd), Np, sm + L.state);
        if (p.mode == 2) continue;
        __nv_bfloat16* a = p.a + (size_t)k0 * p.Pp;
#pragma unroll 2
        for (int t = threadIdx.x; t < p.Pp; t += T) {
            float2 v = make_float2(0.0f, 0.0f);
            if (t < p.P) v = duo_feature(q, p.pairs[t], p.mu[t], p.inv_sd[t]);
            a[t] = __float2bfloat16(v.x);
            if (two) a[p.Pp + t] = __float2bfloat16(v.y);
        }
    }
}

// Larger molecules, one replica at a time: dynamic shared memory holds the
// positions (float4 per atom) and de/dg per pair.
size_t step_large_smem(int N, int Pp) { return step_pos_bytes(N) + 4 * (size_t)Pp; }

__global__ void __launch_bounds__(kStepThreads) mlp_step_large_kernel(const MlpStepParams p) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int N = p.N, Np = p.Np;
    float4* xs4 = reinterpret_cast<float4*>(sm);
    float* gam = reinterpret_cast<float*>(sm + step_pos_bytes(N));
    const int step_index = p.step_index_dev ? *p.step_index_dev : p.step_index;
    const uint32_t step = (p.dev_counters ? p.dev_counters[0] : 0u) + p.step0 + (uint32_t)step_index;
    const float sE = (float)p.sigma_E;
    for (long long k = blockIdx.x; k < p.R; k += gridDim.x) {
        float* st = p.state + (size_t)k * 6 * Np;
        __syncthreads();  // the previous replica is done with every buffer
        load_pos4(st, N, Np, xs4);
        if (p.mode != 0) {
            load_gamma(p.ga + (size_t)k * p.Pp, p.inv_sd, p.P, gam);
            __syncthreads();
            // forces of the current positions, F = -dE/dx (thread i: atom i)
            const int i = threadIdx.x;
            float3 f = make_float3(0.0f, 0.0f, 0.0f);
            if (i < N) f = atom_force4(i, xs4, gam, N);
            f = make_float3(sE * f.x, sE * f.y, sE * f.z);
            __syncthreads();  // every force sum has read xs4
            if (i < N) {
                const float4 x4 = xs4[i];
                StepAtom s{x4.x, x4.y, x4.z, st[3 * Np + i], st[4 * Np + i], st[5 * Np + i]};
                if (p.mode == 1) {
                    advance_atom(p, i, k, step, step_index > 0, f, s);
                    xs4[i] = make_float4(s.x, s.y, s.z, 0.0f);
                    st[i] = s.x;
                    st[Np + i] = s.y;
                    st[2 * Np + i] = s.z;
                } else {
                    finish_atom(p, i, k, f, s);
                }
                if (p.mode == 1 || p.theta > 0) {
                    st[3 * Np + i] = s.vx;
                    st[4 * Np + i] = s.vy;
                    st[5 * Np + i] = s.vz;
                }
            }
            if (p.mode == 2) {
                __syncthreads();  // the final state is in memory
                if (threadIdx.x < 32) finish_replica(p, k, [&](int c, int a) { return st[c * Np + a]; });
                continue;
            }
        }
        __syncthreads();  // positions complete in xs4
        pass_features(xs4, p.pairs, p.P, p.Pp, p.mu, p.inv_sd, p.a + (size_t)k * p.Pp);
    }
}

using StepKernel = void (*)(const MlpStepParams);
StepKernel step_kernel(int N, int* threads) {
    if (!gamma_matrix(N)) {
        *threads = kStepThreads;
        return mlp_step_large_kernel;
    }
    *threads = duo_threads_wide(N);
    return *threads == 64 ? mlp_step_duo_kernel<64> : *threads == 128 ? mlp_step_duo_kernel<128> : mlp_step_duo_kernel<384>;
}

// Last node of a captured MD loop's body: advance the step index and keep the
// WHILE node looping until theta steps have run.
__global__ void mlp_loop_next_kernel(cudaGraphConditionalHandle h, int* ctr, int theta) {
    const int c = *ctr + 1;
    *ctr = c;
    cudaGraphSetConditional(h, c < theta ? 1u : 0u);
}

}  // namespace

size_t mlp_step_smem(int N, int Np, int Pp) {
    return gamma_matrix(N) ? step_smem(N, Np, Pp).total : step_large_smem(N, Pp);
}

cudaError_t launch_mlp_step(const MlpStepParams& p, cudaStream_t s) {
    // the resident grid for this shared-memory size on the current device
    // (one block per resident slot; each block walks the replicas with
    // stride gridDim.x), looked up once per device, kernel and size
    static std::mutex mu;
    static std::map<std::tuple<int, StepKernel, size_t>, int> resident;
    int dev = 0, threads = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const StepKernel fn = step_kernel(p.N, &threads);
    const size_t smem = mlp_step_smem(p.N, p.Np, p.Pp);
    e = ensure_dyn_smem((const void*)fn, smem);
    if (e != cudaSuccess) return e;
    int grid_max = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        int& r = resident[std::make_tuple(dev, fn, smem)];
        if (r == 0) {
            int per_sm = 0, sms = 0;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
            if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            if (per_sm < 1) return cudaErrorInvalidConfiguration;
            r = per_sm * sms;
        }
        grid_max = r;
    }
    const long long units = gamma_matrix(p.N) ? (p.R + 1) / 2 : p.R;
    fn<<<(int)(units < grid_max ? units : grid_max), threads, smem, s>>>(p);
    return cudaGetLastError();
}

int mlp_propagate(pamd_mlp* m, float* state, double* E, double* ke, double* rg, float* fout,
                  const float* masses, int* status, const uint32_t* dev_counters, long long R,
                  int Np, int theta, double dt, double T, double gamma, unsigned long long seed,
                  uint32_t step0, uint32_t purpose_mol, cudaStream_t s, long long* launches) {
    if (m->broken) {
        set_last_error("force model unusable after an earlier CUDA error");
        return PAMD_ESTATE;
    }
    if (R > m->w.cap) {
        set_last_error("force model workspace smaller than the population");
        return PAMD_ESTATE;
    }
    MlpStepParams p{};
    p.state = state;
    p.E = E;
    p.ke = ke;
    p.rg = rg;
    p.fout = fout;
    p.masses = masses;
    p.status = status;
    p.dev_counters = dev_counters;
    p.R = R;
    p.N = m->N;
    p.Np = Np;
    p.P = m->P;
    p.Pp = m->Pp;
    p.nparts = m->nparts;
    p.theta = theta;
    p.ga = m->w.ga;
    p.part = m->w.part;
    p.mu = m->mu;
    p.inv_sd = m->inv_sd;
    p.pairs = m->pairs;
    p.a = m->w.a;
    p.b3 = m->params + m->ob3;
    p.sigma_E = m->sigma_E;
    p.mu_E = m->mu_E;
    p.hdt = (float)(0.5 * dt);
    const double c1 = std::exp(-gamma * dt);
    p.c1 = (float)c1;
    p.c2kT = (float)std::sqrt((1.0 - c1 * c1) * kBoltzmann * T);
    p.seed = seed;
    p.step0 = step0;
    p.purpose_mol = purpose_mol;
    const long long before = m->launches;
    int rc = PAMD_OK;
    auto step_launch = [&](int mode, int idx) {
        p.mode = mode;
        p.step_index = idx;
        const cudaError_t e = launch_mlp_step(p, s);
        m->launches += 1;
        if (e != cudaSuccess) {
            m->broken = true;
            set_last_error(std::string("surrogate step launch: ") + cudaGetErrorString(e));
            return PAMD_ECUDA;
        }
        return PAMD_OK;
    };
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t ce = cudaStreamIsCapturing(s, &cs);
    if (ce != cudaSuccess) {
        m->broken = true;
        set_last_error(std::string("surrogate propagate: ") + cudaGetErrorString(ce));
        return PAMD_ECUDA;
    }
    rc = step_launch(0, 0);
    if (!rc) rc = mlp_gemms(m, (int)R, true, s, status);
    if (cs == cudaStreamCaptureStatusActive && theta > 0) {
        // In a graph the theta steps are one WHILE node whose body (step
        // kernel, four GEMMs, loop counter) runs theta times; the step index
        // lives in device memory.
        const long long b0 = m->launches;
        if (!rc) rc = mlp_loop_captured(m, p, theta, (int)R, s, status);
        if (!rc) m->launches += (long long)(theta - 1) * (m->launches - b0);
    } else {
        for (int i = 0; i < theta && !rc; ++i) {
            rc = step_launch(1, i);
            if (!rc) rc = mlp_gemms(m, (int)R, true, s, status);
        }
    }
    if (!rc) rc = step_launch(2, 0);
    if (launches) *launches += m->launches - before;
    return rc;
}

int mlp_loop_captured(pamd_mlp* m, MlpStepParams p, int theta, int M, cudaStream_t s, int* status) {
    if (!m->loop_ctr || !m->body_stream) {
        set_last_error("surrogate loop captured without mlp_prepare_capture");
        return PAMD_ESTATE;
    }
    auto bad = [&](cudaError_t e, const char* what) {
        m->broken = true;
        set_last_error(std::string("surrogate loop capture (") + what + "): " + cudaGetErrorString(e));
        return PAMD_ECUDA;
    };
    cudaError_t e = cudaMemsetAsync(m->loop_ctr, 0, sizeof(int), s);
    if (e != cudaSuccess) return bad(e, "counter reset");
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    cudaGraph_t g = nullptr;
    const cudaGraphNode_t* deps = nullptr;
    size_t nd = 0;
    e = cudaStreamGetCaptureInfo(s, &st, nullptr, &g, &deps, nullptr, &nd);
    if (e != cudaSuccess) return bad(e, "capture info");
    cudaGraphConditionalHandle h{};
    e = cudaGraphConditionalHandleCreate(&h, g, 1u, cudaGraphCondAssignDefault);
    if (e != cudaSuccess) return bad(e, "conditional handle");
    cudaGraphNodeParams cp{};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = h;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t node = nullptr;
    e = cudaGraphAddNode(&node, g, deps, nullptr, nd, &cp);
    if (e != cudaSuccess) return bad(e, "WHILE node");
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    e = cudaStreamUpdateCaptureDependencies(s, &node, nullptr, 1, cudaStreamSetCaptureDependencies);
    if (e != cudaSuccess) return bad(e, "capture dependencies");
    cudaStream_t bs = m->body_stream;
    e = cudaStreamBeginCaptureToGraph(bs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return bad(e, "body capture");
    p.mode = 1;
    p.step_index = 0;
    p.step_index_dev = m->loop_ctr;
    int rc = PAMD_OK;
    e = launch_mlp_step(p, bs);
    m->launches += 1;
    if (e != cudaSuccess) rc = bad(e, "step kernel");
    if (!rc) rc = mlp_gemms(m, M, true, bs, status);
    if (!rc) {
        mlp_loop_next_kernel<<<1, 1, 0, bs>>>(h, m->loop_ctr, theta);
        m->launches += 1;
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = bad(e, "loop counter kernel");
    }
    cudaGraph_t out = nullptr;
    e = cudaStreamEndCapture(bs, &out);
    if (!rc && e != cudaSuccess) rc = bad(e, "end of body capture");
    return rc;
}

}  // namespace pamd
