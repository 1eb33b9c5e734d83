// state_io.cu -- replica records to and from the host's [R][N][3] FP64 arrays.
//
// The C interface passes positions, velocities and forces as [R][N][3]
// doubles; the device keeps records of coordinate planes, FP32 in the mixed
// mode.  The layout change, the widening or rounding and the finiteness check
// run here on a staging buffer, so that the host only copies contiguous
// arrays.  On one host core they took most of the call: 75 atoms, R = 8192,
// set_state and forces with the results rounded to FP32, 6.4 ms; now 1.6 ms, of
// which 0.2 ms is the force kernel and the rest 44 MB over the host link.
// Small populations stay with the host loops (convert_on_host in capi.cu).
#include "pamd_internal.h"

namespace pamd {

namespace {

constexpr int kIoThreads = 256;

int io_grid(long long n) {
    const long long b = (n + kIoThreads - 1) / kIoThreads;
    return (int)(b < 8192 ? b : 8192);
}

// One thread per (replica, padded atom): rows of x and v into the record;
// *bad is set when a value is not finite.
template <typename T>
__global__ void __launch_bounds__(kIoThreads) pack_kernel(const double* __restrict__ x, const double* __restrict__ v,
                                                          T* __restrict__ rec, long long n, int N, int Np, int* bad) {
    const long long total = n * Np;
    bool ok = true;
    for (long long t = (long long)blockIdx.x * kIoThreads + threadIdx.x; t < total;
         t += (long long)gridDim.x * kIoThreads) {
        const long long k = t / Np;
        const int i = (int)(t - k * Np);
        double a[6] = {0, 0, 0, 0, 0, 0};
        if (i < N) {
            const size_t e = ((size_t)k * N + i) * 3;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                a[c] = x[e + c];
                a[3 + c] = v[e + c];
                ok = ok && isfinite(a[c]) && isfinite(a[3 + c]);
            }
        }
        T* r = rec + (size_t)k * 6 * Np + i;
#pragma unroll
        for (int c = 0; c < 6; ++c) r[(size_t)c * Np] = (T)a[c];
    }
    if (!ok) *bad = 1;
}

// rows <- planes `first`..first + 2 of records of `planes` planes
template <typename T>
__global__ void __launch_bounds__(kIoThreads) unpack_kernel(const T* __restrict__ rec, double* __restrict__ rows,
                                                            long long n, int N, int Np, int planes, int first) {
    const long long total = n * N;
    for (long long t = (long long)blockIdx.x * kIoThreads + threadIdx.x; t < total;
         t += (long long)gridDim.x * kIoThreads) {
        const long long k = t / N;
        const int i = (int)(t - k * N);
        const T* r = rec + ((size_t)k * planes + first) * Np + i;
#pragma unroll
        for (int c = 0; c < 3; ++c) rows[(size_t)t * 3 + c] = (double)r[(size_t)c * Np];
    }
}

}  // namespace

cudaError_t launch_pack_state(const double* x, const double* v, void* rec, long long n, int N, int Np, bool f64, int* bad,
                              cudaStream_t s) {
    if (f64)
        pack_kernel<double><<<io_grid(n * Np), kIoThreads, 0, s>>>(x, v, (double*)rec, n, N, Np, bad);
    else
        pack_kernel<float><<<io_grid(n * Np), kIoThreads, 0, s>>>(x, v, (float*)rec, n, N, Np, bad);
    return cudaGetLastError();
}

cudaError_t launch_unpack_rows(const void* rec, double* rows, long long n, int N, int Np, int planes, int first, bool f64,
                               cudaStream_t s) {
    if (f64)
        unpack_kernel<double><<<io_grid(n * N), kIoThreads, 0, s>>>((const double*)rec, rows, n, N, Np, planes, first);
    else
        unpack_kernel<float><<<io_grid(n * N), kIoThreads, 0, s>>>((const float*)rec, rows, n, N, Np, planes, first);
    return cudaGetLastError();
}

}  // namespace pamd
