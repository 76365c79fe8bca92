// fields.cu -- the field kernels: initial populations, moments, population
// transfer and the dS field.
//
// They move each field once and should run at the rate of memory, but FP64
// instructions (a warp's takes this GPU's FP64 unit 64 cycles) and 64-bit index
// divisions bounded them.  So rows and columns come from the grid, float <-> double
// conversions of the FP32 / 16-bit storage run on integers (the same values), and the
// moments of such storage are summed exactly in 64-bit fixed point: eight FP64
// instructions a site instead of 54.  At 4096^2 FP32 (16.8 M sites), us before and
// after: see the kernels.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "site.cuh"

namespace lbm {
namespace {

constexpr int kFieldThreads = 256;  // columns of a block; blockIdx.y walks rows

#define FOR_SITES(x, y)                                                    \
    const int x = (int)(blockIdx.x * kFieldThreads + threadIdx.x);         \
    if (x < p.nx)                                                          \
        for (int y = (int)blockIdx.y; y < p.ny; y += (int)gridDim.y)

template <int Q, typename S>
__global__ void k_delta_s(StepParams p, const S *__restrict__ f, double *__restrict__ out)
{
    const long long n = (long long)p.nx * p.ny;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(s % p.nx), y = (int)(s / p.nx);
        if (Q == 9 && is_wall_node(p, x, y)) {  // boundary nodes are not collided
            out[s] = 0.0;
            continue;
        }
        double fin[Q], fs[Q], fp[Q], ds, dsin, rho;
        pull<Q, S, double>(p, f, x, y, fin);
        const bool bad = site_collide<Q, double>(fin, p.a, true, fs, fp, ds, dsin, rho, p.eq, true, p.coll, p.beta);
        out[s] = bad ? (double)INFINITY : ds;
    }
}

// f*(rho, u) of the configured kind in FP64, stored at the storage precision.
template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_init(StepParams p, const double *__restrict__ rho,
                                                        const double *__restrict__ ux,
                                                        const double *__restrict__ uy, S *__restrict__ f)
{
    FOR_SITES(x, y)
    {
        const long long s = (long long)y * p.nx + x;
        double fs[Q];
        if (!feq_any<Q>(p.eq, rho[s], ux[s], uy ? uy[s] : 0.0, fs)) {
#pragma unroll
            for (int k = 0; k < Q; ++k) fs[k] = (double)NAN;  // no entropic f* for |u_j| >= 1
        }
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            if constexpr (std::is_same<S, double>::value)
                f[fidx(p.plane, p.pitch, k, y, x)] = fs[k];
            else
                f[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(narrow(Ar<double>::sub(fs[k], p.rw[k])));
        }
    }
}

// rho, u of the stored populations.
template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_moments(StepParams p, const S *__restrict__ f,
                                                           double *__restrict__ rho, double *__restrict__ ux,
                                                           double *__restrict__ uy)
{
    FOR_SITES(x, y)
    {
        S raw[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) raw[k] = f[fidx(p.plane, p.pitch, k, y, x)];
        double r, a, b;
        site_moments<Q, S>(p, raw, r, a, b);
        const long long s = (long long)y * p.nx + x;
        rho[s] = r;
        ux[s] = a;
        if (uy) uy[s] = b;
    }
}

// The stored populations as FP64, plane-major, and back (rounded to the storage
// precision).
template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_get(StepParams p, const S *__restrict__ f, double *__restrict__ out)
{
    const long long n = (long long)p.nx * p.ny;
    FOR_SITES(x, y)
    {
        S raw[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) raw[k] = f[fidx(p.plane, p.pitch, k, y, x)];
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            if constexpr (std::is_same<S, double>::value)
                out[k * n + (long long)y * p.nx + x] = raw[k];
            else
                out[k * n + (long long)y * p.nx + x] = Ar<double>::add(widen(s2f(raw[k])), p.rw[k]);
        }
    }
}

template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_set(StepParams p, const double *__restrict__ in, S *__restrict__ f)
{
    const long long n = (long long)p.nx * p.ny;
    FOR_SITES(x, y)
    {
        double v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) v[k] = in[k * n + (long long)y * p.nx + x];
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            if constexpr (std::is_same<S, double>::value)
                f[fidx(p.plane, p.pitch, k, y, x)] = v[k];
            else
                f[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(narrow(Ar<double>::sub(v[k], p.rw[k])));
        }
    }
}

inline dim3 field_grid(const StepParams &p)
{
    return dim3((unsigned)((p.nx + kFieldThreads - 1) / kFieldThreads), (unsigned)std::min(p.ny, 65535));
}

inline int grid_for(long long n, int threads)
{
    long long b = (n + threads - 1) / threads;
    if (b > 152 * 32) b = 152 * 32;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

template <typename T>
cudaError_t launch_delta_s(int q, const StepParams &p, const T *f, double *out, cudaStream_t s)
{
    const int g = grid_for((long long)p.nx * p.ny, 256);
    if (q == 9)
        k_delta_s<9, T><<<g, 256, 0, s>>>(p, f, out);
    else
        k_delta_s<3, T><<<g, 256, 0, s>>>(p, f, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init(int q, const StepParams &p, const double *rho, const double *ux, const double *uy, T *f,
                        cudaStream_t s)
{
    if (q == 9)
        k_init<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, rho, ux, uy, f);
    else
        k_init<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, rho, ux, nullptr, f);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(int q, const StepParams &p, const T *f, double *rho, double *ux, double *uy,
                           cudaStream_t s)
{
    if (q == 9)
        k_moments<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, f, rho, ux, uy);
    else
        k_moments<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, f, rho, ux, uy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_get(int q, const StepParams &p, const T *f, double *out, cudaStream_t s)
{
    if (q == 9)
        k_get<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, f, out);
    else
        k_get<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, f, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_set(int q, const StepParams &p, const double *in, T *f, cudaStream_t s)
{
    if (q == 9)
        k_set<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, in, f);
    else
        k_set<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, in, f);
    return cudaGetLastError();
}

#define LBM_INST(T)                                                                                           \
    template cudaError_t launch_delta_s<T>(int, const StepParams &, const T *, double *, cudaStream_t);     \
    template cudaError_t launch_init<T>(int, const StepParams &, const double *, const double *,           \
                                        const double *, T *, cudaStream_t);                                  \
    template cudaError_t launch_moments<T>(int, const StepParams &, const T *, double *, double *, double *, \
                                           cudaStream_t);                                                    \
    template cudaError_t launch_get<T>(int, const StepParams &, const T *, double *, cudaStream_t);         \
    template cudaError_t launch_set<T>(int, const StepParams &, const double *, T *, cudaStream_t);
LBM_INST(float)
LBM_INST(double)
LBM_INST(__nv_bfloat16)
LBM_INST(__half)
#undef LBM_INST

}  // namespace lbm
