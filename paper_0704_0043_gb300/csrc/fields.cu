// fields.cu -- the field kernels: initial populations, moments, population
// transfer and the dS field.
//
// They move each field once and should run at the rate of memory, but FP64
// instructions (a warp's takes this GPU's FP64 unit 64 cycles) and 64-bit index
// divisions bounded them.  So a site's row is its index times a reciprocal of nx (every
// lane has a site, whatever the lattice's width), float <-> double
// conversions of the FP32 / 16-bit storage run on integers (the same values), and the
// moments of such storage are summed exactly in 64-bit fixed point: eight FP64
// instructions a site instead of 54.  4096^2 FP32 (16.8 M sites): moments 1621 -> 239 us;
// 2048^2: set 149 -> 76 us.  4096^2 BF16: get 592 -> 294 us.  A block per 256 columns
// of a row took ten times as long on lattices a few columns wide (2 x 500000: init
// 1913 us, now 157).
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "site.cuh"

namespace lbm {
namespace {

constexpr int kFieldThreads = 128;  // (256: a 100 x 100 get 1.3 us longer, on too few SMs; large lattices alike)

// s / nx for 0 <= s < 2^31 by one multiplication (Granlund and Montgomery, PLDI 1994):
// with 2^(l - 1) < nx <= 2^l and m = ceil(2^(31 + l) / nx) < 2^32 the quotient is
// floor(m s / 2^(31 + l)).  nx = 1 by itself.
struct RowOf {
    unsigned m = 0;
    int shift = 0;  // l - 1; nx = 1: -1
    explicit RowOf(int nx)
    {
        int l = 0;
        while ((1ll << l) < nx) ++l;
        shift = l - 1;
        if (l > 0) m = (unsigned)(((1ull << (31 + l)) + (unsigned)nx - 1) / (unsigned)nx);
    }
    __host__ __device__ int operator()(int s) const
    {
        return shift < 0 ? s : (int)(((unsigned long long)m * (unsigned)s) >> 32 >> shift);
    }
};

// The thread's site s, (x, y); the grid covers the lattice.
#define FOR_SITE(s, x, y)                                                     \
    const long long s = blockIdx.x * (long long)kFieldThreads + threadIdx.x; \
    if (s >= (long long)p.nx * p.ny) return;                                  \
    const int y = Q == 3 ? 0 : row((int)s), x = (int)s - y * p.nx;

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
__global__ void __launch_bounds__(kFieldThreads) k_init(StepParams p, RowOf row, const double *__restrict__ rho,
                                                        const double *__restrict__ ux,
                                                        const double *__restrict__ uy, S *__restrict__ f)
{
    FOR_SITE(s, x, y)
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

// rho, u of the stored populations.
template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_moments(StepParams p, RowOf row, const S *__restrict__ f,
                                                           double *__restrict__ rho, double *__restrict__ ux,
                                                           double *__restrict__ uy)
{
    FOR_SITE(s, x, y)
    S raw[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) raw[k] = f[fidx(p.plane, p.pitch, k, y, x)];
    double r, a, b;
    site_moments<Q, S>(p, raw, r, a, b);
    rho[s] = r;
    ux[s] = a;
    if (uy) uy[s] = b;
}

// The stored populations as FP64, plane-major, and back (rounded to the storage
// precision).
template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_get(StepParams p, RowOf row, const S *__restrict__ f,
                                                       double *__restrict__ out)
{
    const long long n = (long long)p.nx * p.ny;
    FOR_SITE(s, x, y)
    S raw[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) raw[k] = f[fidx(p.plane, p.pitch, k, y, x)];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        if constexpr (std::is_same<S, double>::value)
            out[k * n + s] = raw[k];
        else
            out[k * n + s] = Ar<double>::add(widen(s2f(raw[k])), p.rw[k]);
    }
}

template <int Q, typename S>
__global__ void __launch_bounds__(kFieldThreads) k_set(StepParams p, RowOf row, const double *__restrict__ in,
                                                       S *__restrict__ f)
{
    const long long n = (long long)p.nx * p.ny;
    FOR_SITE(s, x, y)
    double v[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) v[k] = in[k * n + s];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        if constexpr (std::is_same<S, double>::value)
            f[fidx(p.plane, p.pitch, k, y, x)] = v[k];
        else
            f[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(narrow(Ar<double>::sub(v[k], p.rw[k])));
    }
}

inline unsigned field_grid(const StepParams &p)
{
    return (unsigned)(((long long)p.nx * p.ny + kFieldThreads - 1) / kFieldThreads);
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
        k_init<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), rho, ux, uy, f);
    else
        k_init<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), rho, ux, nullptr, f);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_moments(int q, const StepParams &p, const T *f, double *rho, double *ux, double *uy,
                           cudaStream_t s)
{
    if (q == 9)
        k_moments<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), f, rho, ux, uy);
    else
        k_moments<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), f, rho, ux, uy);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_get(int q, const StepParams &p, const T *f, double *out, cudaStream_t s)
{
    if (q == 9)
        k_get<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), f, out);
    else
        k_get<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), f, out);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_set(int q, const StepParams &p, const double *in, T *f, cudaStream_t s)
{
    if (q == 9)
        k_set<9, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), in, f);
    else
        k_set<3, T><<<field_grid(p), kFieldThreads, 0, s>>>(p, RowOf(p.nx), in, f);
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
