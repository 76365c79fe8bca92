// step_cluster.cu -- many limited LBGK steps of a very small lattice by one
// thread-block cluster, the populations held in its shared memory.
//
// What bounds a step of a lattice of a few ten thousand sites is latency: with
// the populations in L2 (step_resident.cu) a step's loads, the fence before the grid
// barrier, the barrier's counter and its polls are about 6 us whatever the size.
// A cluster of 16 blocks has a hardware barrier and reads and writes its
// blocks' shared memory, so here each block keeps a band of rows (D1Q3: of sites)
// of both population buffers, with the two edge rows of each neighbouring band: a
// block stores its edge rows into its neighbours' copies as well, and every pull of
// the next step is local.  Two rows, because the median of an edge site needs dS one
// row outside the band, which the block evaluates itself when such a median is
// formed (rare), so a step has one cluster barrier.  Such sites are finished behind a
// block barrier (a thread keeps the first of its own and evaluates others again).
// The step's sums are formed while the barrier completes and recorded one step later
// by a warp of the first block.  Measured on the 100 x 100 cavity with boundary nodes
// and the median filter: 3.8 us a step against 6.3 us in L2 and 16 us launch by launch.
// With Ehrenfests' steps (their selection needs two more barriers), in FP64 (16 SMs
// have too few FP64 units) and on tubes the resident kernel is as fast or faster.
// The per-site operations are those of the other kernels: the populations are the
// same bit for bit.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "resident.cuh"
#include "select.cuh"
#include "site.cuh"

namespace lbm {
namespace {

namespace cg = cooperative_groups;

constexpr int kCluThreads = kFinThreads;
constexpr int kCluWarps = kCluThreads / 32;
constexpr int kCluMax = 16;     // blocks of the cluster (more than 8 is opt-in)
constexpr int kCluSlots = 4;    // steps whose sums are kept

__device__ __forceinline__ void cluster_arrive()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_barrier()
{
    cluster_arrive();
    cluster_wait();
}

struct CluShared {
    BlockAcc<kCluWarps, float> acc[2];  // steps of each parity
    double fw[2][9];                    // diffusive wall: f*(1, u_wall) of the resting walls and of the lid
    ResRow rows[kCluSlots][kCluMax];    // the first block's: every block's sums
};

// A block's band of the lattice (rows of w = nx sites), and where a population
// lies.  Local row r of the band is lattice row first + r - 2; rows 0, 1 and rows + 2, rows + 3 are the neighbours'.
struct Band {
    float *f;        // [2][9][hs][w]
    float *ds;       // [hs][ldd], a column to the left and right
    int n, w, hs, ldd, rank, first, rows;
    bool wrap, wrapx;  // the rows, the columns wrap
    int below, above, below_rows;  // neighbouring blocks (-1: none)

    static __device__ __forceinline__ int dr(int k) { return Lat<9>::cy(k); }
    static __device__ __forceinline__ int dc(int k) { return Lat<9>::cx(k); }
    __device__ __forceinline__ int first_of(int r) const { return r * n / kCluMax; }
    __device__ __forceinline__ int owner(int row) const  // the block whose band holds the row
    {
        int r = row * kCluMax / n;
        while (row < first_of(r)) --r;
        while (row >= first_of(r + 1)) ++r;
        return r;
    }
    __device__ __forceinline__ int plane() const { return hs * w; }
    __device__ __forceinline__ int at(int b, int r, int x) const { return (b * 9 * hs + r) * w + x; }  // population 0
    template <typename V>
    __device__ __forceinline__ V *in_block(V *p, int r) const
    {
        return cg::this_cluster().map_shared_rank(p, r);
    }

    // Offset, from population 0 of a site (lattice row j, column x), of the source of
    // population k that arrives there (see pull_raw).  `wall`: a boundary node.
    struct Edges {
        bool left, right, bottom, top;  // the site lies at that end of the lattice
    };
    __device__ __forceinline__ Edges edges(int j, int x) const
    {
        return {x == 0, x == w - 1, !wrap && j == 0, !wrap && j == n - 1};
    }
    __device__ __forceinline__ int source(const Edges &e, int k, bool wall) const
    {
        const int o = k * plane() - dr(k) * w - dc(k);
        if (dr(k) == 0 && dc(k) == 0) return o;
        const bool col = dc(k) > 0 ? e.left : (dc(k) < 0 ? e.right : false);
        const bool row = dr(k) > 0 ? e.bottom : (dr(k) < 0 ? e.top : false);
        if (wrapx && col && !row) return o + (dc(k) > 0 ? w : -w);
        return (row || (col && !wrapx)) ? (wall ? k : Lat<9>::opp(k)) * plane() : o;
    }

    // A site's populations (v, all Q) into buffer b at local row r, and into the copies
    // of the neighbours that pull them or evaluate its dS.
    __device__ __forceinline__ void store(int b, int r, int x, const float v[9]) const
    {
        const int o = at(b, r, x);
#pragma unroll
        for (int k = 0; k < 9; ++k) f[o + k * plane()] = v[k];
        // the first two rows are rows below_rows + 2, + 3 of the band below (of the second
        // only what moves towards it is read there)
        if (r <= 3 && below >= 0) {
            float *to = in_block(f, below) + at(b, below_rows + r, x);
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (dr(k) <= 0 || r == 2) to[k * plane()] = v[k];
        }
        if (r >= rows && above >= 0) {  // the last two: rows 0, 1 of the band above
            float *to = in_block(f, above) + at(b, r - rows, x);
#pragma unroll
            for (int k = 0; k < 9; ++k)
                if (dr(k) >= 0 || r == rows + 1) to[k * plane()] = v[k];
        }
    }
    // Population 0 of lattice row j, column x, buffer b, in its own block.
    __device__ __forceinline__ const float *site_any(int b, int j, int x) const
    {
        const int o = owner(j);
        return in_block(f, o) + at(b, j - first_of(o) + 2, x);
    }
};

// The stats record of step s by one warp of the first block.
__device__ __noinline__ void record_step(const ResArgs &a, const CluShared &sh, int s, long long step0, long long rec0,
                                         unsigned &status)
{
    const int lane = threadIdx.x & 31, slot = s % kCluSlots;
    double tot[4];
    long long cnt[4];
    // statistic lane / 8: rows lane % 8 and lane % 8 + 8
    {
        const int st = lane >> 3, r0 = lane & 7;
        static_assert(kCluMax == 16, "two rows a lane");
        double v = sh.rows[slot][r0].v[st] + sh.rows[slot][r0 + 8].v[st];
        int c = sh.rows[slot][r0].c[st] + sh.rows[slot][r0 + 8].c[st];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            v += __shfl_xor_sync(kFull, v, o);
            c += __shfl_xor_sync(kFull, c, o);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            tot[i] = __shfl_sync(kFull, v, 8 * i);
            cnt[i] = __shfl_sync(kFull, c, 8 * i);
        }
    }
    if (lane == 0) {
        const DevStats st = step_record<false>(a, tot, cnt, 0.0, 0, 0, status, step0 + s + 1);
        a.f.stats_ring[(rec0 + s) % a.f.ring_len] = st;
        *a.f.sel_count = 0;
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kCluThreads, 1) k_cluster(const __grid_constant__ ResArgs a)
{
    extern __shared__ float dyn[];
    __shared__ CluShared sh;
    const StepParams &p = a.p;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    Band bd;
    bd.rank = (int)blockIdx.x;
    bd.n = p.ny;
    bd.w = p.nx;
    bd.hs = (bd.n + kCluMax - 1) / kCluMax + 4;
    bd.ldd = bd.w + 2;
    bd.first = bd.first_of(bd.rank);
    bd.rows = bd.first_of(bd.rank + 1) - bd.first;
    bd.wrap = bc_wrap_y(p.boundary);
    bd.wrapx = bc_wrap_x(p.boundary);
    bd.below = bd.rank > 0 ? bd.rank - 1 : (bd.wrap ? kCluMax - 1 : -1);
    bd.above = bd.rank + 1 < kCluMax ? bd.rank + 1 : (bd.wrap ? 0 : -1);
    bd.below_rows = bd.below >= 0 ? bd.first_of(bd.below + 1) - bd.first_of(bd.below) : 0;
    bd.ds = dyn;
    bd.f = dyn + bd.hs * bd.ldd;
    CluShared *lead = cg::this_cluster().map_shared_rank(&sh, 0);

    ResK kk{};
    kk.a = (float)p.a;
    kk.b2 = (float)(1.0 + p.a);
    const float dm = (float)p.delta_m;
    const bool med_on = (p.limiters & 4u) != 0;
    const int sites = bd.rows * bd.w;
    // threads that carry sites, in whole warps
    const int warps = min(kCluWarps, (sites + 31) / 32);
    const long long step0 = bd.rank == 0 ? a.f.counters[0] : 0, rec0 = bd.rank == 0 ? a.f.counters[1] : 0;
    unsigned status = *p.status;  // brought on in the recording lane

    // the band and its neighbours' edge rows
    {
        const float *src = (const float *)a.buf[a.cur];
        for (int i = t; i < (bd.rows + 4) * bd.w; i += kCluThreads) {
            const int r = i / bd.w, x = i % bd.w;
            int j = bd.first + r - 2;
            if (bd.wrap) j = j < 0 ? j + bd.n : (j >= bd.n ? j - bd.n : j);
            for (int k = 0; k < 9; ++k)
                bd.f[bd.at(0, r, x) + k * bd.plane()] = j >= 0 && j < bd.n ? src[fidx(p.plane, p.pitch, k, j, x)] : 0.f;
        }
        if (t < 2) {
            sh.acc[t].clear();
            if (p.boundary == 4) wall_star(p, t == 1, sh.fw[t]);
        }
    }
    cluster_barrier();

    const int step_r = kCluThreads / bd.w, step_x = kCluThreads % bd.w;
    const int r0 = t / bd.w + 2, x0 = t % bd.w;
    for (int s = 0; s < a.nsteps; ++s) {
        const int b = s & 1, slot = s % kCluSlots;
        ResSums<float> sum;
        // the finished site (r, x) with its limiters' phi: stored, summed
        auto finish = [&](const SiteState<9, float> &v, int r, int x, float phi_pos, float phi_med) {
            const float phi = phi_pos < phi_med ? phi_pos : phi_med;
            sum.pos += phi_pos < 1.f;
            sum.med += phi_med < 1.f;
            float out[9];
            if (phi < 1.f) {
                const float c = limit_weight(phi, kk.a, true);
#pragma unroll
                for (int k = 0; k < 9; ++k) out[k] = fmaf(-c, v.nq[k], v.fin[k]);
                sum.lim.add(__fmul_rn(__fsub_rn(1.f, __fmul_rn(phi, phi)), v.ds));
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) out[k] = v.fp[k];
            }
            bd.store(b ^ 1, r, x, out);
            sum.mass.add(__fsub_rn(v.rho, p.rho_ref));  // each term exact
            if (v.bad) {
                ++sum.bad;
                return;
            }
            sum.ds.add(v.ds);
            sum.din.add(v.dsin);
        };
        // dS of a site for the medians (its column's copy beyond the other end where the columns wrap)
        auto put_ds = [&](int r, int x, float ds) {
            float *d = bd.ds + r * bd.ldd;
            d[x + 1] = ds;
            if (bd.wrapx) {
                if (x == 0) d[bd.w + 1] = ds;
                if (x == bd.w - 1) d[0] = ds;
            }
        };
        // the site's evaluation; returns phi of the positivity rule
        auto evaluate = [&](SiteState<9, float> &v, int r, int x) -> float {
            const int j = bd.first + r - 2;
            float raw[9], phi_pos = 1.f;
            const float *at = bd.f + bd.at(b, r, x);
            const auto e = bd.edges(j, x);
#pragma unroll
            for (int k = 0; k < 9; ++k) raw[k] = at[bd.source(e, k, false)];
            pulled<9, float, float>(p, j, raw, v.fin);
            eval_site<9, float>(p, kk, v, true);
            if (!v.bad && (p.limiters & 1u)) {
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    const float fpa = p.rwf[k] + v.fp[k];  // absolute f'
                    if (fpa < 0.f) phi_pos = fminf(phi_pos, v.fa[k] / (v.fa[k] - fpa));
                }
            }
            return phi_pos;
        };

        unsigned later = 0;  // this thread's sites whose median is formed
        bool edge_later = false;
        SiteState<9, float> kept;  // the first of them, as evaluated
        float kept_pos = 1.f;
        int r = r0, x = x0;
        for (int i = t, it = 0; i < sites; i += kCluThreads, ++it) {
            const int j = bd.first + r - 2;
            float ds = 0.f;
            if (is_wall_node(p, x, j)) {
                float raw[9], fin[9];
                const float *at = bd.f + bd.at(b, r, x);
                const auto e = bd.edges(j, x);
#pragma unroll
                for (int k = 0; k < 9; ++k) raw[k] = at[bd.source(e, k, true)];
                wall_node<float, float>(p, raw, x, j, sh.fw[wall_lid(p, x, j) ? 1 : 0], fin);
                bd.store(b ^ 1, r, x, fin);
                add_wall_mass<float>(p, x, j, fin, sum.mass);
            } else {
                SiteState<9, float> v;
                const float phi_pos = evaluate(v, r, x);
                ds = v.ds;
                if (med_on && !v.bad && v.ds > dm) {
                    if (later == 0) {
                        kept = v;
                        kept_pos = phi_pos;
                    }
                    later |= 1u << it;
                    edge_later = edge_later || r == 2 || r == bd.rows + 1;
                } else {
                    finish(v, r, x, phi_pos, 1.f);
                }
            }
            if (med_on) put_ds(r, x, ds);
            r += step_r;
            x += step_x;
            if (x >= bd.w) {
                x -= bd.w;
                ++r;
            }
        }
        if (med_on) {
            if (__syncthreads_or(edge_later)) {
                // dS of the rows just outside the band
                for (int i = t; i < 2 * bd.w; i += kCluThreads) {
                    const int rr = i < bd.w ? 1 : bd.rows + 2, xx = i < bd.w ? i : i - bd.w;
                    int j = bd.first + rr - 2;
                    if (bd.wrap) j = j < 0 ? j + bd.n : (j >= bd.n ? j - bd.n : j);
                    float ds = 0.f;
                    if (j >= 0 && j < bd.n && !is_wall_node(p, xx, j)) {
                        SiteState<9, float> v;
                        evaluate(v, rr, xx);
                        ds = v.ds;
                    }
                    put_ds(rr, xx, ds);
                }
                __syncthreads();
            }
            for (bool again = false; later; again = true) {
                const int it = __ffs(later) - 1, i = t + it * kCluThreads, rr = i / bd.w + 2, xx = i % bd.w;
                const int j = bd.first + rr - 2;
                later &= later - 1u;
                float phi_med = 1.f, med;
                if (again) kept_pos = evaluate(kept, rr, xx);
                if (stencil_median<9, float>(p, bd.ds + rr * bd.ldd + xx + 1, bd.ldd, 0, 0, xx, j, med))
                    phi_med = phi_median<float>(kept.ds, med, dm, p.median_mode);
                finish(kept, rr, xx, kept_pos, phi_med);
            }
        }
        cluster_arrive();
        if (warp < warps && add_warp(sh.acc[b], sum, warps, false))
            take_row(sh.acc[b], &lead->rows[slot][bd.rank], warps);
        cluster_wait();
        if (bd.rank == 0 && warp == kCluWarps - 1) {
            // the rows of the step before are complete since this step's barrier
            if (s > 0) record_step(a, sh, s - 1, step0, rec0, status);
            if (a.f.probe != nullptr && lane == 0) {
                // the control point's moments after the whole step, as lbm_moments gives them
                float raw[9];
                const float *at = bd.site_any(b ^ 1, a.f.probe_site / p.nx, a.f.probe_site % p.nx);
#pragma unroll
                for (int k = 0; k < 9; ++k) raw[k] = at[k * bd.plane()];
                double r, u, v;
                site_moments<9, float>(p, raw, r, u, v);
                double *to = a.f.probe + 3 * ((step0 + s) % a.f.probe_cap);
                to[0] = r;
                to[1] = u;
                to[2] = v;
            }
            __syncwarp();
        }
    }
    cluster_barrier();  // the last rows, and every access to another block's memory
    if (bd.rank == 0 && warp == kCluWarps - 1) {
        record_step(a, sh, a.nsteps - 1, step0, rec0, status);
        if (lane == 0) {
            a.f.counters[0] = step0 + a.nsteps;
            a.f.counters[1] = rec0 + a.nsteps;
        }
    }
    float *dst = (float *)a.buf[(a.cur + a.nsteps) & 1];
    for (int i = t; i < sites; i += kCluThreads) {
        const int r = i / bd.w, x = i % bd.w;
        for (int k = 0; k < 9; ++k)
            dst[fidx(p.plane, p.pitch, k, bd.first + r, x)] = bd.f[bd.at(a.nsteps & 1, r + 2, x) + k * bd.plane()];
    }
}

// Dynamic shared memory of a block.
size_t cluster_bytes(int nx, int ny)
{
    const size_t hs = (size_t)(ny + kCluMax - 1) / kCluMax + 4;
    return (hs * (nx + 2) + 2 * 9 * hs * nx) * sizeof(float);
}

cudaLaunchConfig_t cluster_config(size_t bytes, cudaStream_t s, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)kCluMax);
    cfg.blockDim = dim3(kCluThreads);
    cfg.dynamicSmemBytes = bytes;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)kCluMax;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// Whether the current device runs the cluster (16 blocks of this size): asked once for each
// device, as the kernel's attributes are set for each.  Two threads that ask at once set the
// same.
bool cluster_runs()
{
    constexpr int kDevices = 64;
    static std::atomic<int> known[kDevices];  // 0: not asked, 1: it does not, 2: it does
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) {
        cudaGetLastError();
        return false;
    }
    if (known[dev].load() == 0) {
        cudaLaunchAttribute attr;
        const cudaLaunchConfig_t cfg = cluster_config(kCluMaxBytes, nullptr, &attr);
        int fit = 0;
        const bool ok =
            cudaFuncSetAttribute(k_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCluMaxBytes) == cudaSuccess &&
            cudaFuncSetAttribute(k_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
            cudaOccupancyMaxActiveClusters(&fit, k_cluster, &cfg) == cudaSuccess && fit > 0;
        if (!ok) cudaGetLastError();
        known[dev].store(ok ? 2 : 1);
    }
    return known[dev].load() == 2;
}

}  // namespace

bool cluster_applies(const lbm_config &c)
{
    // at least two rows a block
    return resident_applies(c) && c.lattice == LBM_D2Q9 && c.precision == LBM_FP32 && !(c.limiters & LBM_LIM_EHRENFEST) &&
           c.ny >= 2 * kCluMax && (long long)c.nx * c.ny <= kCluMaxSites && cluster_bytes(c.nx, c.ny) <= kCluMaxBytes;
}

cudaError_t launch_cluster(ResArgs a, cudaStream_t s)
{
    if (!cluster_runs()) return cudaErrorNotSupported;
    a.rest = rest_mass(a.p);
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(cluster_bytes(a.p.nx, a.p.ny), s, &attr);
    return cudaLaunchKernelEx(&cfg, k_cluster, a);
}

}  // namespace lbm
