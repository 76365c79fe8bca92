// step_resident.cu -- many limited LBGK steps of a small lattice in one launch.
//
// A step of a lattice that fits in L2 takes a few microseconds of work, but a
// pair of launches per step (step kernel, tail) costs 16 to 20 us: the host
// enqueues about 10 us apart, each kernel starts from a cold instruction cache
// (about 10 ns per instruction fetched), and the tail runs alone.  Here one
// cooperative launch takes up to kResMaxSteps steps.  Its blocks, one per SM,
// keep their tiles for the whole launch and meet at a grid barrier (a counter in
// L2) after every step; the two population buffers swap roles from step to step.
//  * Worker blocks finish the sites of their tiles, a site per thread: free
//    flight, collision, dS, positivity rule, median filter, candidates.  Tiles do
//    not overlap: the median of a tile's edge sites needs dS of sites outside it,
//    which are evaluated only when an edge site's median is formed (dS above
//    delta, rare).
//  * The last block is the tail: sums, stats record, control point, Ehrenfests'
//    selection and step (select.cuh).  It works on step s while the workers
//    already take step s + 1; only a step that recorded candidates makes them
//    wait for its selection (the step's arrival counter carries its candidate count,
//    so a step without any costs no further read).  FP32 / 16-bit storage: the FP64
//    keys of more than a few candidates are evaluated by all blocks first.
// The per-site operations are those of the fused, tube and tiled kernels, so the
// populations are the same bit for bit.  Sums, in a fixed order: a thread's and a
// warp's in the storage's compute type (FP32 with the rounding errors kept beside the
// sums, see SumOf), block rows in FP64 and in block order.
// Every wait is bounded (kResSpin polls, over a second); a block that gives up
// sets kStatTimeout and leaves, and the others follow when their own waits end.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "resident.cuh"
#include "select.cuh"
#include "site.cuh"

namespace lbm {
namespace {

constexpr int kResThreads = kFinThreads;   // the tail block runs the selection of select.cuh
constexpr int kResWarps = kResThreads / 32;
constexpr unsigned kTailKeys = 12;         // candidates of a step that the tail keys alone (three a warp: a warp on each sub-partition)
constexpr int kPoller = kResThreads - 32;  // worker thread that waits: its warp seldom has sums to add first
constexpr unsigned kResSpin = 4u << 20;    // polls of a wait before giving up (0.5 to 1 us each)

__device__ __forceinline__ unsigned long long ld_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void red_release(unsigned *p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_release(unsigned *p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Polls *p (a counter that only grows within the launch) until it reaches
// `target`; false when the wait gave up.
__device__ __forceinline__ bool wait_for(const unsigned *p, unsigned target, unsigned *status)
{
    for (unsigned i = 0; i < kResSpin; ++i)
        if (ld_acquire(p) >= target) return true;
    atomicOr(status, kStatTimeout);
    return false;
}
// Waits for all W workers' arrivals at step s; *n receives the candidates of the step.
// seen: the caller's candidate totals of the slots so far.
__device__ __forceinline__ bool wait_arrivals(const ResState *rs, int s, int W, unsigned *seen, unsigned *n,
                                              unsigned *status)
{
    const int slot = s % kResSlots;
    const unsigned target = (unsigned)W * (unsigned)(s / kResSlots + 1);
    for (unsigned i = 0; i < kResSpin; ++i) {
        const unsigned long long v = ld_acquire(&rs->arrived[slot]);
        if ((unsigned)v >= target) {
            *n = (unsigned)(v >> 32) - seen[slot];
            seen[slot] = (unsigned)(v >> 32);
            return true;
        }
    }
    atomicOr(status, kStatTimeout);
    return false;
}

// A worker block's shared memory.
template <typename T>
struct WorkShared {
    T ds[2][(kResWarps + 2) * 34];  // dS of the tile (D2Q9: rows of 34 with the halo; D1Q3: 32 aw + 2)
    BlockAcc<kResWarps, T> acc[2];     // the block's sums, steps of each parity
    int ncand[2];
    double fw[2][9];                // diffusive wall: f*(1, u_wall) of the resting walls and of the lid
    unsigned n;                     // candidates of the step (after the barrier)
    unsigned seen[kResSlots];       // the waiting thread's: see wait_arrivals
    int go;                         // 0: a wait gave up
    int stop;                       // 1: the wait for a row's place gave up
};

// dS(f') of a site outside the tile (0 at boundary nodes and off the lattice).
template <int Q, typename S>
__device__ __noinline__ compute_t<S> halo_ds(const StepParams &p, ResK kk, const S *src, int x, int y)
{
    using T = compute_t<S>;
    if (bc_wrap_x(p.boundary)) x = x < 0 ? x + p.nx : (x >= p.nx ? x - p.nx : x);
    if (Q == 9 && bc_wrap_y(p.boundary)) y = y < 0 ? y + p.ny : (y >= p.ny ? y - p.ny : y);
    if (x < 0 || x >= p.nx || y < 0 || y >= p.ny || (Q == 9 && is_wall_node(p, x, y))) return T(0);
    SiteState<Q, T> v;
    pull<Q, S, T>(p, src, x, y, v.fin);
    eval_site<Q, S>(p, kk, v, false);
    return v.ds;
}

// One tile: aw rows of 32 sites (D2Q9; a warp per row) or 32 aw consecutive sites
// (D1Q3).  Every site is stored, candidates recorded, sums taken.  Every thread
// of the block calls it; warps from aw on only take part in the barriers.
template <int Q, typename S>
__device__ __forceinline__ void do_tile(const StepParams &p, const ResK &kk, const S *src, S *dst, int tile, int gx, int aw,
                                        compute_t<S> *sds, const double (*fw)[9], int *ncand,
                                        ResSums<compute_t<S>> &sum)
{
    using T = compute_t<S>;
    using A = Ar<T>;
    constexpr bool F64 = std::is_same<T, double>::value;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int by = Q == 9 ? tile / gx : 0, bx = Q == 9 ? tile - by * gx : tile;
    const int x0 = Q == 9 ? 32 * bx : 32 * aw * bx, y0 = Q == 9 ? aw * by : 0;
    const int x = Q == 9 ? x0 + lane : x0 + t, y = Q == 9 ? y0 + warp : 0;
    const bool own_site = warp < aw && x < p.nx && y < p.ny;
    const int ld = Q == 9 ? 34 : 0;
    const int at = Q == 9 ? (warp + 1) * ld + lane + 1 : t + 1;  // the site's place in sds
    SiteState<Q, T> v;
    bool wall = false;
    T phi_pos = T(1), phi_med = T(1);
    const bool med_on = (p.limiters & 4u) != 0;
    T dm;
    if constexpr (F64)
        dm = p.delta_m;
    else
        dm = kk.dm;
    // (the warp's vote: its loads go out together, at the edges of the lattice too)
    const bool edge_warp = __any_sync(kFull, own_site && (x == 0 || x == p.nx - 1 || (Q == 9 && (y == 0 || y == p.ny - 1))));
    bool need = false;
    bool acts = !F64;  // FP64: a limiter may act (spares the comparisons of phi)
    if (own_site) {
        wall = Q == 9 && is_wall_node(p, x, y);
        S raw[Q];
        pull_raw<Q, S>(p, src, x, y, edge_warp, wall, raw);
        if (wall) {
            if constexpr (Q == 9) wall_node<S, T>(p, raw, x, y, fw[wall_lid(p, x, y) ? 1 : 0], v.fin);
            v.ds = T(0);
        } else {
            pulled<Q, S, T>(p, y, raw, v.fin);
            eval_site<Q, S>(p, kk, v, true);
            if (!v.bad) {
                if (p.limiters & 1u) {
                    if constexpr (F64) {
                        bool neg = false;
#pragma unroll
                        for (int k = 0; k < Q; ++k) neg |= lt0(v.fp[k]);
                        if (neg) phi_pos = phi_positivity<Q, T>(v.fs, v.fp);
                        acts |= neg;
                    } else {
#pragma unroll
                        for (int k = 0; k < Q; ++k) {
                            const float fpa = p.rwf[k] + v.fp[k];  // absolute f'
                            if (fpa < 0.f) phi_pos = fminf(phi_pos, v.fa[k] / (v.fa[k] - fpa));
                        }
                    }
                }
                if constexpr (F64)
                    need = med_on && above64(v.ds, dm);
                else
                    need = med_on && v.ds > dm;
                acts |= need;
            }
        }
    }
    if (med_on) {
        if (own_site) sds[at] = v.ds;
        // the stencils of the tile's edge sites reach outside it: evaluate dS there
        // only when one of them forms its median
        const bool edge = Q == 9 ? (lane == 0 || lane == 31 || warp == 0 || warp == aw - 1) : (t == 0 || t == 32 * aw - 1);
        const bool part = x == p.nx - 1 || (Q == 9 && y == p.ny - 1);  // sites beyond the lattice's end (periodic lattices)
        if (__syncthreads_or(need && (edge || part))) {
            if constexpr (Q == 9) {
                const int w = min(32, p.nx - x0), h = min(aw, p.ny - y0);
                for (int i = t; i < 2 * (w + 2) + 2 * h; i += kResThreads) {
                    int hx, hy;
                    if (i < 2 * (w + 2)) {
                        hy = i < w + 2 ? -1 : h;
                        hx = (i < w + 2 ? i : i - (w + 2)) - 1;
                    } else {
                        const int j = i - 2 * (w + 2);
                        hx = j < h ? -1 : w;
                        hy = j < h ? j : j - h;
                    }
                    sds[(hy + 1) * ld + hx + 1] = halo_ds<Q, S>(p, kk, src, x0 + hx, y0 + hy);
                }
            } else {
                const int w = min(32 * aw, p.nx - x0);
                if (t < 2) sds[t == 0 ? 0 : w + 1] = halo_ds<Q, S>(p, kk, src, t == 0 ? x0 - 1 : x0 + w, 0);
            }
            __syncthreads();
        }
        if (need) {
            T med;
            // (the stencil's centre is given by the pointer)
            if (stencil_median<Q, T>(p, sds + at, Q == 9 ? ld : 0, 0, 0, x, y, med)) phi_med = phi_median<T>(v.ds, med, dm, p.median_mode);
        }
    }
    if (!own_site) return;
    if (wall) {
#pragma unroll
        for (int k = 0; k < Q; ++k) dst[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(v.fin[k]);
        if constexpr (Q == 9) add_wall_mass<T>(p, x, y, v.fin, sum.mass);
        return;
    }
    T phi = T(1);
    if (acts) {
        phi = phi_pos < phi_med ? phi_pos : phi_med;
        sum.pos += phi_pos < T(1);
        sum.med += phi_med < T(1);
    }
    if (acts && phi < T(1)) {
        if constexpr (F64) {
#pragma unroll
            for (int k = 0; k < Q; ++k)
                dst[fidx(p.plane, p.pitch, k, y, x)] = A::add(v.fs[k], A::mul(phi, A::sub(v.fp[k], v.fs[k])));
            sum.lim.add(A::mul(A::sub(1.0, A::mul(phi, phi)), v.ds));
        } else {
            const float c = limit_weight(phi, kk.a, true);
#pragma unroll
            for (int k = 0; k < Q; ++k) dst[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(fmaf(-c, v.nq[k], v.fin[k]));
            sum.lim.add(__fmul_rn(__fsub_rn(1.f, __fmul_rn(phi, phi)), v.ds));
        }
    } else {
#pragma unroll
        for (int k = 0; k < Q; ++k) dst[fidx(p.plane, p.pitch, k, y, x)] = f2s<S>(v.fp[k]);
    }
    if constexpr (F64)
        sum.mass.add(v.rho);
    else
        sum.mass.add(__fsub_rn(v.rho, p.rho_ref));  // each term exact
    if (v.bad) {
        ++sum.bad;
        return;
    }
    sum.ds.add(v.ds);
    sum.din.add(v.dsin);
    if (p.limiters & 2u) {
        // Ehrenfests' candidate: FP64 storage with its key; FP32 / 16-bit storage near
        // or above the threshold, keyed by the tail where it can matter
        bool is;
        if constexpr (F64)
            is = above64(v.ds, p.delta_e);
        else
            is = v.ds > kk.thr_e;
        if (is) {
            atomicAdd(ncand, 1);
            const int slot = atomicAdd(p.cand_count, 1);
            if (slot < p.cand_cap) {  // at most one per site: always, but after a launch that gave up
                Cand c;
                c.key = F64 ? (double)v.ds : __longlong_as_double(0x7ff8000000000000LL);
                c.phi = (double)phi;
                c.site = y * p.nx + x;
                c.ds32 = (float)v.ds;
                p.cand[slot] = c;
            } else {
                atomicOr(p.status, kStatCandOverflow);
            }
        }
    }
}

// A worker warp's sums of step s into the block's; the block's last warp to come
// writes the block's row and reports it (the tail reads the rows of a step when
// every worker has reported).  Runs while the grid barrier completes.
template <int Q, typename T>
__device__ __forceinline__ void block_sums(const ResArgs &a, WorkShared<T> &w, const ResSums<T> &sum, int s, int aw)
{
    const int lane = threadIdx.x & 31, b = s & 1;
    if (!add_warp(w.acc[b], sum, aw, Q == 3 && a.tiles < (int)gridDim.x)) return;
    // the rows of step s - kResRows are read before this one takes their place
    if (s >= kResRows && lane == 0 && !wait_for(&a.rs->stats_done, (unsigned)(s - kResRows + 1), a.p.status))
        w.stop = 1;  // the block leaves at its next barrier
    __syncwarp();
    take_row(w.acc[b], &a.rs->rows[s % kResRows][blockIdx.x], aw);
    if (lane == 0) red_release(&a.rs->rows_in[s % kResRows], 1u);
}

// A worker's share of the keys of a step with n > kTailKeys candidates: three to
// a warp (a lane per direction) while that is one round, else a lane each.
template <int Q, typename S>
__device__ __noinline__ void key_share(const StepParams &p, const S *src, int n, int W)
{
    const int t = threadIdx.x, lane = t & 31;
    const KeyGeom kg = key_geom(p);
    // warp numbers run over the blocks first, so that a few candidates spread over the SMs
    const int w = (t >> 5) * W + (int)blockIdx.x, nw = W * kResWarps;
    if (Q == 9 && n <= 3 * nw) {
        const int g = lane < 27 ? lane / 9 : 0;
        if (3 * w < n) {
            const int i = min(3 * w + g, n - 1);
            const double key = key_dS9_group<S>(kg, src, p.cand[i].site, p.delta_e);
            if (lane < 27 && lane % 9 == 0 && 3 * w + g < n) p.cand[i].key = key;
        }
    } else {
        for (int i = 32 * w + lane; i < n; i += 32 * nw)
            p.cand[i].key = key_dS_lane<Q, S>(kg, src, p.cand[i].site, p.delta_e);
    }
}

template <int Q, typename S>
__device__ __forceinline__ void work_block(const ResArgs &a, WorkShared<compute_t<S>> &w)
{
    using T = compute_t<S>;
    const int t = threadIdx.x, warp = t >> 5;
    const StepParams &p = a.p;
    const int W = (int)gridDim.x - 1, aw = a.aw;
    const bool ehr = (p.limiters & 2u) != 0;
    ResK kk{};
    if constexpr (!std::is_same<T, double>::value) {
        kk.a = (float)p.a;
        kk.b2 = (float)(1.0 + p.a);
        kk.dm = (float)p.delta_m;
        kk.thr_e = (float)(p.delta_e * (1.0 - 1.0 / 64.0));
    }
    if (t < 2) {
        w.acc[t].clear();
        w.ncand[t] = 0;
        if (Q == 9 && p.boundary == 4) wall_star(p, t == 1, w.fw[t]);
    }
    if (t < kResSlots) w.seen[t] = 0;
    if (t == 0) w.stop = 0;
    __syncthreads();
    int tile_no = 0;
    for (int s = 0; s < a.nsteps; ++s) {
        const S *src = (const S *)a.buf[(a.cur + s) & 1];
        S *dst = (S *)a.buf[(a.cur + s + 1) & 1];
        ResSums<T> sum;
        for (int tile = blockIdx.x; tile < a.tiles; tile += W)
            do_tile<Q, S>(p, kk, src, dst, tile, a.gx, aw, w.ds[tile_no++ & 1], w.fw, &w.ncand[s & 1], sum);
        __syncthreads();  // the block's sites are stored and its candidates counted
        if (t == 0) {
            red_release(&a.rs->arrived[s % kResSlots], 1ull | ((unsigned long long)(unsigned)w.ncand[s & 1] << 32));
            w.ncand[s & 1] = 0;
        }
        if (warp < aw) block_sums<Q, T>(a, w, sum, s, aw);
        const bool end = s + 1 == a.nsteps;
        if (end && !ehr) return;
        if (t == kPoller) w.go = wait_arrivals(a.rs, s, W, w.seen, &w.n, p.status);
        __syncthreads();
        if (!w.go || w.stop) return;
        const unsigned n = min(w.n, (unsigned)p.cand_cap);
        if (n > kTailKeys && !std::is_same<S, double>::value) {
            key_share<Q, S>(p, src, (int)n, W);
            __syncthreads();
            if (t == 0) red_release(&a.rs->keyed, 1u);
        }
        if (end) return;
        if ((n > 0 || a.f.probe != nullptr)) {
            // the tail equilibrates the chosen sites (and reads the control point) first
            if (t == kPoller) {
                const unsigned *flag = a.f.probe != nullptr ? &a.rs->stats_done : &a.rs->done;
                w.go = wait_for(flag, (unsigned)(s + 1), p.status);
            }
            __syncthreads();
            if (!w.go) return;
        }
    }
}

struct TailShared {
    SelShared sel;
    FinalParams f;
    double tot[4];
    long long cnt[4];
    unsigned n, seen[kResSlots];
    int go;
};

template <int Q, typename S>
__device__ __noinline__ void tail_block(const ResArgs &a, TailShared &h)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int W = (int)gridDim.x - 1;
    constexpr bool F64 = std::is_same<S, double>::value;
    {
        const unsigned *from = reinterpret_cast<const unsigned *>(&a.f);
        unsigned *to = reinterpret_cast<unsigned *>(&h.f);
        for (int i = t; i < (int)(sizeof(FinalParams) / 4); i += kResThreads) to[i] = from[i];
    }
    long long step = a.f.counters[0], rec = a.f.counters[1];
    unsigned dense = 0, status = *a.p.status;
    if (t < kResSlots) h.seen[t] = 0;
    __syncthreads();
    const FinalParams &f = h.f;
    for (int s = 0; s < a.nsteps; ++s) {
        S *dst = (S *)a.buf[(a.cur + s + 1) & 1];
        if (t == 0) {
            h.go = wait_arrivals(a.rs, s, W, h.seen, &h.n, a.p.status);
            h.f.src = a.buf[(a.cur + s) & 1];
            h.sel.nsel = 0;
        }
        __syncthreads();
        if (!h.go) break;
        const unsigned n = min(h.n, (unsigned)f.cand_cap);
        int n_valid = 0;
        double ehr_sum = 0.0;
        if (n > 0) {
            if (n > kTailKeys && !F64) {
                ++dense;
                if (t == 0) h.go = wait_for(&a.rs->keyed, (unsigned)W * dense, a.p.status);
                __syncthreads();
                if (!h.go) break;
            }
            const Cand none{};
            ehr_sum = finish_candidates<Q, S>(f, dst, (int)n, false, false, none, h.sel, n_valid);
            __syncthreads();
            if (t == 0) {
                *f.cand_count = 0;
                st_release(&a.rs->done, (unsigned)(s + 1));
            }
            ehr_sum = h.sel.nsel > 0 ? block_sum0(ehr_sum, h.sel.red, h.sel.nsel <= 32) : 0.0;
        }
        // the step's sums: every worker's row, in block order
        if (t == 0)
            h.go = wait_for(&a.rs->rows_in[s % kResRows], (unsigned)W * (unsigned)(s / kResRows + 1), a.p.status);
        __syncthreads();
        if (!h.go) break;
        if (warp < 4) {
            double v;
            int c;
            sum_rows(a.rs->rows[s % kResRows], W, warp, v, c);
            if (lane == 0) {
                h.tot[warp] = v;
                h.cnt[warp] = c;
            }
        }
        __syncthreads();
        if (t == 0) {
            step += 1;
            const DevStats st = step_record<F64>(a, h.tot, h.cnt, ehr_sum, h.sel.nsel, n_valid, status, step);
            f.stats_ring[rec % f.ring_len] = st;
            rec += 1;
            if (f.probe != nullptr) {
                // the control point's moments after the whole step, as lbm_moments gives them
                const int x = f.probe_site % f.nx, y = f.probe_site / f.nx;
                double r, u, v;
                S raw[Q];
#pragma unroll
                for (int q = 0; q < Q; ++q) raw[q] = dst[fidx(f.plane, f.pitch, q, y, x)];
                site_moments<Q, S>(a.p, raw, r, u, v);
                double *slot = f.probe + 3 * ((step - 1) % f.probe_cap);
                slot[0] = r;
                slot[1] = u;
                slot[2] = v;
            }
            *f.sel_count = h.sel.nsel;
            if (f.probe != nullptr)
                st_release(&a.rs->stats_done, (unsigned)(s + 1));
            else  // the rows are read (their sums are formed): nothing else to order
                *(volatile unsigned *)&a.rs->stats_done = (unsigned)(s + 1);
        }
    }
    if (t == 0) {
        f.counters[0] = step;
        f.counters[1] = rec;
    }
}

// The last block of the grid is the tail, the others are workers.
template <int Q, typename S>
__global__ void __launch_bounds__(kResThreads, 1) k_resident(const __grid_constant__ ResArgs a)
{
    using T = compute_t<S>;
    union alignas(16) Shared {
        char work[sizeof(WorkShared<T>)];
        char tail[sizeof(TailShared)];
    };
    __shared__ Shared sh;
    if (blockIdx.x + 1 == gridDim.x)
        tail_block<Q, S>(a, *reinterpret_cast<TailShared *>(sh.tail));
    else
        work_block<Q, S>(a, *reinterpret_cast<WorkShared<T> *>(sh.work));
}

}  // namespace

bool resident_applies(const lbm_config &c)
{
    if (c.kernel != LBM_KERNEL_AUTO || c.equilibrium != LBM_EQ_POLYNOMIAL || (c.limiters & kLimEnsemble)) return false;
    if (c.lattice == LBM_D1Q3 && c.precision != LBM_FP64 && c.precision != LBM_FP32) return false;
    const long long most = c.precision == LBM_FP64 ? kResMaxSites64 : (c.lattice == LBM_D1Q3 ? kResMaxSites3 : kResMaxSites);
    return (long long)c.nx * c.ny <= most;
}

// What FP32 / 16-bit storage leaves out of the mass: rho_ref per site, and at the
// boundary nodes of a lattice with nodes on the walls rho_ref W_k for the
// populations that stream back.
double rest_mass(const StepParams &p)
{
    if (!bc_node_walls(p.boundary)) return (double)p.rho_ref * (double)((long long)p.nx * p.ny);
    const long long inner = (long long)(p.nx - 2) * (p.ny - 2);
    double m = (double)p.rho_ref * (double)inner;
    for (int k = 0; k < 9; ++k) {
        // nodes whose neighbour in direction k is on the lattice, less the inner ones
        const long long all = (long long)(p.nx - (Lat<9>::cx(k) != 0)) * (p.ny - (Lat<9>::cy(k) != 0));
        m += (double)(all - inner) * p.rw[k];
    }
    return m;
}

// Time of one round of a worker, a tile of `rows` rows of 32 sites, in units that only
// compare.  FP64: its units bound a round, 12.5 / 20 / 37.3 us for 4 / 8 / 16 rows of
// D2Q9 (tubes: a third, in the same proportion).  FP32 and 16-bit: latency does, 1.4 us
// and 0.06 a row.  us a step at 4 / 8 / 16 rows:
//   FP32 cavities 100^2 12.4 / 12.1 / 12.3, 200^2 15.7 / 14.3 / 12.1, 400^2 24.6 / 18.4 /
//   16.9, 2000 x 100 28.4 / 20.7 / 16.8, boundary nodes 150^2 8.2 / 5.1 / 5.6;
//   FP64 cavities 100^2 30.8 / 31.6 / 46.1, 200^2 55 / 59 / 46, 400^2 123 / 117 / 133,
//   700^2 317 / 266 / 276;
//   tubes FP32 2e5 13.1 / 11.1 / 9.8, 7e5 26.9 / 18.2 / 13.3; FP64 5e5 124 / 100 / 106.
int round_cost(bool fp64, int rows)
{
    if (!fp64) return rows + 22;
    if (rows <= 4) return 250;
    if (rows <= 8) return 250 + (rows - 4) * 150 / 4;
    return 400 + (rows - 8) * 346 / 8;
}

bool resident_grid(const lbm_config &c, int streams, ResGrid *g)
{
    const bool fp64 = c.precision == LBM_FP64, tube = c.lattice == LBM_D1Q3;
    // A cooperative grid starts when all of its blocks have a place, and a block takes the
    // whole SM.  So one SM is left to whatever else runs for long (a kernel of one block on
    // another stream would hold up the steps until it ends), and a grid of several rounds
    // has no more blocks than its rounds need.
    const int sms = std::min(sm_count(), kResMaxBlocks), workers = std::max(1, sms - 2);
    // warps that carry sites (rows of a tile): the least time of the busiest SM, its rounds
    // times the time of one, rows beyond the lattice left out
    long long best = -1;
    for (int w = 4; w <= kResWarps; w *= 2) {
        const int gx = tube ? 1 : (c.nx + 31) / 32;
        const int tiles = tube ? (c.nx + 32 * w - 1) / (32 * w) : gx * ((c.ny + w - 1) / w);
        const long long rounds = (tiles + workers - 1) / workers;
        const long long cost = rounds * round_cost(fp64, tube ? w : std::min(w, c.ny));
        if (streams > 1 && tiles + 1 > sms / streams) continue;
        if (best >= 0 && cost >= best) continue;
        best = cost;
        *g = {w, gx, tiles, (int)((tiles + rounds - 1) / rounds) + 1, 0};
    }
    if (best < 0) return false;
    // units of round_cost: 1/20 us in FP64 (tubes a third), 1/16 us otherwise
    const double us = 8.0 + (double)best * (fp64 ? (tube ? 1.0 / 60 : 1.0 / 20) : 1.0 / 16);
    g->most_steps = std::max(16, std::min(kResMaxSteps, (int)(kResLaunchUs / us)));
    return true;
}

template <typename S>
cudaError_t launch_resident(int q, ResArgs a, cudaStream_t s)
{
    a.rest = rest_mass(a.p);
    cudaError_t e = cudaMemsetAsync(a.rs, 0, offsetof(ResState, rows), s);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.blocks);
    cfg.blockDim = dim3(kResThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if constexpr (std::is_same<S, double>::value || std::is_same<S, float>::value)
        if (q == 3) return cudaLaunchKernelEx(&cfg, k_resident<3, S>, a);
    return cudaLaunchKernelEx(&cfg, k_resident<9, S>, a);
}

template cudaError_t launch_resident<float>(int, ResArgs, cudaStream_t);
template cudaError_t launch_resident<double>(int, ResArgs, cudaStream_t);
template cudaError_t launch_resident<__nv_bfloat16>(int, ResArgs, cudaStream_t);
template cudaError_t launch_resident<__half>(int, ResArgs, cudaStream_t);

}  // namespace lbm
