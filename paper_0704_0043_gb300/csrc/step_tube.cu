// step_tube.cu -- one limited LBGK step of a D1Q3 lattice (the shock tube of
// Sec. 4.3) as a single streaming pass.
//
// The step is that of the tiled kernel for Q = 3 (free flight, Eq. lbgkLB or
// Eq. elbm, dS of Sec. 3.6 / Eq. DelS, the positivity rule of Sec. 3.1, the
// three-point median filter of Sec. 3.5, Ehrenfests' candidates of Sec. 3.2,
// the sums of Sec. 3.4), evaluated per site with the same device functions,
// so the stored populations are the same bit for bit.  What differs is the
// decomposition, made for a one-dimensional lattice:
//   * a warp owns a contiguous chunk of sites and finishes all of them (no
//     overlapping tiles, no shared memory, no block barrier in the step); each
//     lane loads V consecutive sites of every plane as one 16-byte vector
//     (FP32: 4 sites, FP64: 2), or one site with V = 1;
//   * the streamed neighbours come from the adjacent lanes by shuffles; only
//     the two chunk-edge values are loaded on their own;
//   * the median needs dS of the neighbour sites: inside the chunk they are in
//     registers or on the adjacent lane, and dS of a site just outside the
//     chunk is evaluated on demand, only for an edge site whose median is
//     formed (dS above delta_M; rare);
//   * FP64 storage is bound by this GPU's FP64 units, which take a warp's FP64
//     instruction in 64 cycles whatever the number of active lanes: a short
//     tube runs one site per lane (V = 1) and one warp per block, so its warps
//     land on separate SM sub-partitions and the step lasts one site's chain;
//   * FP32 storage with four sites a lane evaluates them as two pairs with the
//     paired FP32 instructions.  A chunk of 128 sites on which nothing acts (no
//     limiter, no end of the tube, no Ehrenfests' candidate) is finished there
//     with three vector stores; in any other, the pairs on which nothing acts
//     are, and an out-of-line function takes the rest, so the walk's registers
//     hold little more than the common case needs.  Bound by HBM at 1e8
//     sites (523 -> 414 us, 86 % of the copy rate); at 1e7 (72 -> 62 us a step, 493 ->
//     331 warp instructions a chunk) by the warps that meet the front's chunks, whose
//     cold code makes them end later than the others; 3e6 sites with all three
//     limiters 42 -> 37 us, with 0.5 % of the sites limited 63 -> 62 us; 24 warps at
//     80 registers spill, 1e7 sites 82 us.  Leaving whole chunks to the function:
//     62 us, but 72 us with 0.5 % of 3e6 sites limited.
// Ensemble-dependent limiters and 16-bit storage stay on the tiled kernel.
#include <type_traits>

#include "internal.h"
#include "lattice.cuh"

namespace lbm {
namespace {

__device__ __forceinline__ long long tidx(const StepParams &p, int k, int x) { return (long long)k * p.plane + kLead + x; }

// Stored value as a compute value (as in the tiled kernel): FP64 storage is f,
// FP32 storage the deviation g, read as g in FP32 or as (double) g + rw_k.
template <typename S, typename T>
__device__ __forceinline__ T tload(const StepParams &p, S v, int k)
{
    if constexpr (std::is_same<S, double>::value)
        return T(v);
    else if constexpr (std::is_same<T, double>::value)
        return Ar<double>::add((double)v, p.rw[k]);
    else
        return v;
}

// Free flight of one site (pull, Sec. 2): index 1 moves left (v = -1) and
// arrives from x + 1, index 2 from x - 1; closed ends reflect (halfway
// bounce-back: f_in_k = f_opp(k) of the site itself), periodic ends wrap.
template <typename S, typename T>
__device__ void tube_pull(const StepParams &p, const S *__restrict__ f, int x, T fin[3])
{
    const bool wrap = bc_wrap_x(p.boundary);
    int r = x + 1, l = x - 1;
    if (r >= p.nx) r = wrap ? 0 : -1;
    if (l < 0) l = wrap ? p.nx - 1 : -1;
    fin[0] = tload<S, T>(p, f[tidx(p, 0, x)], 0);
    fin[1] = tload<S, T>(p, f[tidx(p, r >= 0 ? 1 : 2, r >= 0 ? r : x)], 1);  // W_1 = W_2
    fin[2] = tload<S, T>(p, f[tidx(p, l >= 0 ? 2 : 1, l >= 0 ? l : x)], 2);
}

template <typename S, typename T>
__device__ __forceinline__ void tube_read(const StepParams &p, const S *__restrict__ f, int x, T fin[3])
{
#pragma unroll
    for (int k = 0; k < 3; ++k) fin[k] = tload<S, T>(p, f[tidx(p, k, x)], k);
}

// Per-thread constants of FP32 storage (the FP64 parameters converted once).
struct TubeK {
    float a, b2, dm, thr_e;
};

// Collision and dS of one site (site_collide / site_collide_dev, as the tiled
// kernel calls them).  dS = +inf for a site that cannot be limited.
template <typename T>
__device__ __forceinline__ bool tube_eval(const StepParams &p, const TubeK &kk, const T fin[3], T fs[3], T fp[3],
                                          T fa[3], float nq[3], T &ds, T &dsin, T &rho, bool need_in)
{
    bool bad;
    if constexpr (std::is_same<T, double>::value) {
        bad = site_collide<3, double>(fin, p.a, p.collide != 0, fs, fp, ds, dsin, rho, p.eq, need_in, p.coll, p.beta);
#pragma unroll
        for (int k = 0; k < 3; ++k) fa[k] = fs[k];
        (void)nq;
    } else {
        bad = site_collide_dev<3>(fin, kk.a, kk.b2, p.collide != 0, p.rho_ref, p.rwf, fs, nq, fp, fa, ds, dsin, rho,
                                  p.eq);
    }
    if (bad) ds = T(INFINITY);
    return bad;
}

// dS(f') of site x alone (a median neighbour outside the warp's chunk).
template <typename S>
__device__ compute_t<S> tube_ds(const StepParams &p, const TubeK &kk, const S *__restrict__ src, int x)
{
    using T = compute_t<S>;
    T fin[3], fs[3], fp[3], fa[3], ds, dsin, rho;
    float nq[3];
    if (p.collide)
        tube_pull<S, T>(p, src, x, fin);
    else
        tube_read<S, T>(p, src, x, fin);
    tube_eval<T>(p, kk, fin, fs, fp, fa, nq, ds, dsin, rho, false);
    return ds;
}

// The polynomial FP32 collision of two sites at once: site_collide_dev (eq = 0,
// after a collision) in paired FP32 instructions (F2), the same explicitly
// rounded operations in the same order, so each site gets the same bits.
// Returns f' - rho_ref W (gp), dS(f'), dS(f_in), rho, and whether each site
// cannot be limited (rho <= 0, some f*_k <= 0, dS not finite).
__device__ __forceinline__ void tube_pair_eval(const TubeK &kk, float rho_ref, const float *rwf, const float2 g[3],
                                               float2 gp[3], float2 &ds, float2 &din, float2 &rho, bool &bad_x,
                                               bool &bad_y)
{
    using O = F2;
    const float2 drho = O::add(O::add(g[0], g[1]), g[2]);
    rho = O::add(O::s(rho_ref), drho);
    const float2 u = O::mul(O::sub(g[2], g[1]), O::rcp_rn(rho));
    const float2 A = O::mul(O::s(1.0f / 6.0f), O::fma(O::mul(O::mul(O::s(3.0f), rho), u), u, drho));
    const float2 B = O::mul(O::mul(O::s(0.5f), rho), u);
    float2 gs[3], n[3];
    gs[1] = O::sub(A, B);
    gs[2] = O::add(A, B);
    gs[0] = O::sub(drho, O::add(gs[1], gs[2]));
#pragma unroll
    for (int k = 0; k < 3; ++k) n[k] = O::sub(g[k], gs[k]);
    const float2 rm = O::add(O::add(n[0], n[1]), n[2]);
    const float2 hx = O::mul(O::s(0.5f), O::sub(n[2], n[1]));
    n[0] = O::sub(n[0], rm);
    n[2] = O::sub(n[2], hx);
    n[1] = O::add(n[1], hx);
    float2 d = O::s(0.f);
    float mx = 3.4e38f, my = 3.4e38f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float2 fsa = O::add(O::s(rwf[k]), gs[k]);
        d = O::fma(O::mul(n[k], n[k]), O::rcp_fast(fsa), d);
        gp[k] = O::fma(O::s(-kk.b2), n[k], g[k]);
        mx = fminf(mx, fsa.x);
        my = fminf(my, fsa.y);
    }
    din = d;
    ds = O::mul(O::s(__fmul_rn(kk.a, kk.a)), d);
    bad_x = !(rho.x > 0.f) || !(mx > 0.f) || !isfinite(ds.x);
    bad_y = !(rho.y > 0.f) || !(my > 0.f) || !isfinite(ds.y);
}

// The sums and counts of one site finished by tube_site32.
struct SiteSums {
    float mass, ds, din, lim;
    int bad, pos, med;
};

// One FP32 site that the paired fast path did not finish (a limiter acts on
// its pair, its lane holds an end of the tube, or the pass is not a
// polynomial collision), from its pull f_in: the evaluation, the positivity
// rule, the three-point median (the neighbours' dS dsl / dsr, or evaluated
// here for the sites xlo / xro outside the warp's chunk, -1 when given), the
// limited or free update, its sums, the Ehrenfests' candidate and the dS
// field.  The operations are those of the tiled kernel's FP32 path.  Not
// inlined: the site's state stays out of the walk's registers.
template <typename S>
__device__ __noinline__ SiteSums tube_site32(const StepParams &p, TubeK kk, const S *__restrict__ src,
                                             S *__restrict__ dst, int x, float f0, float f1, float f2, float dsl,
                                             float dsr, int xlo, int xro, int2 *klist, int *kcount)
{
    SiteSums r{0.f, 0.f, 0.f, 0.f, 0, 0, 0};
    const float fin[3] = {f0, f1, f2};
    float fs[3], fp[3], fa[3], nq[3], ds, dsin, rho;
    const bool bad = tube_eval<float>(p, kk, fin, fs, fp, fa, nq, ds, dsin, rho, true);
    const int nx = p.nx;
    float phi_pos = 1.f, phi_med = 1.f;
    if (!bad) {
        if (p.limiters & 1u) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const float fpa = p.rwf[k] + fp[k];  // absolute f'
                if (fpa < 0.f) phi_pos = fminf(phi_pos, fa[k] / (fa[k] - fpa));
            }
        }
        // three-point median (the two end sites of a closed tube are not
        // filtered; a periodic tube's end sites wrap around to each other)
        const bool end = p.boundary == 0 && (x == 0 || x == nx - 1);
        if ((p.limiters & 4u) && ds > kk.dm && !end) {
            const float left = xlo >= 0 ? tube_ds<S>(p, kk, src, xlo) : dsl;
            const float right = xro >= 0 ? tube_ds<S>(p, kk, src, xro) : dsr;
            phi_med = phi_median<float>(ds, med3(left, ds, right), kk.dm, p.median_mode);
        }
    }
    const float phi = phi_pos < phi_med ? phi_pos : phi_med;
    if (phi < 1.f) {
        const float cw = limit_weight(phi, kk.a, p.collide != 0);
#pragma unroll
        for (int k = 0; k < 3; ++k) dst[tidx(p, k, x)] = fmaf(-cw, nq[k], fin[k]);
        if (p.eq == 1) {
            float dout[3];
            const float m = p.collide ? __fmul_rn(-phi, kk.a) : phi;
#pragma unroll
            for (int k = 0; k < 3; ++k) dout[k] = __fmul_rn(m, nq[k]);
            const float so = rel_entropy_dev<3>(dout, fa);
            if (isfinite(ds) && isfinite(so)) r.lim = __fsub_rn(ds, so);
        } else {
            r.lim = __fmul_rn(__fsub_rn(1.f, __fmul_rn(phi, phi)), ds);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) dst[tidx(p, k, x)] = f2s<S>(fp[k]);
    }
    r.mass = __fsub_rn(rho, p.rho_ref);  // exact
    if (!bad) {
        if (p.eq == 1) {
            if (isfinite(ds)) r.ds = ds;
            if (isfinite(ds) && isfinite(dsin)) r.din = __fsub_rn(dsin, ds);
        } else {
            r.ds = ds;
            r.din = dsin;
        }
    } else {
        r.bad = 1;
        atomicOr(p.status, kStatNonfinite);
    }
    r.pos = phi_pos < 1.f;
    r.med = phi_med < 1.f;
    // Ehrenfests' candidate: near or above the threshold, keyed in FP64 after the chunk
    if ((p.limiters & 2u) && !bad && ds > kk.thr_e) klist[atomicAdd(kcount, 1)] = make_int2(x, __float_as_int(phi));
    if (p.ds_out) p.ds_out[x] = (double)ds;
    return r;
}

// Asynchronous copy of N = 4, 8 or 16 bytes global -> shared (cp.async; the
// 16-byte form bypasses L1), and the per-thread group bookkeeping.
template <int N>
__device__ __forceinline__ void tcopy(void *dst_smem, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
    if constexpr (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(N) : "memory");
}
__device__ __forceinline__ void tcommit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void twait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ double wsum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// V sites per lane, blockDim.x / 32 warps per block.  The grid is at most one
// wave of resident blocks; warp w of the grid takes chunks w, w + W, w + 2W ...
// (W warps in the grid) of 32 V sites each.  Chunks stream through a per-warp
// ring of kTubeRing shared-memory slots filled by asynchronous copies (each
// lane copies its V sites of every plane, lane 0 and lane 31 also the values
// streaming in from the neighbour chunks), kTubeRing - 1 chunks ahead of the
// arithmetic.  `chunked`: the grid has more blocks than one chunk of the
// tail's reduction, so the last block of each kChunkRows blocks sums their
// rows; otherwise the tail reads the block rows.
constexpr int kTubeRing = 3;
constexpr int kTubeWarps = 8;  // the most warps a block has
constexpr int kTubeGroup = 8;  // chunks of a batched work item
constexpr int kTubeBlocks = 2;  // FP32 storage, four sites a lane: resident blocks per SM
// The statistics a warp gathers.  FP64 storage sums FP64 terms per lane.  FP32
// storage: each lane sums its FP32 terms over the whole walk with Kahan's
// compensation (sums s - c; two interleaved chains of a paired instruction for
// mass, dS and dS_in), no lane exchange and no conversion per chunk (FP64 adds
// kept this GPU's FP64 units a third busy; a butterfly and a 128-bit addition a
// chunk were 70 of its 490 instructions).
struct TubeAcc {
    double t_mass, t_ds, t_in, t_lim;
    float2 s_mass, c_mass, s_ds, c_ds, s_in, c_in;
    float s_lim, c_lim;
    int c_pos, c_med, c_bad, c_own;
};

// One compensated addition (Kahan 1965): s - c += v.
__device__ __forceinline__ void kahan2(float2 &s, float2 &c, float2 v)
{
    const float2 y = F2::sub(v, c), t = F2::add(s, y);
    c = F2::sub(F2::sub(t, s), y);
    s = t;
}

// Sum of two unevaluated pairs (hi, lo): Knuth's two-sum of the high parts, the
// low parts and the error renormalised.
__device__ __forceinline__ float2 df_add(float2 a, float2 b)
{
    const float s = __fadd_rn(a.x, b.x), bb = __fsub_rn(s, a.x);
    float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(s, bb)), __fsub_rn(b.x, bb));
    e = __fadd_rn(e, __fadd_rn(a.y, b.y));
    const float hi = __fadd_rn(s, e);
    return make_float2(hi, __fsub_rn(e, __fsub_rn(hi, s)));
}

// FP32 storage: the four totals of the warp's walk, in every lane: a butterfly over
// the lanes' pairs (each of its first two levels halves the sums a lane carries:
// lane 0 ends with mass, 8 dS, 16 dS_in, 24 dS_lim), then one conversion.  V = 1:
// the walk is a single chunk, a site per lane, and plain FP32 additions add it.
template <int V>
__device__ __forceinline__ void tube_totals(const TubeAcc &acc, double &mass, double &ds, double &din, double &lim)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto add = [](float2 a, float2 b) { return V == 1 ? make_float2(__fadd_rn(a.x, b.x), 0.f) : df_add(a, b); };
    auto both = [&](float2 s, float2 c) { return add(make_float2(s.x, -c.x), make_float2(s.y, -c.y)); };
    auto swap = [](float2 v, int o) { return make_float2(__shfl_xor_sync(kAll, v.x, o), __shfl_xor_sync(kAll, v.y, o)); };
    const float2 m = both(acc.s_mass, acc.c_mass), d = both(acc.s_ds, acc.c_ds), i = both(acc.s_in, acc.c_in);
    const float2 l = make_float2(acc.s_lim, -acc.c_lim);
    const bool hi16 = (lane & 16) != 0, hi8 = (lane & 8) != 0;
    const float2 x0 = add(hi16 ? i : m, swap(hi16 ? m : i, 16));
    const float2 x1 = add(hi16 ? l : d, swap(hi16 ? d : l, 16));
    float2 z = add(hi8 ? x1 : x0, swap(hi8 ? x0 : x1, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z = add(z, swap(z, o));
    const double v = (double)z.x + (double)z.y;
    mass = __shfl_sync(kAll, v, 0);
    ds = __shfl_sync(kAll, v, 8);
    din = __shfl_sync(kAll, v, 16);
    lim = __shfl_sync(kAll, v, 24);
}

// a ring slot: the three planes of a chunk of 32 V sites, f_1 with the site right of
// the chunk after it, f_2 with the site left of it in front (padded to 16 bytes)
template <typename S, int V>
struct alignas(16) TubeSlot {
    static constexpr int kPad = 16 / (int)sizeof(S);
    S f0[32 * V], f1[32 * V + kPad], f2[kPad + 32 * V];
};

// An Ehrenfests' candidate into the context's list.
__device__ __forceinline__ void tube_record(const StepParams &p, int x, double key, double phi)
{
    const int slot = atomicAdd(p.cand_count, 1);
    if (slot < p.cand_cap) {
        Cand cd;
        cd.key = key;
        cd.site = x;
        cd.phi = phi;
        cd.ds32 = (float)key;
        p.cand[slot] = cd;
    } else {
        atomicOr(p.status, kStatCandOverflow);
    }
}

// The chunk's sites that the paired fast path of tube_walk did not finish (FP32
// storage; the whole warp).  done: bits 0 and 1, the lane's pairs already finished;
// bit 2, ds_ holds dS of its sites (otherwise evaluated here: a lane that holds an
// end of the tube, or a pass that is not a polynomial collision).  Then the FP64 keys
// of all of the chunk's candidates, a lane each: a chunk holding many of them costs
// one FP64 evaluation per 32, not one per site a lane carries.  Returns the sums of
// the sites finished here; the counts are four bits each (bad, pos, med).
struct ChunkSums {
    float mass, ds, din, lim;
    unsigned counts;
};
template <int V>
__device__ __noinline__ ChunkSums tube_chunk32(const StepParams &p, const TubeK kk, const float *__restrict__ src,
                                               float *__restrict__ dst, const TubeSlot<float, V> *slot, int c,
                                               unsigned done, float4 ds_, int2 *klist, int *kcount)
{
    using S = float;
    const TubeSlot<S, V> &sl = *slot;
    const int lane = threadIdx.x & 31, nx = p.nx, xl = c * 32 * V + lane * V;
    ChunkSums r{0.f, 0.f, 0.f, 0.f, 0u};
    float ds[V];
#pragma unroll
    for (int j = 0; j < V; ++j) ds[j] = j == 0 ? ds_.x : (j == 1 ? ds_.y : (j == 2 ? ds_.z : ds_.w));
    // the lane's pull of its site j (free flight with the tube's ends, or the stored
    // values of a limiter pass)
    auto build_fin = [&](int j, float f3[3]) {
        const int x = xl + j, i = lane * V + j;
        f3[0] = sl.f0[i];
        if (p.collide) {
            f3[1] = sl.f1[i + 1];
            f3[2] = sl.f2[TubeSlot<S, V>::kPad + i - 1];
            if (x == nx - 1)  // right end: reflect or wrap
                f3[1] = bc_wrap_x(p.boundary) ? src[tidx(p, 1, 0)] : sl.f2[TubeSlot<S, V>::kPad + i];
            if (x == 0)  // left end
                f3[2] = bc_wrap_x(p.boundary) ? src[tidx(p, 2, nx - 1)] : sl.f1[i];
        } else {
            f3[1] = sl.f1[i];
            f3[2] = sl.f2[TubeSlot<S, V>::kPad + i];
        }
    };
    if (!(done & 4u)) {
#pragma unroll 1
        for (int j = 0; j < V; ++j) {
            float d = 0.f;
            if (xl + j < nx) {
                float f3[3], fs3[3], fp3[3], fa3[3], nq3[3], din, rho;
                build_fin(j, f3);
                tube_eval<float>(p, kk, f3, fs3, fp3, fa3, nq3, d, din, rho, false);
            }
#pragma unroll
            for (int i = 0; i < V; ++i)
                if (i == j) ds[i] = d;
        }
    }
    __syncwarp();
    // the median's neighbours: dS of the adjacent lanes' edge sites
    const float dl_lane = __shfl_up_sync(0xffffffffu, ds[V - 1], 1);
    const float dr_lane = __shfl_down_sync(0xffffffffu, ds[0], 1);
#pragma unroll 1
    for (int j = 0; j < V; ++j) {
        const int x = xl + j;
        if (x >= nx) break;
        // this site's dS and its neighbours', or the site to evaluate (outside the chunk)
        float d = ds[0], dl = dl_lane, dr = dr_lane;
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (i == j) {
                d = ds[i];
                if (i > 0) dl = ds[i - 1];
                if (i + 1 < V) dr = ds[i + 1];
            }
        if ((done >> (j >> 1)) & 1u) {
            if ((p.limiters & 2u) && d > kk.thr_e) klist[atomicAdd(kcount, 1)] = make_int2(x, __float_as_int(1.f));
            continue;
        }
        int xlo = -1, xro = -1;
        if (x == 0)
            xlo = nx - 1;
        else if (j == 0 && lane == 0)
            xlo = x - 1;
        if (x == nx - 1)
            xro = 0;
        else if (j == V - 1 && lane == 31)
            xro = x + 1;
        float f3[3];
        build_fin(j, f3);
        const SiteSums q = tube_site32<S>(p, kk, src, dst, x, f3[0], f3[1], f3[2], dl, dr, xlo, xro, klist, kcount);
        r.mass = __fadd_rn(r.mass, q.mass);
        r.ds = __fadd_rn(r.ds, q.ds);
        r.din = __fadd_rn(r.din, q.din);
        r.lim = __fadd_rn(r.lim, q.lim);
        r.counts += (unsigned)q.bad | (unsigned)q.pos << 4 | (unsigned)q.med << 8;
    }
    __syncwarp();
    const int nk = *kcount;
    for (int i = lane; i < nk; i += 32) {
        const int2 e = klist[i];
        double fin64[3], fs64[3], fp64[3], d64, din64, r64;
        if (p.collide)
            tube_pull<S, double>(p, src, e.x, fin64);
        else
            tube_read<S, double>(p, src, e.x, fin64);
        const bool b64 = site_collide<3, double>(fin64, p.a, p.collide != 0, fs64, fp64, d64, din64, r64, p.eq, false);
        if (!b64 && d64 > p.delta_e) tube_record(p, e.x, d64, (double)__int_as_float(e.y));
    }
    __syncwarp();
    if (lane == 0) *kcount = 0;
    __syncwarp();
    return r;
}

// One warp's walk over chunks c0, c0 + stride, ... (< c_end) of lattice p:
// a1-a9 at every site, the Ehrenfests' candidates, the sums into acc.  `my`:
// the warp's ring; klist / kcount: the warp's candidate list (FP32 storage).
// Every lane of the warp takes part.
template <typename S, int V>
__device__ __forceinline__ void tube_walk(const StepParams &p, const S *__restrict__ src, S *__restrict__ dst,
                                          int c0, int stride, int c_end, TubeSlot<S, V> *my, int2 *klist,
                                          int *kcount, TubeAcc &acc)
{
    using T = compute_t<S>;
    using A = Ar<T>;
    using Slot = TubeSlot<S, V>;
    constexpr bool F64 = std::is_same<T, double>::value;
    constexpr int CW = 32 * V;  // sites of a chunk
    const int lane = threadIdx.x & 31;
    const int nx = p.nx;
    TubeK kk{};
    if constexpr (!F64) {
        kk.a = (float)p.a;
        kk.b2 = (float)(1.0 + p.a);
        kk.dm = (float)p.delta_m;
        kk.thr_e = (float)(p.delta_e * (1.0 - 1.0 / 64.0));
    }
    // the fast path's flags and constants in registers (the batched kernel's lie in
    // shared memory)
    const bool fast = V == 4 && !F64 && p.collide && p.eq == 0 && !p.ds_out;
    const bool lim_pos = (p.limiters & 1u) != 0, lim_ehr = (p.limiters & 2u) != 0, lim_med = (p.limiters & 4u) != 0;
    const float rho_ref = p.rho_ref, rwf[3] = {p.rwf[0], p.rwf[1], p.rwf[2]};
    const float d_act = lim_med ? kk.dm : INFINITY, d_cand = lim_ehr ? kk.thr_e : INFINITY;

    // copies of chunk c into slot `sl` (nothing past the last chunk; the group
    // is committed either way).  The chunk's window lies inside the padded row
    // (kTail zero elements follow the lattice), so whole vectors may be copied
    // past its end.
    auto issue = [&](int c, int sl) {
        if (c < c_end) {
            const int x0 = c * CW, xl = x0 + lane * V;
            if (xl < nx) {
                tcopy<(int)sizeof(S) * V>(&my[sl].f0[lane * V], src + tidx(p, 0, xl));
                tcopy<(int)sizeof(S) * V>(&my[sl].f1[lane * V], src + tidx(p, 1, xl));
                tcopy<(int)sizeof(S) * V>(&my[sl].f2[Slot::kPad + lane * V], src + tidx(p, 2, xl));
            }
            if (lane == 0 && x0 > 0) tcopy<(int)sizeof(S)>(&my[sl].f2[Slot::kPad - 1], src + tidx(p, 2, x0 - 1));
            if (lane == 31 && xl + V < nx) tcopy<(int)sizeof(S)>(&my[sl].f1[32 * V], src + tidx(p, 1, xl + V));
        }
        tcommit();
    };

#pragma unroll
    for (int i = 0; i < kTubeRing - 1; ++i) issue(c0 + i * stride, i);
    int get = 0;
    for (int c = c0; c < c_end; c += stride) {
        __syncwarp();                                                   // every lane is done with the slot refilled now
        issue(c + (kTubeRing - 1) * stride, get == 0 ? kTubeRing - 1 : get - 1);
        twait<kTubeRing - 1>();                                         // this lane's copies of chunk c have landed
        __syncwarp();                                                   // and so have the other lanes'
        const Slot &sl = my[get];
        get = get + 1 == kTubeRing ? 0 : get + 1;
        const int x0 = c * CW, xl = x0 + lane * V;
        if constexpr (!F64) {
            // the chunk's sums: the pairs' interleaved terms; the sites finished by tube_chunk32
            float2 m2 = F2::s(0.f), d2s = F2::s(0.f), i2s = F2::s(0.f);
            unsigned done = 0u;
            bool rest = true;
            float4 ds = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (V == 4) {
                if (fast) {
                    const float4 f0 = *reinterpret_cast<const float4 *>(&sl.f0[lane * V]);
                    const float4 f1 = *reinterpret_cast<const float4 *>(&sl.f1[lane * V]);
                    const float4 f2 = *reinterpret_cast<const float4 *>(&sl.f2[Slot::kPad + lane * V]);
                    const float r1 = sl.f1[lane * V + V], l2 = sl.f2[Slot::kPad + lane * V - 1];
                    const float2 ga[3] = {make_float2(f0.x, f0.y), make_float2(f1.y, f1.z), make_float2(l2, f2.x)};
                    const float2 gb[3] = {make_float2(f0.z, f0.w), make_float2(f1.w, r1), make_float2(f2.y, f2.z)};
                    float2 pa[3], pb[3], da, db, ia, ib, ra, rb;
                    bool ba, bb, bc, bd;
                    tube_pair_eval(kk, rho_ref, rwf, ga, pa, da, ia, ra, ba, bb);
                    tube_pair_eval(kk, rho_ref, rwf, gb, pb, db, ib, rb, bc, bd);
                    // a pair on which something acts: a bad site, a negative f' of the
                    // positivity rule, dS above the median filter's delta
                    bool act_a = ba || bb || fmaxf(da.x, da.y) > d_act, act_b = bc || bd || fmaxf(db.x, db.y) > d_act;
                    if (lim_pos) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            act_a = act_a || fminf(rwf[k] + pa[k].x, rwf[k] + pa[k].y) < 0.f;
                            act_b = act_b || fminf(rwf[k] + pb[k].x, rwf[k] + pb[k].y) < 0.f;
                        }
                    }
                    const bool inside = xl >= 1 && xl + V <= nx - 1;
                    const bool cand = fmaxf(fmaxf(da.x, da.y), fmaxf(db.x, db.y)) > d_cand;
                    rest = __any_sync(0xffffffffu, act_a || act_b || cand || !inside);
                    const float2 ma = F2::sub(ra, F2::s(rho_ref)), mb = F2::sub(rb, F2::s(rho_ref));  // exact
                    float *const to = dst + tidx(p, 0, xl);
                    if (!rest) {
#pragma unroll
                        for (int k = 0; k < 3; ++k)
                            *reinterpret_cast<float4 *>(to + k * p.plane) =
                                make_float4(pa[k].x, pa[k].y, pb[k].x, pb[k].y);
                        m2 = F2::add(ma, mb);
                        d2s = F2::add(da, db);
                        i2s = F2::add(ia, ib);
                    } else if (inside) {
                        // a site that cannot be limited has dS = +inf (as tube_eval gives it)
                        ds = make_float4(ba ? INFINITY : da.x, bb ? INFINITY : da.y, bc ? INFINITY : db.x,
                                         bd ? INFINITY : db.y);
                        done = 4u;
                        if (!act_a) {
                            done |= 1u;
#pragma unroll
                            for (int k = 0; k < 3; ++k) *reinterpret_cast<float2 *>(to + k * p.plane) = pa[k];
                            m2 = ma;
                            d2s = da;
                            i2s = ia;
                        }
                        if (!act_b) {
                            done |= 2u;
#pragma unroll
                            for (int k = 0; k < 3; ++k) *reinterpret_cast<float2 *>(to + k * p.plane + 2) = pb[k];
                            m2 = F2::add(m2, mb);
                            d2s = F2::add(d2s, db);
                            i2s = F2::add(i2s, ib);
                        }
                    }
                }
            }
            if (rest) {
                const ChunkSums r = tube_chunk32<V>(p, kk, src, dst, &sl, c, done, ds, klist, kcount);
                m2.x = __fadd_rn(m2.x, r.mass);
                d2s.x = __fadd_rn(d2s.x, r.ds);
                i2s.x = __fadd_rn(i2s.x, r.din);
                const float y = __fsub_rn(r.lim, acc.c_lim), t = __fadd_rn(acc.s_lim, y);
                acc.c_lim = __fsub_rn(__fsub_rn(t, acc.s_lim), y);
                acc.s_lim = t;
                acc.c_bad += (int)(r.counts & 15u);
                acc.c_pos += (int)(r.counts >> 4 & 15u);
                acc.c_med += (int)(r.counts >> 8 & 15u);
            }
            kahan2(acc.s_mass, acc.c_mass, m2);
            kahan2(acc.s_ds, acc.c_ds, d2s);
            kahan2(acc.s_in, acc.c_in, i2s);
            acc.c_own += max(0, min(V, nx - xl));
        } else {
            const S r1 = sl.f1[lane * V + V], l2 = sl.f2[Slot::kPad + lane * V - 1];
            double ds[V], fin[V][3], fs[V][3], fp[V][3], dsin[V], rho[V];
            double s_mass = 0.0, s_ds = 0.0, s_in = 0.0, s_lim = 0.0;
            bool bad[V];
#pragma unroll
            for (int j = 0; j < V; ++j) {
                const int x = xl + j, i = lane * V + j;
                ds[j] = 0.0;
                dsin[j] = 0.0;
                rho[j] = 0.0;
                bad[j] = false;
                if (x >= nx) continue;
                fin[j][0] = sl.f0[i];
                if (p.collide) {
                    fin[j][1] = j + 1 < V ? sl.f1[i + 1] : r1;
                    fin[j][2] = j > 0 ? sl.f2[Slot::kPad + i - 1] : l2;
                    if (x == nx - 1)  // right end: reflect or wrap
                        fin[j][1] = bc_wrap_x(p.boundary) ? src[tidx(p, 1, 0)] : sl.f2[Slot::kPad + i];
                    if (x == 0)  // left end
                        fin[j][2] = bc_wrap_x(p.boundary) ? src[tidx(p, 2, nx - 1)] : sl.f1[i];
                } else {
                    fin[j][1] = sl.f1[i];
                    fin[j][2] = sl.f2[Slot::kPad + i];
                }
                bad[j] = site_collide<3, double>(fin[j], p.a, p.collide != 0, fs[j], fp[j], ds[j], dsin[j], rho[j],
                                                 p.eq, true, p.coll, p.beta);
                if (bad[j]) ds[j] = INFINITY;
            }

            // the median's neighbours: dS of the adjacent lanes' edge sites
            const double dl_lane = __shfl_up_sync(0xffffffffu, ds[V - 1], 1);
            const double dr_lane = __shfl_down_sync(0xffffffffu, ds[0], 1);

#pragma unroll
            for (int j = 0; j < V; ++j) {
                const int x = xl + j;
                if (x >= nx) continue;
                ++acc.c_own;
                double phi_pos = 1.0, phi_med = 1.0;
                if (!bad[j]) {
                    if (lim_pos) phi_pos = phi_positivity<3, double>(fs[j], fp[j]);
                    // three-point median (the two end sites of a closed tube are not
                    // filtered; a periodic tube's end sites wrap around to each other)
                    const bool end = p.boundary == 0 && (x == 0 || x == nx - 1);
                    if (lim_med && ds[j] > p.delta_m && !end) {
                        double left, right;
                        if (x == 0)
                            left = tube_ds<S>(p, kk, src, nx - 1);
                        else if (j > 0)
                            left = ds[j - 1];
                        else if (lane > 0)
                            left = dl_lane;
                        else
                            left = tube_ds<S>(p, kk, src, x - 1);
                        if (x == nx - 1)
                            right = tube_ds<S>(p, kk, src, 0);
                        else if (j + 1 < V)
                            right = ds[j + 1];
                        else if (lane < 31)
                            right = dr_lane;
                        else
                            right = tube_ds<S>(p, kk, src, x + 1);
                        const double med = med3(left, ds[j], right);
                        phi_med = (p.phi_rule == 1 && p.eq == 1)
                                      ? phi_median_entropy<3>(fp[j], fs[j], ds[j], med, p.delta_m, p.median_mode)
                                      : phi_median<double>(ds[j], med, p.delta_m, p.median_mode);
                    }
                }
                const double phi = phi_pos < phi_med ? phi_pos : phi_med;
                double lim = 0.0;
                if (phi < 1.0) {
                    double fo[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        fo[k] = A::add(fs[j][k], A::mul(phi, A::sub(fp[j][k], fs[j][k])));
                        dst[tidx(p, k, x)] = fo[k];
                    }
                    if (p.eq == 1) {
                        const double dout = rel_entropy<3>(fo, fs[j]);
                        if (isfinite(ds[j]) && isfinite(dout)) lim = A::sub(ds[j], dout);
                    } else {
                        lim = A::mul(A::sub(1.0, A::mul(phi, phi)), ds[j]);
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 3; ++k) dst[tidx(p, k, x)] = fp[j][k];
                }
                s_lim = A::add(s_lim, lim);
                s_mass = A::add(s_mass, rho[j]);
                if (!bad[j]) {
                    double tds = 0.0, tin = 0.0;
                    if (p.eq == 1) {
                        if (isfinite(ds[j])) tds = ds[j];
                        if (isfinite(ds[j]) && isfinite(dsin[j])) tin = A::sub(dsin[j], ds[j]);
                    } else {
                        tds = ds[j];
                        tin = dsin[j];
                    }
                    s_ds = A::add(s_ds, tds);
                    s_in = A::add(s_in, tin);
                } else {
                    ++acc.c_bad;
                    atomicOr(p.status, kStatNonfinite);
                }
                acc.c_pos += phi_pos < 1.0;
                acc.c_med += phi_med < 1.0;
                // Ehrenfests' candidates on dS(f') itself
                if (lim_ehr && !bad[j] && ds[j] > p.delta_e) tube_record(p, x, ds[j], phi);
                if (p.ds_out) p.ds_out[x] = ds[j];
            }
            acc.t_mass = A::add(acc.t_mass, s_mass);
            acc.t_ds = A::add(acc.t_ds, s_ds);
            acc.t_in = A::add(acc.t_in, s_in);
            acc.t_lim = A::add(acc.t_lim, s_lim);
        }
    }
    twait<0>();
}

template <typename S, int V>
__global__ void __launch_bounds__(256, V == 4 ? kTubeBlocks : (V > 1 ? 2 : 1))
    k_tube(const __grid_constant__ StepParams p, const S *__restrict__ src, S *__restrict__ dst, int chunked)
{
    constexpr bool F64 = std::is_same<compute_t<S>, double>::value;
    __shared__ TubeSlot<S, V> ring[kTubeWarps][kTubeRing];
    // FP32 storage: the chunk's sites whose FP32 dS(f') lies near or above the
    // threshold (site, phi), keyed in FP64 after the chunk with one lane each:
    // a chunk holding many of them costs one FP64 evaluation per 32, not one per
    // site a lane carries
    __shared__ int2 klist[kTubeWarps][F64 ? 1 : 32 * V];
    __shared__ int kcount[kTubeWarps];
    // the tail of the previous pass may still run (programmatic launch)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) kcount[warp] = 0;
    __syncwarp();
    TubeAcc acc{};
    tube_walk<S, V>(p, src, dst, blockIdx.x * nw + warp, (int)gridDim.x * nw, (p.nx + 32 * V - 1) / (32 * V),
                    ring[warp], klist[warp], &kcount[warp], acc);
    double t_mass = acc.t_mass, t_ds = acc.t_ds, t_in = acc.t_in, t_lim = acc.t_lim;
    if constexpr (!F64) tube_totals<V>(acc, t_mass, t_ds, t_in, t_lim);
    int c_pos = acc.c_pos, c_med = acc.c_med, c_bad = acc.c_bad, c_own = acc.c_own;

    // block partial row: warp sums, then the warps in order; counts as integers
    __shared__ double sred[kTubeWarps][P_NSTAT];
    if constexpr (F64) {
        t_mass = wsum(t_mass);
        t_ds = wsum(t_ds);
        t_in = wsum(t_in);
        t_lim = wsum(t_lim);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c_pos += __shfl_down_sync(0xffffffffu, c_pos, o);
        c_med += __shfl_down_sync(0xffffffffu, c_med, o);
        c_bad += __shfl_down_sync(0xffffffffu, c_bad, o);
        c_own += __shfl_down_sync(0xffffffffu, c_own, o);
    }
    if (lane == 0) {
        sred[warp][P_MASS] = F64 ? t_mass : (double)p.rho_ref * (double)c_own + t_mass;
        sred[warp][P_SUM_DS] = t_ds;
        sred[warp][P_SUM_IN] = t_in;
        sred[warp][P_DS_LIM] = t_lim;
        sred[warp][P_NPOS] = (double)c_pos;
        sred[warp][P_NMED] = (double)c_med;
        sred[warp][P_NBAD] = (double)c_bad;
    }
    __syncthreads();
    const int bid = blockIdx.x, tid = threadIdx.x;
    if (tid < P_NSTAT) {
        double v = sred[0][tid];
        for (int w = 1; w < nw; ++w) v += sred[w][tid];
        p.partials[(long long)bid * P_NSTAT + tid] = v;
    }
    if (!chunked) return;
    // the last block of each chunk of kChunkRows blocks sums the chunk's rows in
    // row order (a ticket, no waiting)
    __shared__ int s_last;
    const int chunk = bid / kChunkRows;
    const int rows = min(kChunkRows, (int)gridDim.x - chunk * kChunkRows);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(p.chunk_cnt + chunk, 1u) == (unsigned)(rows - 1);
    __syncthreads();
    if (s_last) {
        __threadfence();
        const double *base = p.partials + (long long)chunk * kChunkRows * P_NSTAT;
        for (int stat = warp; stat < P_NSTAT; stat += nw) {
            double v = 0.0;
            for (int r = lane; r < rows; r += 32) v += __ldcg(base + (long long)r * P_NSTAT + stat);
            v = wsum(v);
            if (lane == 0) p.partials2[(long long)chunk * P_NSTAT + stat] = v;
        }
        if (tid == 0) p.chunk_cnt[chunk] = 0u;  // for the next launch
    }
}

// Batched tubes (FP32 storage): work item i is group map[i].y (kTubeGroup
// chunks of 128 sites) of tube map[i].x of `table`; a warp runs its first item
// (its index in the grid), then takes items from the counter *work (cleared by
// the first tube's tail).  It keeps its tube's arguments in shared memory and
// writes each item's sums into the tube's partial row of that group (a fixed
// evaluation order per item, so the sums do not depend on which warp ran it).
template <int V>
__global__ void __launch_bounds__(256, kTubeBlocks) k_tube_batched(const TubeArgs *__restrict__ table,
                                                         const int2 *__restrict__ map, int items, int *work)
{
    using S = float;
    __shared__ TubeSlot<S, V> ring[kTubeWarps][kTubeRing];
    __shared__ int2 klist[kTubeWarps][32 * V];
    __shared__ int kcount[kTubeWarps];
    __shared__ __align__(16) TubeArgs sA[kTubeWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) kcount[warp] = 0;
    __syncwarp();
    int cur = -1;
    int item = blockIdx.x * nw + warp;
    while (item < items) {
        const int2 m = map[item];
        if (m.x != cur) {
            __syncwarp();
            const unsigned *from = reinterpret_cast<const unsigned *>(table + m.x);
            unsigned *to = reinterpret_cast<unsigned *>(&sA[warp]);
            for (int i = lane; i < (int)(sizeof(TubeArgs) / 4); i += 32) to[i] = from[i];
            __syncwarp();
            cur = m.x;
        }
        const StepParams &p = sA[warp].p;
        const int nch = (p.nx + 32 * V - 1) / (32 * V);
        const int c0 = m.y * kTubeGroup, c1 = min(c0 + kTubeGroup, nch);
        TubeAcc acc{};
        tube_walk<S, V>(p, (const S *)sA[warp].src, (S *)sA[warp].dst, c0, 1, c1, ring[warp], klist[warp],
                               &kcount[warp], acc);
        // the item's totals; the counts are per lane
        double t_mass, t_ds, t_in, t_lim;
        tube_totals<V>(acc, t_mass, t_ds, t_in, t_lim);
        const int c_pos = __reduce_add_sync(0xffffffffu, acc.c_pos), c_med = __reduce_add_sync(0xffffffffu, acc.c_med);
        const int c_bad = __reduce_add_sync(0xffffffffu, acc.c_bad), c_own = __reduce_add_sync(0xffffffffu, acc.c_own);
        if (lane == 0) {
            double *row = p.partials + (long long)m.y * P_NSTAT;
            row[P_MASS] = (double)p.rho_ref * (double)c_own + t_mass;
            row[P_SUM_DS] = t_ds;
            row[P_SUM_IN] = t_in;
            row[P_DS_LIM] = t_lim;
            row[P_NPOS] = (double)c_pos;
            row[P_NMED] = (double)c_med;
            row[P_NBAD] = (double)c_bad;
        }
        int next = 0;
        if (lane == 0) next = (int)gridDim.x * nw + atomicAdd(work, 1);
        item = __shfl_sync(0xffffffffu, next, 0);
    }
}

// Launch shape: sites per lane, warps per block and blocks.  A tube of up to
// one chunk per SM sub-partition (4 x 152 chunks of 32 sites) runs one site per
// lane and a warp per block; longer tubes take 16-byte vectors (FP32 4 sites a
// lane, FP64 2) in blocks of 8 / 4 warps, at most one wave of resident blocks.
struct TubeShape {
    int v, warps, blocks;
};

template <typename S, int V>
int resident_blocks(int threads)
{
    static int per_sm = 0;
    if (per_sm == 0 &&
        (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tube<S, V>, threads, 0) != cudaSuccess || per_sm < 1)) {
        cudaGetLastError();
        per_sm = 2;
    }
    return per_sm * sm_count();
}

TubeShape tube_shape(bool fp64, int nx, bool launch)
{
    TubeShape t{};
    const long long slots = 4LL * sm_count();
    if ((long long)nx <= 32 * slots) {
        t.v = 1;
        t.warps = 1;
    } else {
        t.v = fp64 ? 2 : 4;
        t.warps = fp64 ? 4 : 8;
    }
    const long long per_block = 32LL * t.v * t.warps;
    long long blocks = (nx + per_block - 1) / per_block;
    if (t.v > 1) {
        // one wave: the occupancy of the kernel when launching, a bound (every
        // SM full of blocks of this size) when sizing the partial-sum rows
        const long long cap = !launch ? 2048LL / (32 * t.warps) * sm_count()
                                      : (fp64 ? resident_blocks<double, 2>(32 * t.warps)
                                              : resident_blocks<float, 4>(32 * t.warps));
        blocks = std::min(blocks, cap);
    }
    t.blocks = (int)blocks;
    return t;
}

}  // namespace

bool tube_applies(const lbm_config &c, unsigned limiters)
{
    return c.lattice == LBM_D1Q3 && (c.precision == LBM_FP64 || c.precision == LBM_FP32) &&
           (c.boundary == LBM_BC_WALLS || c.boundary == LBM_BC_PERIODIC) && !(limiters & kLimEnsemble) &&
           (c.kernel == LBM_KERNEL_AUTO || c.kernel == LBM_KERNEL_TUBE);
}

int tube_blocks(bool fp64, int nx) { return tube_shape(fp64, nx, false).blocks; }

template <typename S>
cudaError_t launch_tube(const StepParams &p, const S *src, S *dst, int *nblocks, bool *chunked, cudaStream_t s)
{
    constexpr bool fp64 = std::is_same<S, double>::value;
    const TubeShape t = tube_shape(fp64, p.nx, true);
    const int ch = t.blocks > kChunkRows ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)t.blocks);
    cfg.blockDim = dim3((unsigned)(32 * t.warps));
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaError_t e;
    if constexpr (fp64)
        e = t.v == 1 ? cudaLaunchKernelEx(&cfg, k_tube<S, 1>, p, src, dst, ch)
                     : cudaLaunchKernelEx(&cfg, k_tube<S, 2>, p, src, dst, ch);
    else
        e = t.v == 1 ? cudaLaunchKernelEx(&cfg, k_tube<S, 1>, p, src, dst, ch)
                     : cudaLaunchKernelEx(&cfg, k_tube<S, 4>, p, src, dst, ch);
    *nblocks = t.blocks;
    *chunked = ch != 0;
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

int tube_groups(int nx) { return (nx + 128 * kTubeGroup - 1) / (128 * kTubeGroup); }

cudaError_t launch_tube_batched(const TubeArgs *table, const int2 *map, int items, int *work, cudaStream_t s)
{
    if (items <= 0) return cudaSuccess;
    static int per_sm = 0;
    if (per_sm == 0 &&
        (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tube_batched<4>, 256, 0) != cudaSuccess || per_sm < 1)) {
        cudaGetLastError();
        per_sm = 1;
    }
    const int blocks = std::min((items + kTubeWarps - 1) / kTubeWarps, per_sm * sm_count());
    k_tube_batched<4><<<blocks, 32 * kTubeWarps, 0, s>>>(table, map, items, work);
    return cudaGetLastError();
}

template cudaError_t launch_tube<float>(const StepParams &, const float *, float *, int *, bool *, cudaStream_t);
template cudaError_t launch_tube<double>(const StepParams &, const double *, double *, int *, bool *, cudaStream_t);

}  // namespace lbm
