// resident.cuh -- what the kernels that take many steps in one launch share
// (step_resident.cu, step_cluster.cu): a site's evaluation, the sums of a block.
#pragma once

#include <type_traits>

#include "internal.h"
#include "lattice.cuh"
#include "select.cuh"
#include "site.cuh"

namespace lbm {
namespace {

// FP32 parameters, converted once per thread.
struct ResK {
    float a, b2, dm, thr_e;
};

// What a site gives the finishing code.
template <int Q, typename T>
struct SiteState {
    T fin[Q], fs[Q], fp[Q];
    float nq[Q];  // FP32
    float fa[Q];  // FP32: absolute f*
    T ds, dsin, rho;
    bool bad;
};

template <int Q, typename S>
__device__ __forceinline__ void eval_site(const StepParams &p, const ResK &kk, SiteState<Q, compute_t<S>> &v, bool need_in)
{
    using T = compute_t<S>;
    if constexpr (std::is_same<T, double>::value) {
        v.bad = site_poly64<Q>(v.fin, p.a, true, v.fs, v.fp, v.ds, v.dsin, v.rho, need_in);
    } else {
        v.bad = site_collide_dev<Q>(v.fin, kk.a, kk.b2, true, p.rho_ref, p.rwf, v.fs, v.nq, v.fp, v.fa, v.ds, v.dsin,
                                    v.rho, 0);
    }
    if (v.bad) v.ds = T(INFINITY);
}

// A sum.  FP64: plain additions.  FP32: the rounding error of each addition is kept
// beside the sum (Knuth's two-sum) up to the block's row, which is FP64: a thread sums
// several sites and a boundary node's populations, and the sums are to be no less
// accurate than those of the kernels that take one step a launch, which go to FP64
// after one site a lane.  The errors are added apart and not renormalised into the
// sum, so a level of a tree waits for one addition, not for eight (100 x 100
// cavity with boundary nodes: 3.8 us a step, 3.9 with renormalised pairs, 3.5 with no
// errors kept).
template <typename T>
struct SumOf {
    T v = T(0);
    using Total = T;
    __device__ __forceinline__ void add(T x) { v = Ar<T>::add(v, x); }
    __device__ __forceinline__ Total total() const { return v; }
    static __device__ __forceinline__ Total plus(Total a, Total b, bool) { return Ar<T>::add(a, b); }
    static __device__ __forceinline__ Total from(Total a, int o) { return __shfl_xor_sync(kFull, a, o); }
};
template <>
struct SumOf<float> {
    float v = 0.f, c = 0.f;
    using Total = float2;
    __device__ __forceinline__ void add(float x)
    {
        const Total t = plus(total(), make_float2(x, 0.f), false);
        v = t.x;
        c = t.y;
    }
    __device__ __forceinline__ Total total() const { return make_float2(v, c); }
    static __device__ __forceinline__ Total plus(Total a, Total b, bool plain)
    {
        const float t = __fadd_rn(a.x, b.x), z = __fsub_rn(t, a.x);
        const float e = __fadd_rn(__fsub_rn(a.x, __fsub_rn(t, z)), __fsub_rn(b.x, z));
        return make_float2(t, plain ? 0.f : __fadd_rn(__fadd_rn(a.y, b.y), e));
    }
    static __device__ __forceinline__ Total from(Total a, int o)
    {
        return make_float2(__shfl_xor_sync(kFull, a.x, o), __shfl_xor_sync(kFull, a.y, o));
    }
};

// Sums of the worker's sites of one step (per thread).
template <typename T>
struct ResSums {
    SumOf<T> mass, ds, din, lim;
    int pos = 0, med = 0, bad = 0;
};

// A boundary node's share of the mass (FP32: of the deviations; see rest_mass).
template <typename T>
__device__ __forceinline__ void add_wall_mass(const StepParams &p, int x, int y, const T fin[9], SumOf<T> &mass)
{
    if constexpr (std::is_same<T, double>::value) {
        mass.add(wall_mass<T>(p, x, y, fin));
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k)
            if (wall_counts(p, x, y, k)) mass.add(fin[k]);
    }
}

// The sums of a warp's step, into lanes 0 (mass), 8 (dS), 16 (dS_in), 24 (dS_lim):
// a butterfly in which each level halves the sums a lane carries.  `plain` (FP32): plain
// additions, for tubes with one site a lane, whose sums are then rounded as those of the
// kernels that take one step a launch are.
template <typename T>
__device__ __forceinline__ typename SumOf<T>::Total warp_totals(const ResSums<T> &s, int lane, bool plain)
{
    using O = SumOf<T>;
    using V = typename O::Total;
    const V mass = s.mass.total(), ds = s.ds.total(), din = s.din.total(), lim = s.lim.total();
    const bool hi16 = (lane & 16) != 0, hi8 = (lane & 8) != 0;
    const V a0 = O::plus(hi16 ? din : mass, O::from(hi16 ? mass : din, 16), plain);
    const V a1 = O::plus(hi16 ? lim : ds, O::from(hi16 ? ds : lim, 16), plain);
    V z = O::plus(hi8 ? a1 : a0, O::from(hi8 ? a0 : a1, 8), plain);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) z = O::plus(z, O::from(z, o), plain);
    return z;
}

// A block's sums of one step, gathered warp by warp.
template <int NW, typename T>
struct BlockAcc {
    typename SumOf<T>::Total part[NW][4];  // the warps' sums
    int cnt[3];     // positivity, median, flagged sites
    int ticket;
    __device__ void clear()
    {
        for (int i = 0; i < 3; ++i) cnt[i] = 0;
        ticket = 0;
    }
};

// Adds a warp's sums; true in the last of the block's `warps` warps to come.
template <int NW, typename T>
__device__ __forceinline__ bool add_warp(BlockAcc<NW, T> &w, const ResSums<T> &sum, int warps, bool plain)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const typename SumOf<T>::Total z = warp_totals<T>(sum, lane, plain);
    if ((lane & 7) == 0) w.part[warp][lane >> 3] = z;
    if (__any_sync(kFull, (sum.pos | sum.med | sum.bad) != 0)) {
        const int pos = __reduce_add_sync(kFull, sum.pos), med = __reduce_add_sync(kFull, sum.med);
        const int bad = __reduce_add_sync(kFull, sum.bad);
        if (lane < 3) atomicAdd(&w.cnt[lane], lane == 0 ? pos : (lane == 1 ? med : bad));
    }
    __threadfence_block();
    __syncwarp();
    int last = 0;
    if (lane == 0) last = atomicAdd(&w.ticket, 1) == warps - 1;
    if (!__shfl_sync(kFull, last, 0)) return false;
    __threadfence_block();
    return true;
}

// The last warp writes the block's row and clears the sums, added in a fixed order: FP64
// parts in warp order, FP32 parts as pairs by a tree (lane l takes parts l and l + 32,
// lanes with one statistic are added by shuffles), whose two halves FP64 then adds.
template <int NW, typename T>
__device__ __forceinline__ void take_row(BlockAcc<NW, T> &w, ResRow *row, int warps)
{
    const int lane = threadIdx.x & 31;
    double v = 0.0;
    if constexpr (std::is_same<T, double>::value) {
        if (lane < 4)
            for (int j = 0; j < warps; ++j) v = Ar<double>::add(v, w.part[j][lane]);
    } else {
        static_assert(NW <= 16, "two parts a lane");
        using O = SumOf<float>;
        const float2 none = make_float2(0.f, 0.f);
        float2 z = O::plus(lane >> 2 < warps ? w.part[lane >> 2][lane & 3] : none,
                           8 + (lane >> 2) < warps ? w.part[8 + (lane >> 2)][lane & 3] : none, false);
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) z = O::plus(z, O::from(z, o), false);
        v = Ar<double>::add(widen(z.x), widen(z.y));
    }
    if (lane < 4) row->v[lane] = v;
    if (lane < 3) row->c[lane] = w.cnt[lane];
    __syncwarp();
    if (lane == 0) w.clear();
    __syncwarp();
}

// The sums of a step from its block rows (lane r, r + 32, ... of each of the first
// four warps' statistic, or one warp for all four).
__device__ __forceinline__ void sum_rows(const ResRow *rows, int n, int stat, double &v, int &c)
{
    const int lane = threadIdx.x & 31;
    v = 0.0;
    c = 0;
    for (int r = lane; r < n; r += 32) {
        v += __ldcg(&rows[r].v[stat]);
        c += __ldcg(&rows[r].c[stat]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    c = __reduce_add_sync(kFull, c);
}

// The stats record of a step from its sums (tot: P_MASS .. P_DS_LIM, cnt: positivity,
// median, flagged sites).  `status`: the recorder's copy of the status word, read
// when the launch begins and brought on with each step's own flagged sites.  A read of
// the word itself would see those of later steps: the other blocks are ahead of the
// record by one step and more.  So only the recorder sets kStatNonfinite there.
template <bool F64>
__device__ __forceinline__ DevStats step_record(const ResArgs &a, const double *tot, const long long *cnt,
                                                double ehr_sum, int nsel, int n_valid, unsigned &status, long long step)
{
    if (cnt[2] != 0 && !(status & kStatNonfinite)) {  // a site was nonfinite
        status |= kStatNonfinite;
        atomicOr(a.p.status, kStatNonfinite);
    }
    DevStats st;
    st.step = step;
    // FP32 storage: the rows hold sums of rho - rho_ref and of the deviations of the
    // boundary nodes' populations; their rest values add up to `rest`
    st.mass = F64 ? tot[P_MASS] : tot[P_MASS] + a.rest;
    st.sum_dS = tot[P_SUM_DS];
    st.dS_lbgk = Ar<double>::mul(a.f.one_minus_a2, tot[P_SUM_IN]);
    st.dS_lim = Ar<double>::add(tot[P_DS_LIM], ehr_sum);
    st.n_pos = cnt[0];
    st.n_med = cnt[1];
    st.n_bad = cnt[2];
    st.n_ehr = nsel;
    st.n_cand = n_valid;
    st.status = (status & kStatNonfinite) ? 4 : ((status & kStatTimeout) ? 5 : 0);
    st.reserved = 0;
    return st;
}

}  // namespace
}  // namespace lbm
