// finalize.cu -- the per-step tail: fixed-order FP64 reduction of the step
// kernel's block partials, Ehrenfests' selection and step, and the stats record.
//
// Ehrenfests' regularisation (Sec. 3.2; Sec. 4.3.2): among the sites whose
// dS(f') exceeds delta, at most k with the largest dS are equilibrated,
// f -> f*(m(f)).  Ties in dS go to the lower site index, so the chosen set is
// unique.  When there are more than k candidates, a single block finds the k-th
// largest (dS, -site) pair by radix selection: eight 8-bit digit passes over the
// 64-bit pattern of dS (positive doubles order like their bit patterns), then
// four passes over the site index among the candidates tied at the threshold.
//
// The kernel sits between two step launches, so it is built for latency: one
// block runs it, most candidates arrive with their FP64 keys, the selection
// (select.cuh) keys only those of the others that can matter, and sums use warp
// shuffles or exact integer arithmetic.  The tail starts from a cold instruction
// cache (about 10 ns per instruction fetched), so rarely taken parts are out of
// line.  When a pass records more candidates than the block holds in shared
// memory (a state far from equilibrium), the
// tail runs as a cooperative grid of one block per SM that first preselects
// them (dense_select): the FP32 dS recorded with each candidate is within 1/64
// of its FP64 key, so a radix search over the FP32 values bounds the k-th
// largest key, and only the candidates near that bound or near delta need
// their FP64 keys; block 0 then selects among the short list.
#include <type_traits>

#include "internal.h"
#include "keys.cuh"
#include "lattice.cuh"
#include "select.cuh"

namespace lbm {
namespace {

// candidates a thread reads at once in dense_select (2.2 M of a 2048^2 lattice: four steps
// with set and get 1562 us at one, 1490 at four, 1530 at eight)
constexpr int kSelLoads = 4;
constexpr unsigned kSelSpinLimit = 1u << 21;  // grid-barrier polls (about a second) before giving up

// Grid barrier of the cooperative tail: each block adds one arrival to *bar;
// with `wait` it polls until `target` blocks have arrived.  The poll is
// bounded: past kSelSpinLimit polls the block sets kStatTimeout in *status and
// goes on (the pass's results are then not trusted; the host reports
// LBM_ERR_TIMEOUT).  Every thread of the block calls it; returns whether this
// block gave up.
__device__ bool grid_sync(unsigned *bar, unsigned target, bool wait, unsigned *status, int *s_flag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        int gave_up = 0;
        __threadfence();
        atomicAdd(bar, 1u);
        if (wait) {
            unsigned polls = 0;
            while (*(volatile unsigned *)bar < target) {
                if (++polls > kSelSpinLimit) {
                    gave_up = 1;
                    atomicOr(status, kStatTimeout);
                    break;
                }
                __nanosleep(64);
            }
        }
        __threadfence();
        *s_flag = gave_up;
    }
    __syncthreads();
    return *s_flag != 0;
}

// The bin holding the rem-th largest entry (rem >= 1) of a kSelBins-bin
// histogram in device memory (bin b counts the keys with digit b, larger
// digits larger keys), and the rank left within that bin.  *s_tot receives the
// histogram's total; when it is below rem no bin holds the entry and *s_bin
// is -1.  Thread t scans bins 8t .. 8t+7 from the top; integer sums, so the
// same on every run.  Every thread of the block calls it.
__device__ void pick_bin(const unsigned *h, long long rem, long long *s_wpart, int *s_bin, long long *s_rem,
                         long long *s_tot)
{
    constexpr int kPer = kSelBins / kFinThreads;
    static_assert(kPer * kFinThreads == kSelBins, "whole bins per thread");
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned c[kPer];
    long long mine = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        c[j] = __ldcg(h + (kSelBins - 1 - (t * kPer + j)));  // written by other blocks' atomics
        mine += c[j];
    }
    long long incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s_wpart[w] = incl;
    if (t == 0) *s_bin = -1;
    __syncthreads();
    for (int j = 0; j < w; ++j) incl += s_wpart[j];
    if (t == kFinThreads - 1) *s_tot = incl;
    const long long excl = incl - mine;
    if (excl < rem && rem <= incl) {  // one thread: its bins hold the entry
        long long acc = excl;
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            if (acc < rem && rem <= acc + c[j]) {
                *s_bin = kSelBins - 1 - (t * kPer + j);
                *s_rem = rem - acc;
            }
            acc += c[j];
        }
    }
    __syncthreads();
}

// Device-wide preselection of n > kCap recorded candidates (all blocks of the
// cooperative tail call it).  R denotes the candidates whose FP32 dS exceeds
// dhi = delta (1 + 1/64): their FP64 keys exceed delta.  When |R| >= k, the
// k-th largest FP32 dS in R is at least T, the lower end of its bin after two
// 12-bit radix levels (bits 30..19, then 18..7, of the FP32 pattern; positive
// floats order like their patterns), so the k-th largest valid FP64 key is
// at least T / (1 + 1/64), and a candidate whose key reaches it has FP32 dS of
// at least T (1 - 1/64) / (1 + 1/64) > T (1 - 1/32) = Tlow.  The list takes
// every valid candidate with FP32 dS >= Tlow (all valid ones when |R| < k):
// it holds every candidate of the exact top k, ties at the k-th key included.
// The valid candidates are counted exactly: a candidate with a key is valid
// when the key exceeds delta; one without a key is keyed here when it is on
// the list's side of Tlow or within 1/64 of delta (at or below dhi), and
// otherwise valid when its FP32 dS exceeds dhi.  Block 0 then reads the list
// (returns true when it fits in kSelList) and resets the shared state for
// the next pass; the other blocks return false.  Not inlined: the one-block
// tail runs from a cold instruction cache every step, and its code stays
// compact without this rarely taken path.
template <int Q, typename S>
__device__ __noinline__ bool dense_select(const FinalParams &p, int n, unsigned *sh, long long *s_wpart, int *s_bin,
                             long long *s_rem, long long *s_tot, int *s_flag, int *s_qn, unsigned *s_acc,
                             unsigned *s_cnt, unsigned *s_nv)
{
    SelState *ss = p.sel_state;
    const int t = threadIdx.x, lane = t & 31;
    const unsigned nb = gridDim.x;
    const int dhi_bits = __float_as_int((float)(p.delta_e * (1.0 + 1.0 / 64.0)));
    const long long stride = (long long)nb * kFinThreads;
    const long long base0 = (long long)blockIdx.x * kFinThreads;
    auto in_r = [&](int u) { return u > dhi_bits && u < 0x7f800000; };  // FP32 dS above dhi (finite)

    // level 1: bits 30..19 of the candidates in R
    // lanes with the same bin add once (most candidates fall in a few bins)
    auto count_bin = [&](int bin) {
        const unsigned peers = __match_any_sync(kFull, bin);
        if (bin >= 0 && lane == __ffs(peers) - 1) atomicAdd(&sh[bin], (unsigned)__popc(peers));
    };
    for (int b = t; b < kSelBins; b += kFinThreads) sh[b] = 0;
    __syncthreads();
    // kSelLoads candidates of a thread are read together: 16 warps an SM do not hide
    // the latency of one read each
    for (long long base = base0; base < n; base += kSelLoads * stride) {  // whole warps per round
        int u[kSelLoads];
#pragma unroll
        for (int j = 0; j < kSelLoads; ++j) {
            const long long i = base + j * stride + t;
            u[j] = i < n ? __float_as_int(p.cand[i].ds32) : 0x7f800000;  // not in R
        }
#pragma unroll
        for (int j = 0; j < kSelLoads; ++j) count_bin(in_r(u[j]) ? u[j] >> 19 : -1);
    }
    __syncthreads();
    for (int b = t; b < kSelBins; b += kFinThreads)
        if (sh[b]) atomicAdd(&ss->hist1[b], sh[b]);
    grid_sync(&ss->bar, nb, true, p.status, s_flag);

    // level 2: bits 18..7 within the level-1 bin of the k-th largest
    pick_bin(ss->hist1, p.k_max, s_wpart, s_bin, s_rem, s_tot);
    const bool all = *s_tot < p.k_max;  // fewer than k in R: every valid candidate is listed
    const int b1 = *s_bin;
    const long long rem1 = *s_rem;
    for (int b = t; b < kSelBins; b += kFinThreads) sh[b] = 0;
    __syncthreads();
    if (!all) {
        for (long long base = base0; base < n; base += kSelLoads * stride) {
            int u[kSelLoads];
#pragma unroll
            for (int j = 0; j < kSelLoads; ++j) {
                const long long i = base + j * stride + t;
                u[j] = i < n ? __float_as_int(p.cand[i].ds32) : 0x7f800000;
            }
#pragma unroll
            for (int j = 0; j < kSelLoads; ++j)
                count_bin(in_r(u[j]) && (u[j] >> 19) == b1 ? (u[j] >> 7) & (kSelBins - 1) : -1);
        }
        __syncthreads();
        for (int b = t; b < kSelBins; b += kFinThreads)
            if (sh[b]) atomicAdd(&ss->hist2[b], sh[b]);
    }
    grid_sync(&ss->bar, 2 * nb, true, p.status, s_flag);

    // the bound, the keys, the count and the list
    int tlow_bits = 0;
    if (!all) {
        pick_bin(ss->hist2, rem1, s_wpart, s_bin, s_rem, s_tot);
        const unsigned ulb = ((unsigned)b1 << 19) | ((unsigned)*s_bin << 7);
        tlow_bits = __float_as_int(__uint_as_float(ulb) * 0.96875f);
    }
    // Candidates without a key that need one are queued in shared memory (the
    // histogram is no longer needed) and keyed a block at a time, every lane
    // busy: FP64 is slow on this GPU, and keying them where they lie would
    // run most warps' FP64 code for one or two lanes.
    int *queue = reinterpret_cast<int *>(sh);  // at most 2 kFinThreads - 1 entries
    if (t == 0) {
        *s_acc = 0;
        *s_qn = 0;
    }
    __syncthreads();
    constexpr bool kKeyHere = !std::is_same<S, double>::value && Q == 9;  // candidates recorded without a key
    const KeyGeom kg = key_geom(p);
    unsigned nv = 0;
    // warp-aggregated list append (every lane of the warp calls it)
    auto append = [&](bool listed, long long i) {
        const unsigned m = __ballot_sync(kFull, listed);
        unsigned at = 0;
        if (lane == 0 && m) at = atomicAdd(&ss->count, (unsigned)__popc(m));
        at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
        if (listed && at < (unsigned)kSelList) ss->list[at] = (int)i;
    };
    // key queue entries from .. from + cnt - 1 (cnt <= kFinThreads), one per thread
    auto drain = [&](int from, int cnt) {
        bool listed = false;
        long long i = -1;
        if (t < cnt) {
            i = queue[from + t];
            const Cand c = p.cand[i];
            const double key = key_dS9_lane<S>(kg, (const S *)p.src, c.site, p.delta_e);
            p.cand[i].key = key;
            const bool valid = key > p.delta_e;
            nv += valid;
            listed = valid && __float_as_int(c.ds32) >= tlow_bits;
        }
        append(listed, i);
    };
    int queued = 0;  // queue entries, the same in every thread: each counts them itself
    for (long long base = base0; base < n; base += kSelLoads * stride) {  // whole blocks per round
        Cand cs[kSelLoads];
#pragma unroll
        for (int j = 0; j < kSelLoads; ++j) {
            const long long i = base + j * stride + t;
            if (i < n) cs[j] = p.cand[i];
        }
#pragma unroll
        for (int j = 0; j < kSelLoads; ++j) {
            if (base + j * stride >= n) break;  // the same for the whole block
            const long long i = base + j * stride + t;
            bool valid = false, listed = false, need = false;
            if (i < n) {
                const int u = __float_as_int(cs[j].ds32);
                const bool top = u >= tlow_bits;
                need = kKeyHere && isnan(cs[j].key) && (top || u <= dhi_bits);
                valid = !need && (isnan(cs[j].key) ? in_r(u) : cs[j].key > p.delta_e);
                listed = top && valid;
            }
            append(listed, i);
            nv += valid;
            if constexpr (kKeyHere) {
                const unsigned m = __ballot_sync(kFull, need);
                int at = 0;
                if (lane == 0 && m) at = atomicAdd(s_qn, __popc(m));
                at = __shfl_sync(kFull, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (need) queue[at] = (int)i;
                // (the count is not read from s_qn: a warp that is ahead adds to it again)
                queued += __syncthreads_count(need);
                if (queued >= kFinThreads) {
                    queued -= kFinThreads;
                    drain(queued, kFinThreads);
                    __syncthreads();  // the entries are read before new ones overwrite them
                    if (t == 0) *s_qn = queued;
                    __syncthreads();
                }
            }
        }
    }
    if constexpr (kKeyHere) drain(0, queued);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nv += __shfl_down_sync(kFull, nv, o);
    if (lane == 0 && nv) atomicAdd(s_acc, nv);
    __syncthreads();
    if (t == 0 && *s_acc) atomicAdd(&ss->n_valid, *s_acc);
    // block 0 waits for every block's list entries and count
    grid_sync(&ss->bar, 3 * nb, blockIdx.x == 0, p.status, s_flag);
    if (blockIdx.x != 0) return false;
    if (t == 0) {
        *s_cnt = __ldcg(&ss->count);
        *s_nv = __ldcg(&ss->n_valid);
        ss->count = 0;
        ss->n_valid = 0;
        ss->bar = 0;
    }
    for (int b = t; b < kSelBins; b += kFinThreads) {
        ss->hist1[b] = 0;
        ss->hist2[b] = 0;
    }
    __syncthreads();
    return *s_cnt <= (unsigned)kSelList;
}

// BATCHED: block b finishes instance b of `table`; otherwise the single (p0, f0).
// GRID: the cooperative grid of one block per SM (dense candidates are
// preselected by all blocks; block 0 runs the tail); otherwise one block.
template <int Q, typename S, bool BATCHED, bool GRID = false>
__global__ void __launch_bounds__(kFinThreads, BATCHED ? 2 : 1) k_finalize(const __grid_constant__ FinalParams p0, S *__restrict__ f0,
                                                          const FinalArgs *__restrict__ table)
{
    using T = compute_t<S>;
    // Launched as a programmatic dependent of the step kernel: wait for it to
    // finish before any memory access, then let the next step kernel be
    // scheduled early.  Both are no-ops in an ordinary launch.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // The next launch may be scheduled now.  In a grid launch it starts only
    // when every block of this grid has passed this point, i.e. when all of
    // them are resident, so its blocks cannot keep one of ours from running
    // (the grid barriers below wait for resident blocks only).
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    __shared__ SelShared sh;
    __shared__ long long s_wpart[kFinWarps], s_rem2, s_tot;
    __shared__ int s_bin, s_flag, s_qn;
    __shared__ unsigned s_acc, s_cnt, s_nv;
    // dense candidates in a grid launch: every block preselects, then block 0
    // runs the tail over the list (use_list) or, when the list overflowed,
    // over all candidates; otherwise block 0 alone runs the tail
    bool use_list = false;
    if constexpr (GRID) {
        const int nrec = p0.ehrenfest ? *p0.cand_count : 0;
        const int n0 = nrec < p0.cand_cap ? nrec : p0.cand_cap;
        const bool dense = n0 > kCap && p0.sel_state != nullptr && p0.k_max > 0;
        if (!dense && blockIdx.x != 0) return;
        if (dense) {
            use_list = dense_select<Q, S>(p0, n0, reinterpret_cast<unsigned *>(sh.key), s_wpart, &s_bin, &s_rem2,
                                          &s_tot, &s_flag, &s_qn, &s_acc, &s_cnt, &s_nv);
            if (blockIdx.x != 0) return;
        }
    }
    __shared__ __align__(16) FinalArgs sA;
    if constexpr (BATCHED) {
        const unsigned *from = reinterpret_cast<const unsigned *>(table + blockIdx.x);
        unsigned *to = reinterpret_cast<unsigned *>(&sA);
        for (int i = threadIdx.x; i < (int)(sizeof(FinalArgs) / 4); i += kFinThreads) to[i] = from[i];
        __syncthreads();
    }
    const FinalParams &p = BATCHED ? sA.p : p0;
    S *__restrict__ f = BATCHED ? (S *)sA.f : f0;
    __shared__ double tot[P_NSTAT];
    __shared__ long long s_step, s_rec;
    __shared__ unsigned s_status;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;

    // every thread reads the candidate count (one broadcast load) and loads its
    // first candidate slot at once (any slot below the capacity is readable,
    // so the load does not wait for the count), and both loads overlap the
    // reduction of the step's sums; list entry i is candidate cidx(i) (the
    // preselected list, or all candidates)
    int n = 0;
    if (use_list) {
        n = (int)s_cnt;
    } else if (p.ehrenfest) {
        const int nrec = *p.cand_count;
        n = nrec < p.cand_cap ? nrec : p.cand_cap;
    }
    Cand first{};
    if (!BATCHED && p.ehrenfest && (use_list ? t < n : t < p.cand_cap)) first = p.cand[use_list ? p.sel_state->list[t] : t];
    if (t == 0) {
        s_step = p.counters[0];
        s_rec = p.counters[1];
        s_status = *p.status;
        sh.nsel = 0;
        sh.valid = use_list ? (int)s_nv : 0;
    }
    if (p.fixed) {
        // the fused kernel's kFxRows fixed-point accumulator rows (exact integer
        // sums, so the order does not matter), reduced by warp 0 alone: lane l
        // reads 16-byte chunk l % 8 of rows l / 8 and l / 8 + 4 and clears them
        // for the next step.  Chunk c < 4 is FP statistic c (low, high word),
        // chunk 4 the site and positivity counts, chunk 5 the median and
        // nonfinite counts, chunk 6 the nonfinite bits.
        static_assert(kFxRows == 8 && kFxWords == 16, "warp 0 reads 8 rows of 8 chunks");
        if (warp == 0) {
            const int c = lane & 7;
            ulonglong2 *chunks = reinterpret_cast<ulonglong2 *>(p.partials);
            const ulonglong2 w0 = chunks[lane], w1 = chunks[lane + 32];
            chunks[lane] = make_ulonglong2(0ull, 0ull);
            chunks[lane + 32] = make_ulonglong2(0ull, 0ull);
            unsigned __int128 v = 0;
            unsigned long long u0 = 0, u1 = 0;
            if (c < 4) {
                v = (((unsigned __int128)w0.y << 64) | w0.x) + (((unsigned __int128)w1.y << 64) | w1.x);
            } else if (c < 6) {
                u0 = w0.x + w1.x;
                u1 = w0.y + w1.y;
            } else if (c == 6) {
                u0 = w0.x | w1.x;
            }
#pragma unroll
            for (int o = 8; o <= 16; o <<= 1) {  // lanes holding the same chunk
                const unsigned long long lo = __shfl_xor_sync(kFull, (unsigned long long)v, o);
                const unsigned long long hi = __shfl_xor_sync(kFull, (unsigned long long)(v >> 64), o);
                const unsigned long long a0 = __shfl_xor_sync(kFull, u0, o), a1 = __shfl_xor_sync(kFull, u1, o);
                v += ((unsigned __int128)hi << 64) | lo;
                u0 = c == 6 ? (u0 | a0) : u0 + a0;
                u1 += a1;
            }
            // lanes 0..7 hold chunk totals; lanes 0..3 need the site count
            // (chunk 4) and the nonfinite bits (chunk 6)
            const unsigned long long sites = __shfl_sync(kFull, u0, 4), bits = __shfl_sync(kFull, u0, 6);
            if (lane < 4) {  // FP statistic lane
                double d = ((bits >> lane) & 1u) ? __longlong_as_double(0x7ff8000000000000LL) : fx_value(v);
                if (lane == P_MASS) d = Ar<double>::add(d, Ar<double>::mul((double)sites, (double)p.rho_ref));
                tot[lane] = d;
            } else if (lane == 4) {
                tot[P_NPOS] = (double)u1;
            } else if (lane == 5) {
                tot[P_NMED] = (double)u0;
                tot[P_NBAD] = (double)u1;
            }
        }
    } else if (warp < 2 * P_NSTAT) {
        // block partials: warps 2s and 2s+1 reduce statistic s over alternate
        // 32-row groups, in a fixed order (short FP64 dependency chains)
        const int stat = warp >> 1, half = warp & 1;
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
        int r = lane + 32 * half;
        for (; r + 192 < p.nblocks; r += 256) {
            v0 += p.partials[(long long)r * P_NSTAT + stat];
            v1 += p.partials[(long long)(r + 64) * P_NSTAT + stat];
            v2 += p.partials[(long long)(r + 128) * P_NSTAT + stat];
            v3 += p.partials[(long long)(r + 192) * P_NSTAT + stat];
        }
        for (; r < p.nblocks; r += 64) v0 += p.partials[(long long)r * P_NSTAT + stat];
        double v = (v0 + v1) + (v2 + v3);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
        if (lane == 0) sh.red[warp] = v;
    }
    __syncthreads();
    if (!p.fixed && t < P_NSTAT) tot[t] = sh.red[2 * t] + sh.red[2 * t + 1];
    __syncthreads();
    int n_valid = 0;
    double ehr_sum = 0.0;
    if (n > 0) ehr_sum = finish_candidates<Q, S>(p, f, n, use_list, !BATCHED, first, sh, n_valid);
    // thread r applied chosen site r: with at most 32 of them only warp 0
    // holds terms
    const double esum = sh.nsel > 0 ? block_sum0(ehr_sum, sh.red, sh.nsel <= 32) : 0.0;
    if (t == 0) {
        long long step = s_step;
        if (p.collide) {
            step += 1;
            p.counters[0] = step;
        }
        const long long rec = s_rec;
        p.counters[1] = rec + 1;
        DevStats st;
        st.step = step;
        st.mass = tot[P_MASS];
        st.sum_dS = tot[P_SUM_DS];
        st.dS_lbgk = p.collide ? Ar<double>::mul(p.one_minus_a2, tot[P_SUM_IN]) : 0.0;
        st.dS_lim = Ar<double>::add(tot[P_DS_LIM], esum);
        st.n_pos = (long long)tot[P_NPOS];
        st.n_med = (long long)tot[P_NMED];
        st.n_ehr = sh.nsel;
        st.n_cand = n_valid;
        st.n_bad = (long long)tot[P_NBAD];
        // the step kernel set its status bits before this launch began
        const unsigned sb = s_status;
        st.status = (sb & kStatNonfinite) ? 4 : ((sb & kStatTimeout) ? 5 : 0);
        st.reserved = 0;
        p.stats_ring[rec % p.ring_len] = st;
        if (p.probe != nullptr && p.collide) {
            // the control point's moments after the whole step (Ehrenfests' writes
            // are visible: the block synchronised after them), as lbm_moments
            // evaluates them
            const int x = p.probe_site % p.nx, y = p.probe_site / p.nx;
            double r, a, b;
            S raw[Q];
#pragma unroll
            for (int q = 0; q < Q; ++q) raw[q] = f[fidx(p.plane, p.pitch, q, y, x)];
            site_moments<Q, S>(p, raw, r, a, b);
            double *slot = p.probe + 3 * ((step - 1) % p.probe_cap);
            slot[0] = r;
            slot[1] = a;
            slot[2] = b;
        }
        *p.sel_count = sh.nsel;
        *p.cand_count = 0;
        if (p.work != nullptr) *p.work = 0;  // the next fused launch starts at its first item
    }
}

}  // namespace

template <typename T>
cudaError_t launch_finalize(int q, const FinalParams &p, T *f, cudaStream_t s, int grid)
{
    // programmatic dependent launch (see k_finalize); a grid is a cooperative
    // launch, so that its blocks are resident together for the grid barrier
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid > 1 ? grid : 1);
    cfg.blockDim = dim3(kFinThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeCooperative;
    attr[1].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = grid > 1 ? 2 : 1;
    FinalParams pp = p;
    if (grid <= 1) pp.sel_state = nullptr;
    const FinalArgs *none = nullptr;
    if (grid > 1) {
        if (q == 9) return cudaLaunchKernelEx(&cfg, k_finalize<9, T, false, true>, pp, f, none);
        return cudaLaunchKernelEx(&cfg, k_finalize<3, T, false, true>, pp, f, none);
    }
    if (q == 9) return cudaLaunchKernelEx(&cfg, k_finalize<9, T, false>, pp, f, none);
    return cudaLaunchKernelEx(&cfg, k_finalize<3, T, false>, pp, f, none);
}

template <typename T>
int finalize_grid(int q)
{
    int dev = 0, coop = 0, per_sm = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) return 0;
    const cudaError_t e = q == 9
        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_finalize<9, T, false, true>, kFinThreads, 0)
        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_finalize<3, T, false, true>, kFinThreads, 0);
    if (e != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        return 0;
    }
    return sm_count();
}

cudaError_t launch_finalize_batched_f32(int q, const FinalArgs *table, int n, cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const FinalParams none{};
    if (q == 9)
        k_finalize<9, float, true><<<n, kFinThreads, 0, s>>>(none, nullptr, table);
    else
        k_finalize<3, float, true><<<n, kFinThreads, 0, s>>>(none, nullptr, table);
    return cudaGetLastError();
}

template cudaError_t launch_finalize<float>(int, const FinalParams &, float *, cudaStream_t, int);
template cudaError_t launch_finalize<double>(int, const FinalParams &, double *, cudaStream_t, int);
template cudaError_t launch_finalize<__nv_bfloat16>(int, const FinalParams &, __nv_bfloat16 *, cudaStream_t, int);
template cudaError_t launch_finalize<__half>(int, const FinalParams &, __half *, cudaStream_t, int);
template int finalize_grid<float>(int);
template int finalize_grid<double>(int);
template int finalize_grid<__nv_bfloat16>(int);
template int finalize_grid<__half>(int);

}  // namespace lbm
