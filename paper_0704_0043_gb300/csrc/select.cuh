// select.cuh -- Ehrenfests' selection and step of one pass by one block: the
// candidates' FP64 keys, the top k, f -> f*(m(f)) at the chosen sites (Sec. 3.2;
// Sec. 4.3.2).  Used by the per-step tail (finalize.cu) and by the resident
// kernel (step_resident.cu).
#pragma once

#include <type_traits>

#include "internal.h"
#include "keys.cuh"
#include "lattice.cuh"
#include "site.cuh"

namespace lbm {
namespace {

constexpr int kFinThreads = 512;
constexpr int kFinWarps = kFinThreads / 32;
constexpr int kCap = 2048;    // candidates held (and selected sets sorted) in shared memory
constexpr int kRankCap = 512;  // candidates ranked by counting, one per thread
constexpr int kRank32 = 96;    // candidates whose FP32 bound is found by counting (more: two radix digits)
constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned long long key_bits(double d) { return (unsigned long long)__double_as_longlong(d); }

// The pass's input at site (x, y) in FP32: after free flight (collide) with the
// step kernels' FP32 arithmetic (bounce-back, lid term added as hi + lo), or
// the stored populations themselves (limiter pass).  The loads do not wait for
// one another (see pull).
template <int Q, typename S>
__device__ __forceinline__ void pull_dev(const FinalParams &p, int x, int y, float g[Q])
{
    const S *src = (const S *)p.src;
    const bool wrapx = bc_wrap_x(p.boundary), wrapy = Q == 9 && bc_wrap_y(p.boundary);
    const int xl = x > 0 ? x - 1 : (wrapx ? p.nx - 1 : -1), xr = x + 1 < p.nx ? x + 1 : (wrapx ? 0 : -1);
    const int yl = y > 0 ? y - 1 : (wrapy ? p.ny - 1 : -1), yr = y + 1 < p.ny ? y + 1 : (wrapy ? 0 : -1);
    S raw[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int sx = Lat<Q>::cx(k) > 0 ? xl : (Lat<Q>::cx(k) < 0 ? xr : x);
        const int sy = Lat<Q>::cy(k) > 0 ? yl : (Lat<Q>::cy(k) < 0 ? yr : y);
        const bool own = !p.collide, out = sx < 0 || sy < 0;
        raw[k] = src[fidx(p.plane, p.pitch, !own && out ? Lat<Q>::opp(k) : k, own || out ? y : sy, own || out ? x : sx)];
    }
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        g[k] = s2f(raw[k]);
        if (Q == 9 && Lat<Q>::cy(k) < 0 && yr < 0 && p.collide) g[k] = __fadd_rn(__fadd_rn(g[k], p.lidf[k]), p.lidlo[k]);
    }
}

// Sum over the block in a fixed order (same result every run): warp shuffle
// trees, then a shuffle tree over the warp totals; thread 0 gets the sum.
// FP64 additions are slow on this GPU, so the dependent chain is kept short.
// `warp0_only`: the other warps hold zeros, so warp 0's tree is the sum (the
// same bits: adding the zero totals changes nothing).
__device__ double block_sum0(double v, double *red, bool warp0_only)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    if (warp0_only && warp != 0) return 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
    if (warp0_only) return v;
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double r = lane < kFinWarps ? red[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(kFull, r, o);
        v = r;
    }
    return v;
}


// The digit of a radix-selection pass: hist[d] counts the keys with digit d
// among those still in play, and the rem-th of them is wanted, counting from
// the top digit down (desc) or from digit 0 up.  Threads 0..255 scan the
// counts with warp shuffles (integer sums, so the same on every run) and the
// block picks the digit with __syncthreads_count; every thread of the block
// must call this.  Writes the digit to *digit and the rank left within it to
// *rem_left.
__device__ void pick_digit(const unsigned *hist, long long rem, bool desc, unsigned long long *part,
                           unsigned long long *digit, long long *rem_left)
{
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    unsigned long long c = 0;
    if (t < 256) {
        c = hist[desc ? 255 - t : t];  // position t of the scan order
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, c, o);
            if (lane >= o) c += y;
        }
        if (lane == 31) part[w] = c;
    }
    __syncthreads();
    if (t < 256)
        for (int j = 0; j < w; ++j) c += part[j];
    // c = inclusive count up to scan position t; the wanted digit is the first
    // position whose inclusive count reaches rem
    const int before = __syncthreads_count(t < 256 && (long long)c < rem);
    if (t == before && t < 256) {
        *digit = (unsigned long long)(desc ? 255 - t : t);
        *rem_left = rem - ((long long)c - (long long)hist[desc ? 255 - t : t]);
    }
    __syncthreads();
}

// The geometry of the FP64 key evaluation (FP32 / 16-bit storage).
template <typename P>
__device__ __forceinline__ KeyGeom key_geom(const P &p)
{
    KeyGeom kg;
    kg.nx = p.nx;
    kg.ny = p.ny;
    kg.pitch = p.pitch;
    kg.boundary = p.boundary;
    kg.plane = p.plane;
    kg.a = p.a;
    kg.rw0 = p.rw[0];
    kg.rw1 = p.rw[1];
    kg.rw5 = p.rw[5];
    kg.lid4 = p.lid[4];
    kg.lid7 = p.lid[7];
    kg.lid8 = p.lid[8];
    kg.eq = p.eq;
    return kg;
}


// What the selection keeps in shared memory.
struct SelShared {
    double key[kCap];
    float ds[kCap];  // FP32 dS the candidate was recorded on
    int site[kCap];
    int idx[kCap];
    long long rkey[kRankCap];  // keys in play, packed
    unsigned hist[256];
    unsigned long long part[8], digit;
    double red[2 * P_NSTAT + 2 > kFinWarps + 1 ? 2 * P_NSTAT + 2 : kFinWarps + 1];
    long long rem;
    int nsel, valid, count, tlow;
};

// use(i, load(i)) for this thread's entries i of 0 .. n - 1, four loads at a time: on a
// list that shared memory does not hold, the block's 16 warps do not hide the latency of
// one load each (10^6 keyed candidates of a tube, set and four steps: 16.3 ms one at a
// time, 6.3 four at a time).
template <typename Load, typename Use>
__device__ __forceinline__ void over_entries(int n, Load load, Use use)
{
    constexpr int kLoads = 4;
    for (int b = threadIdx.x; b < n; b += kLoads * kFinThreads) {
        decltype(load(0)) v[kLoads];
#pragma unroll
        for (int j = 0; j < kLoads; ++j) v[j] = load(min(b + j * kFinThreads, n - 1));
#pragma unroll
        for (int j = 0; j < kLoads; ++j)
            if (b + j * kFinThreads < n) use(b + j * kFinThreads, v[j]);
    }
}

// The FP32 bit pattern that candidate i is placed by: of its key rounded, or, with the key
// owed, of the FP32 dS it was recorded on.
__device__ __forceinline__ int cand_pattern(const FinalParams &p, int i, bool small, const SelShared &sh)
{
    if (small) return __float_as_int(sh.ds[i]);
    const double key = p.cand[i].key;
    return __float_as_int(nan64(key) ? p.cand[i].ds32 : narrow(key));
}

// Pattern from which a candidate can be among the k largest: of T (1 - 1/32), T a lower
// bound of the k-th largest among the candidates R that are certainly above delta
// (pattern above that of delta (1 + 1/64); finite).  0 when R has fewer than k.  The FP32
// dS is within 1/64 of the FP64 key (the caller sees to that: mark_unsure), so a
// candidate below that bound cannot reach the k-th largest key.  `keyed`: every candidate
// has its key, and rounded they order as the keys do, so T itself is the bound.  Every
// thread of the block calls it.
template <typename S>
__device__ __noinline__ int fp32_bound(const FinalParams &p, int n, bool small, bool keyed, SelShared &sh)
{
    const int t = threadIdx.x, lane = t & 31;
    const long long k = p.k_max;
    const int dhi_bits = __float_as_int((float)(p.delta_e * (1.0 + 1.0 / 64.0)));
    auto u = [&](int i) -> int { return cand_pattern(p, i, small, sh); };
    auto in_r = [&](int v) { return v > dhi_bits && v < 0x7f800000; };
    if (t == 0) {
        sh.tlow = 0;
        sh.count = 0;
    }
    __syncthreads();
    int mine = 0;
    for (int i = t; i < n; i += kFinThreads) mine += in_r(u(i));
    mine = __reduce_add_sync(kFull, mine);
    if (lane == 0 && mine) atomicAdd(&sh.count, mine);
    __syncthreads();
    if (sh.count < k) return 0;
    if (n <= kRank32) {
        if (t < n) {
            const int v = u(t);
            int rank = 0;
            for (int j = 0; j < n; ++j) {
                const int w = u(j);
                rank += in_r(w) && (w > v || (w == v && j < t));
            }
            if (in_r(v) && rank == (int)k - 1) sh.tlow = v;
        }
        __syncthreads();
    } else {
        // the exponent, then the upper eight (all keyed: sixteen) bits of the mantissa
        int prefix = 0;
        long long rem = k;
        const int low = keyed ? 7 : 15;
#pragma unroll 1
        for (int shift = 23; shift >= low; shift -= 8) {
            if (t < 256) sh.hist[t] = 0;
            __syncthreads();
            for (int base = 0; base < n; base += kFinThreads) {
                const int i = base + t;
                const int v = i < n ? u(i) : 0;
                const int bin = i < n && in_r(v) && ((v ^ prefix) >> (shift + 8)) == 0 ? (v >> shift) & 255 : -1;
                const unsigned peers = __match_any_sync(kFull, bin);
                if (bin >= 0 && lane == __ffs(peers) - 1) atomicAdd(&sh.hist[bin], (unsigned)__popc(peers));
            }
            __syncthreads();
            pick_digit(sh.hist, rem, true, sh.part, &sh.digit, &sh.rem);
            prefix |= (int)sh.digit << shift;
            rem = sh.rem;
            __syncthreads();
        }
        if (t == 0) sh.tlow = prefix;
        __syncthreads();
    }
    return keyed ? sh.tlow - 1 : __float_as_int(__int_as_float(sh.tlow) * 0.96875f);
}

// Where the FP32 dS stands for the key: within 1/64 of it.  dS is the square of a norm of
// n = f - f*, whose FP32 error is a few 2^-24 of the largest f*, over sqrt(f*_k) in the
// norm: with every f*_k at least rho_ref / 256 and rho at most 2 rho_ref, below
// 3e-5 sqrt(rho_ref), so dS of 1e-5 rho_ref and more is within 1/64 (delta of at least
// kSureDelta rho_ref leaves a margin of six).  As f*_k >= rho W_k (1 - 3 u^2) / 2 (D1Q3:
// rho W_k / 4), rho (1 - 3 u^2) of at least kSureFlow rho_ref suffices.  Entropic f*: the
// exact dS of a population near zero may be finite in FP32 and +inf in the key, so it
// never stands for it.  Elsewhere every owed key is evaluated.
constexpr double kSureDelta = 1.0 / 16384.0;
constexpr float kSureFlow = 72.0f / 256.0f, kSureRho = 2.0f;
__device__ __forceinline__ bool sure_delta(const FinalParams &p)
{
    return p.eq != 1 && p.delta_e >= kSureDelta * (double)p.rho_ref;
}
// Owed candidates outside those limits of rho and u get an FP32 dS of +inf: no member of
// R (see fp32_bound), and above every bound, so they are keyed.  (Tested at the candidates
// and not where they are recorded: a test there cost the step kernel registers, 256
// batched cavities 1.3 %.)
template <int Q, typename S>
__device__ __noinline__ void mark_unsure(const FinalParams &p, int n, bool small, SelShared &sh)
{
    for (int i = threadIdx.x; i < n; i += kFinThreads) {
        if (!nan64(small ? sh.key[i] : p.cand[i].key)) continue;
        const int site = small ? sh.site[i] : p.cand[i].site;
        float g[Q], drho, rho, ux, uy;
        pull_dev<Q, S>(p, site % p.nx, site / p.nx, g);
        moments_dev<Q>(g, p.rho_ref, drho, rho, ux, uy);
        const float flow = rho * (1.0f - 3.0f * (ux * ux + uy * uy));
        if (flow >= kSureFlow * p.rho_ref && rho <= kSureRho * p.rho_ref) continue;
        if (small)
            sh.ds[i] = INFINITY;
        else
            p.cand[i].ds32 = INFINITY;
    }
    __syncthreads();
}

// The owed keys of a pass's n candidates (see finish_candidates); returns this
// thread's count of the candidates that are certainly above delta without one.
// Not inlined, like choose_many: the tail starts from a cold instruction cache,
// and a common path that runs straight through costs a few us less than one that
// jumps over rarely taken blocks.
template <int Q, typename S>
__device__ __noinline__ int settle_owed(const FinalParams &p, int n, bool small, int tlow, SelShared &sh)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int nv = 0;
    const int dhi_bits = __float_as_int((float)(p.delta_e * (1.0 + 1.0 / 64.0)));
    auto u = [&](int i) -> int { return __float_as_int(small ? sh.ds[i] : p.cand[i].ds32); };
    const KeyGeom kg = key_geom(p);
    if (t == 0) sh.count = 0;
    __syncthreads();
    for (int i = t; i < n; i += kFinThreads) {
        const double key = small ? sh.key[i] : p.cand[i].key;
        if (!nan64(key)) continue;
        const int v = u(i);
        if (v >= tlow || v <= dhi_bits) {
            if (small) {
                sh.idx[atomicAdd(&sh.count, 1)] = i;  // keyed below, the lanes busy
            } else {
                p.cand[i].key = key_dS_lane<Q, S>(kg, (const S *)p.src, p.cand[i].site, p.delta_e);
            }
        } else {
            ++nv;  // certainly above delta, certainly not among the k largest
            if (small)
                sh.key[i] = -1.0;
            else
                p.cand[i].key = -1.0;
        }
    }
    __syncthreads();
    const int nq = small ? sh.count : 0;
    if (Q == 9 && p.eq != 1 && nq <= 3 * kFinWarps) {
        // three per warp, the warps' first ones on different sub-partitions
        const int g = lane < 27 ? lane / 9 : 0;
        for (int b = warp * 3; b < nq; b += 3 * kFinWarps) {
            const int i = sh.idx[min(b + g, nq - 1)];
            const double key = key_dS9_group<S>(kg, (const S *)p.src, sh.site[i], p.delta_e);
            if (lane < 27 && lane % 9 == 0 && b + g < nq) sh.key[i] = key;
        }
    } else {
        for (int q = t; q < nq; q += kFinThreads) {
            const int i = sh.idx[q];
            sh.key[i] = key_dS_lane<Q, S>(kg, (const S *)p.src, sh.site[i], p.delta_e);
        }
    }
    __syncthreads();
    return nv;
}

// FP64 keys of n <= 32 candidates, into sh.key; `site`: lane i's candidate, the same
// in every warp.  Three to a warp with a lane per direction (D2Q9, polynomial),
// else a lane each in the first warp.  Every thread of the block calls it.
template <int Q, typename S>
__device__ __noinline__ void key_few(const FinalParams &p, int n, int site, SelShared &sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const KeyGeom kg = key_geom(p);
    if (Q == 9 && p.eq != 1) {
        const int g = lane < 27 ? lane / 9 : 0, i = min(3 * warp + g, n - 1);
        const int st = __shfl_sync(kFull, site, i);
        if (3 * warp < n) {
            const double key = key_dS9_group<S>(kg, (const S *)p.src, st, p.delta_e);
            if (lane < 27 && lane % 9 == 0 && 3 * warp + g < n) sh.key[i] = key;
        }
    } else if (threadIdx.x < n) {
        sh.key[lane] = key_dS_lane<Q, S>(kg, (const S *)p.src, site, p.delta_e);
    }
    __syncthreads();
}

// The chosen candidates among more than kRankCap in play: a radix selection
// (eight 8-bit digits of the key, four of the site among ties), the chosen list
// in sh.idx and p.sel, sorted by site when it fits.  Returns the chosen count.
template <typename S>
__device__ __noinline__ int choose_many(const FinalParams &p, int n, bool use_list, bool small, bool take_all,
                                        SelShared &sh)
{
    const int t = threadIdx.x;
    const int *const list = use_list ? p.sel_state->list : nullptr;
    const Cand *const cand = p.cand;
    const long long k = p.k_max;
    auto cidx = [&](int i) -> int { return use_list ? list[i] : i; };
    auto key_of = [&](int i) -> double { return small ? sh.key[i] : cand[cidx(i)].key; };
    auto site_of = [&](int i) -> int { return small ? sh.site[i] : cand[cidx(i)].site; };
    unsigned long long kv = 0;  // threshold dS pattern
    int site_thr = 0x7fffffff;
    if (!take_all) {
        unsigned long long prefix = 0, mask = 0;
        long long rem = k;
        for (int shift = 56; shift >= 0; shift -= 8) {
            for (int d = t; d < 256; d += kFinThreads) sh.hist[d] = 0;
            __syncthreads();
            over_entries(n, key_of, [&](int, double key) {
                const unsigned long long u = key_bits(key);
                if ((long long)u > 0 && (u & mask) == prefix) atomicAdd(&sh.hist[(u >> shift) & 255u], 1u);
            });
            __syncthreads();
            pick_digit(sh.hist, rem, true, sh.part, &sh.digit, &sh.rem);
            prefix = prefix | (sh.digit << shift);
            rem = sh.rem;
            mask |= 255ull << shift;
            __syncthreads();
        }
        kv = prefix;
        // among the candidates with dS == kv take the `rem` lowest sites
        unsigned sprefix = 0, smask = 0;
        for (int shift = 24; shift >= 0; shift -= 8) {
            for (int d = t; d < 256; d += kFinThreads) sh.hist[d] = 0;
            __syncthreads();
            over_entries(n, key_of, [&](int i, double key) {
                if ((long long)key_bits(key) <= 0 || key_bits(key) != kv) return;
                const unsigned s = (unsigned)site_of(i);
                if ((s & smask) == sprefix) atomicAdd(&sh.hist[(s >> shift) & 255u], 1u);
            });
            __syncthreads();
            pick_digit(sh.hist, rem, false, sh.part, &sh.digit, &sh.rem);
            sprefix = sprefix | ((unsigned)sh.digit << shift);
            rem = sh.rem;
            smask |= 255u << shift;
            __syncthreads();
        }
        site_thr = (int)sprefix;
    }
    // compaction of the chosen candidates: candidate indices in p.sel, list
    // entries in sh.idx (the first kCap)
    __syncthreads();
    over_entries(n, key_of, [&](int i, double key) {
        const unsigned long long u = key_bits(key);
        const bool chosen = (long long)u > 0 && (take_all || u > kv || (u == kv && site_of(i) <= site_thr));
        if (chosen) {
            const int j = atomicAdd(&sh.nsel, 1);
            if (j < p.sel_cap) p.sel[j] = cidx(i);
            if (j < kCap) sh.idx[j] = i;
        }
    });
    __syncthreads();
    if (t == 0 && sh.nsel > p.sel_cap) sh.nsel = p.sel_cap;
    __syncthreads();
    const int nsel = sh.nsel;
    if (nsel > kCap) return nsel;
        // bitonic sort of the chosen set by site index (padding sorts last).
        // The payload is sh.idx (chosen list entries, -1 for padding); the
        // sort key is the site: read through sh.site when the candidates are
        // held in shared memory, else copied into sh.site first (then free)
        int mm = 1;
        while (mm < nsel) mm <<= 1;
        for (int i = t; i < mm; i += kFinThreads) {
            if (i >= nsel) sh.idx[i] = -1;
            if (!small) sh.site[i] = i < nsel ? site_of(sh.idx[i]) : 0x7fffffff;
        }
        __syncthreads();
        auto skey = [&](int i) -> int {
            if (!small) return sh.site[i];
            const int li = sh.idx[i];
            return li >= 0 ? sh.site[li] : 0x7fffffff;
        };
        for (int size = 2; size <= mm; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int i = t; i < mm; i += kFinThreads) {
                    const int j = i ^ stride;
                    if (j > i) {
                        const bool up = (i & size) == 0;
                        const int ki = skey(i), kj = skey(j);
                        if ((ki > kj) == up) {
                            int a = sh.idx[i]; sh.idx[i] = sh.idx[j]; sh.idx[j] = a;
                            if (!small) {
                                sh.site[i] = kj;
                                sh.site[j] = ki;
                            }
                        }
                    }
                }
                __syncthreads();
            }
        }
    return nsel;
}

// More candidates than shared memory holds: whether this thread's have one without its
// key; and, all keyed or counted (-1), those above delta counted and the others, and
// those below the bound, put out of play.  Out of line, as settle_owed is.
__device__ __noinline__ bool any_owed(const FinalParams &p, int n)
{
    const Cand *const cand = p.cand;
    bool owed = false;
    over_entries(n, [&](int i) { return cand[i].key; }, [&](int, double key) { owed = owed || nan64(key); });
    return owed;
}
__device__ __noinline__ int settle_many(const FinalParams &p, int n, int tlow)
{
    Cand *const cand = p.cand;
    const double delta = p.delta_e;
    int nv = 0;
    over_entries(n, [&](int i) { return cand[i].key; }, [&](int i, double key) {
        const bool valid = above64(key, delta);
        nv += valid && (long long)key_bits(key) > 0;
        if (!valid || (tlow > 0 && __float_as_int(narrow(key)) < tlow)) cand[i].key = -1.0;
    });
    return nv;
}

// The chosen candidates of a pass with more than a few (see finish_candidates): their list
// entries in sh.idx (the first kCap), their count returned and in sh.nsel, and in sh.valid
// that of the candidates above delta.  Out of line: the usual few candidates then run
// straight through a cold instruction cache (2048 x 2048 entropic FP32 282 -> 276 us a
// step, tube of 1e7 sites 68.0 -> 67.0).
template <int Q, typename S>
__device__ __noinline__ int choose(const FinalParams &p, int n, bool use_list, bool preloaded, Cand first, SelShared &sh)
{
    constexpr bool kLowPrec = !std::is_same<S, double>::value;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int *list = use_list ? p.sel_state->list : nullptr;
    auto cidx = [&](int i) -> int { return use_list ? list[i] : i; };
    const bool small = n <= kCap;  // candidates held in shared memory
    const long long k = p.k_max;
    // below the threshold -> -1, so that from here on a key is valid exactly
    // when its bit pattern is a positive integer (compared as integers, as everywhere
    // below: an FP64 comparison takes the FP64 unit as long as an addition does, and a
    // keyed candidate is no NaN)
    auto settle = [&](double key) { return above64(key, p.delta_e) ? key : -1.0; };
    bool owed = false;
    if (t == 0) {
        sh.nsel = 0;
        if (!use_list) sh.valid = 0;
        sh.count = 0;
    }
    if (small) {
        for (int i = t; i < n; i += kFinThreads) {
            const Cand c = preloaded && i == t ? first : p.cand[cidx(i)];
            owed = owed || (kLowPrec && nan64(c.key));
            sh.key[i] = c.key;
            sh.site[i] = c.site;
            sh.ds[i] = nan64(c.key) ? c.ds32 : narrow(c.key);
        }
    } else if (kLowPrec && !use_list) {
        owed = any_owed(p, n);
    }
    owed = __syncthreads_or(owed) != 0;
    if (!use_list) {
        // FP32 dS pattern below which a candidate cannot be among the k largest; 0
        // where the FP32 dS of owed keys does not stand for them, and where it would
        // spare nothing: choose_many goes over all entries of a list that shared
        // memory does not hold, dropped or not (10^6 keyed candidates of a tube, set
        // and four steps: 23.6 ms with the bound's passes, 17.1 without)
        int tlow = 0;
        if (!owed || sure_delta(p)) {
            if constexpr (kLowPrec) {
                if (owed) mark_unsure<Q, S>(p, n, small, sh);
            }
            if (k <= 0)
                tlow = 0x7f800000;
            else if ((small && n > kRank32) || (owed && n > k))
                tlow = fp32_bound<S>(p, n, small, !owed, sh);
        }
        int nv = 0;  // candidates counted as valid here without a key, then those with one
        if constexpr (kLowPrec) {
            if (owed) nv = settle_owed<Q, S>(p, n, small, tlow, sh);
        }
        // every candidate is keyed or counted (-1) now
        if (small) {
            for (int i = t; i < n; i += kFinThreads) {
                double key = settle(sh.key[i]);
                nv += (long long)key_bits(key) > 0;
                if (__float_as_int(sh.ds[i]) < tlow) key = -1.0;  // counted, out of play
                sh.key[i] = key;
            }
        } else {
            nv += settle_many(p, n, tlow);
        }
        nv = __reduce_add_sync(kFull, nv);
        if (lane == 0 && nv) atomicAdd(&sh.valid, nv);
    }
    __syncthreads();
    const int n_valid = sh.valid;
    if (k <= 0 || n_valid <= 0) return 0;  // the same for the whole block

    // the entries still in play (valid, keyed), compacted: the candidates below
    // the FP32 bound drop out here
    int m = n;
    bool packed = false;
    if (small) {
        // who is in play: a ballot per 32 entries (at most 64 of them), the
        // entries' places from the ballots before theirs
        static_assert(kCap <= 64 * 32, "two ballots per lane");
        const int nb = (n + 31) / 32;
        for (int b = warp; b < nb; b += kFinWarps) {
            const int i = 32 * b + lane;
            const unsigned w = __ballot_sync(kFull, i < n && (long long)key_bits(sh.key[i]) > 0);
            if (lane == 0) sh.hist[b] = w;
        }
        __syncthreads();
        const int c0 = lane < nb ? __popc(sh.hist[lane]) : 0, c1 = lane + 32 < nb ? __popc(sh.hist[lane + 32]) : 0;
        m = __reduce_add_sync(kFull, c0 + c1);
        packed = m <= kRankCap;
        for (int b = warp; b < nb && packed; b += kFinWarps) {
            const int before = __reduce_add_sync(kFull, (lane < b ? c0 : 0) + (lane + 32 < b ? c1 : 0));
            const unsigned w = sh.hist[b];
            if ((w >> lane) & 1u) {
                const int at = before + __popc(w & ((1u << lane) - 1u)), i = 32 * b + lane;
                sh.rkey[at] = (long long)key_bits(sh.key[i]);
                sh.idx[at] = i;
            }
        }
        __syncthreads();
    }
    const bool take_all = (long long)n_valid <= k;
    if (packed) {
        // each thread ranks its own entry by counting the keys that beat it
        // (larger dS, or equal dS at a lower site); the rank is its place in the
        // chosen list, so the list's order does not depend on the recording order
        int mine = -1, rank = 0;
        if (t < m) {
            mine = sh.idx[t];
            const long long u = sh.rkey[t];
            int more = 0, same = 0;
#pragma unroll 4
            for (int j = 0; j < m; ++j) {  // broadcast reads
                const long long v = sh.rkey[j];
                more += v > u;
                same += v == u;
            }
            if (same > 1)  // ties (other than the entry itself)
                for (int j = 0; j < m; ++j) more += sh.rkey[j] == u && sh.site[sh.idx[j]] < sh.site[mine];
            rank = more;
        }
        const int nsel = (int)(k < (long long)m ? k : (long long)m);
        __syncthreads();
        if (mine >= 0 && rank < nsel) sh.idx[rank] = mine;
        if (t == 0) sh.nsel = nsel;
        __syncthreads();
        return nsel;
    }
    return choose_many<S>(p, n, use_list, small, take_all, sh);
}

// The candidates of a pass: FP64 keys where they are owed, the count n_valid of
// candidates above delta, the k with the largest keys (ties to the lower site),
// Ehrenfests' step at those.  List entry i < n is candidate i, or with use_list
// candidate p.sel_state->list[i], all keyed and valid, n_valid given.  `first`:
// candidate of entry threadIdx.x, loaded early, when `preloaded`.  Returns this
// thread's share of phi^2 dS over the chosen sites (entropic f*: of the entropy
// the step adds); sh.nsel holds the chosen count; n_valid is set in thread 0.
// Every thread of a block of kFinThreads calls it, n > 0.
//
// Keys are owed (NaN) by FP32 and 16-bit passes.  Only the candidates that can reach the
// k largest by their FP32 dS, those within 1/64 of delta and those whose FP32 dS does not
// stand for the key get one: FP64 is slow on this GPU (one block keying every candidate of a 517 x 389
// cavity, several hundred with k = 20, took 25 us a step), and the others' count
// is certain without it.  A few are keyed three to a warp (a lane per
// direction), more a lane each.
template <int Q, typename S>
__device__ __forceinline__ double finish_candidates(const FinalParams &p, S *f, int n, bool use_list, bool preloaded,
                                                    const Cand &first, SelShared &sh, int &n_valid)
{
    using T = compute_t<S>;
    constexpr bool kLowPrec = !std::is_same<S, double>::value;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int *list = use_list ? p.sel_state->list : nullptr;
    auto cidx = [&](int i) -> int { return use_list ? list[i] : i; };
    const bool small = n <= kCap;  // candidates held in shared memory
    const long long k = p.k_max;
    double ehr_sum = 0.0;

    auto key_of = [&](int i) -> double { return small ? sh.key[i] : p.cand[cidx(i)].key; };
    int nsel = 0;         // chosen sites (few: in the first warp only)
    bool listed = false;  // the chosen list entries are in sh.idx
    const bool few = n <= 32 && !use_list;
    int few_site = 0;     // few: lane r's chosen site, key and phi
    double few_key = 0.0, few_phi = 0.0;
    if (few) {
        // the usual case: one warp selects in registers, without a block barrier
        Cand c{};
        if (lane < n) c = preloaded ? first : p.cand[lane];
        if (preloaded && warp != 0 && lane < n) c = p.cand[lane];
        bool owed = false;
        if constexpr (kLowPrec) {
            owed = __any_sync(kFull, lane < n && isnan(c.key));
            if (owed) key_few<Q, S>(p, n, c.site, sh);  // every warp takes three
        }
        if (warp == 0) {
            if (owed) c.key = lane < n ? sh.key[lane] : -1.0;
            const bool valid = lane < n && c.key > p.delta_e;
            n_valid = __popc(__ballot_sync(kFull, valid));
            nsel = k < (long long)n_valid ? (int)(k > 0 ? k : 0) : n_valid;
            const long long u = valid ? (long long)key_bits(c.key) : -1;
            int rank = 0;
            for (int j = 0; j < n; ++j) {
                const long long v = __shfl_sync(kFull, u, j);
                const int sj = __shfl_sync(kFull, c.site, j);
                rank += v > u || (v == u && sj < c.site);
            }
            if (valid && rank < nsel) sh.idx[rank] = lane;
            __syncwarp();
            const int from = lane < nsel ? sh.idx[lane] : 0;
            few_site = __shfl_sync(kFull, c.site, from);
            few_key = __shfl_sync(kFull, c.key, from);
            few_phi = __shfl_sync(kFull, c.phi, from);
            if (lane == 0) sh.nsel = nsel;
        }
    } else {
        nsel = choose<Q, S>(p, n, use_list, preloaded, first, sh);
        listed = nsel <= kCap;
        n_valid = sh.valid;
    }
    // Ehrenfests' step at each chosen site, in the list's order
    for (int r = t; r < nsel; r += kFinThreads) {
        // the chosen candidate's site and key (from shared memory when listed) and
        // its phi
        int site;
        double key, phi;
        if (few) {
            site = few_site;
            key = few_key;
            phi = few_phi;
            p.sel[r] = site;
        } else if (listed) {
            const int li = sh.idx[r];
            site = small ? sh.site[li] : sh.site[r];
            key = key_of(li);
            phi = p.cand[cidx(li)].phi;
        } else {
            const Cand c = p.cand[p.sel[r]];
            site = c.site;
            key = c.key;
            phi = c.phi;
        }
        const int x = site % p.nx, y = site / p.nx;
        T g[Q], fs[Q], rho, ux, uy;
        bool write = true;
        if constexpr (std::is_same<T, float>::value) {
            // FP32 / 16-bit storage: f*(m) as g - n (the limiter with phi = 0),
            // m taken from the pass's input (the collision conserves m), so
            // mass and momentum are kept and the result is rounded once
            float drho, nq[Q];
            pull_dev<Q, S>(p, x, y, g);
            moments_dev<Q>(g, p.rho_ref, drho, rho, ux, uy);
            if (p.eq == 1) {
                // entropic f*: from the limited state in FP64 (the stored values), the
                // entropy the step adds, dS w.r.t. its own f*; a state whose moments
                // have no entropic f* keeps its populations
                double fl[Q], fsd[Q], r2, a2, b2;
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    fl[q] = Ar<double>::add((double)s2f(f[fidx(p.plane, p.pitch, q, y, x)]), p.rw[q]);
                moments<Q, double>(fl, r2, a2, b2);
                write = feq_any<Q>(1, r2, a2, b2, fsd);
                if (write) {
                    const double d = rel_entropy<Q>(fl, fsd);
                    if (isfinite(d)) ehr_sum = Ar<double>::add(ehr_sum, d);
                    if constexpr (Q == 9)
                        feq_ent9_x<F1>(drho, rho, ux, uy, fs);
                    else
                        feq_ent3_dev(drho, rho, ux, fs);
                } else {
#pragma unroll
                    for (int q = 0; q < Q; ++q) fs[q] = 0.f;
                }
            } else {
                feq_dev<Q>(drho, rho, ux, uy, fs);
            }
            neq_dev<Q>(g, fs, nq);
#pragma unroll
            for (int q = 0; q < Q; ++q) fs[q] = g[q] - nq[q];
        } else {
            // FP64: f*(m(f')) from the stored f', in the oracle's order
#pragma unroll
            for (int q = 0; q < Q; ++q) g[q] = s2f(f[fidx(p.plane, p.pitch, q, y, x)]);
            moments<Q, T>(g, rho, ux, uy);
            if (p.eq == 1) {
                // entropic f*: the step adds dS of the limited state w.r.t. its own f*
                // where the limited state's moments have no entropic f* the site keeps its populations
                write = feq_any<Q>(1, rho, ux, uy, fs);
                const double d = write ? rel_entropy<Q>(g, fs) : (double)NAN;
                if (isfinite(d)) ehr_sum = Ar<double>::add(ehr_sum, d);
            } else {
                feq<Q, T>(rho, ux, uy, fs);
            }
        }
        if (write) {
#pragma unroll
            for (int q = 0; q < Q; ++q) f[fidx(p.plane, p.pitch, q, y, x)] = f2s<S>(fs[q]);
        }
        if (p.eq != 1) ehr_sum = Ar<double>::add(ehr_sum, Ar<double>::mul(Ar<double>::mul(phi, phi), key));
    }
    __syncthreads();
    // the chosen sites, as site indices, for lbm_limited_sites
    if (few) return ehr_sum;
    if (listed) {
        for (int r = t; r < nsel; r += kFinThreads) p.sel[r] = small ? sh.site[sh.idx[r]] : sh.site[r];
    } else {
        // unsorted (more than kCap chosen): convert in place, one owner per slot
        for (int r = t; r < nsel; r += kFinThreads) p.sel[r] = p.cand[p.sel[r]].site;
    }
    return ehr_sum;
}

}  // namespace
}  // namespace lbm
