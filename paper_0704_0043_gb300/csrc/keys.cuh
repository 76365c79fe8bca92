// keys.cuh -- the FP64 Ehrenfests' key dS(f') of one D2Q9 site evaluated by a
// whole warp from FP32 / 16-bit storage (Sec. 3.2; dS in the quadratic form
// of Sec. 3.6).  The fused step kernel keys its candidates where it finds them.
#pragma once

#include "internal.h"
#include "lattice.cuh"

namespace lbm {

// What the FP64 key needs of a D2Q9 lattice (walls, channel or periodic):
// layout, boundary, a = 2 beta - 1, rho_ref W_k (rest, axis, diagonal) and the
// moving-lid terms of the links through the lid (directions 4, 7, 8).
struct KeyGeom {
    int nx, ny, pitch, boundary;
    int eq;  // 1: entropic f* and the exact dS of Eq. DelS (key_ent9)
    long long plane;
    double a;
    double rw0, rw1, rw5;
    double lid4, lid7, lid8;
    __device__ double rw(int k) const { return k == 0 ? rw0 : (k <= 4 ? rw1 : rw5); }
    __device__ double lid(int k) const { return k == 4 ? lid4 : (k == 7 ? lid7 : (k == 8 ? lid8 : 0.0)); }
};

// Population k arriving at site (x, y), in FP64 from FP32 / 16-bit storage
// `src` (layout of internal.h): (double) g + rho_ref W, the value the FP64
// path computes from the same stored state.
template <typename S>
__device__ double pull_one_f64(const KeyGeom &p, const S *src, int x, int y, int k)
{
    const bool wrapx = bc_wrap_x(p.boundary), wrapy = bc_wrap_y(p.boundary);
    int sx = x - Lat<9>::cx(k), sy = y - Lat<9>::cy(k);
    if (wrapx) sx = sx < 0 ? sx + p.nx : (sx >= p.nx ? sx - p.nx : sx);
    if (wrapy) sy = sy < 0 ? sy + p.ny : (sy >= p.ny ? sy - p.ny : sy);
    const bool in = sx >= 0 && sx < p.nx && sy >= 0 && sy < p.ny;
    const int q = in ? k : Lat<9>::opp(k);
    // the address is selected, not the load: several pulls stay in flight together
    const S raw = src[(long long)q * p.plane + (long long)(in ? sy : y) * p.pitch + kLead + (in ? sx : x)];
    double v = Ar<double>::add((double)s2f(raw), p.rw(q));
    if (!in && sy > p.ny - 1) v = Ar<double>::add(v, p.lid(k));
    return v;
}

// FP64 key with entropic f* (Eq. maxwellian) and the exact dS of Eq. DelS, from
// the same pulled FP64 populations: the evaluation of the FP64 path
// (site_collide with eq = 1), so the key is the value an LBM_FP64 context
// would compare with delta_e; +inf for a state with a negative population.
template <typename S>
__device__ __noinline__ double key_ent9(const KeyGeom p, const S *src, int site, double delta_e)
{
    const int x = site % p.nx, y = site / p.nx;
    double fin[9], fs[9], fp[9], ds, dsin, rho;
#pragma unroll
    for (int k = 0; k < 9; ++k) fin[k] = pull_one_f64<S>(p, src, x, y, k);
    const bool bad = site_collide<9, double>(fin, p.a, true, fs, fp, ds, dsin, rho, 1, false);
    return !bad && ds > delta_e ? ds : -1.0;
}

// FP64 keys dS(f') of up to three sites by the whole (converged) warp: lanes
// 9 g .. 9 g + 8 take the site that lane's `site` argument names (lanes 27 .. 31
// repeat group 0), a lane per direction.  Lane 0 of a group sums rho, lane 1
// rho u_x and lane 2 rho u_y, each in k order as the sequential evaluation does;
// the two quotients run together; every lane then evaluates its f*_k and its dS
// term, and the terms are added in k order: the key is that of key_dS9_lane bit
// for bit, in 48 FP64 instructions where one lane alone needs about 190.  Returns the key,
// or -1 for a site at or below delta_e or one that cannot be limited; every
// lane of a group returns the same value.  key_dS9_core: from the lane's pulled
// population `mine` (a2b = 2 beta - 1).  The whole is not inlined: the caller's hot
// loop keeps its registers, and the call is rare.
__device__ __forceinline__ double key_dS9_core(double mine, double a2b, double delta_e)
{
    using A = Ar<double>;
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, base = lane < 27 ? lane / 9 * 9 : 0, k = lane < 27 ? lane % 9 : lane - 27;
    // lane 0: f0 + f1 + ... + f8; lane 1: f1 - f3 + f5 - f6 - f7 + f8; lane 2: f2 - f4 + f5
    // + f6 - f7 - f8 (four bits per term: direction, 15 for none; a bit per sign)
    const unsigned long long order = k == 1 ? 0xfff876531ull : (k == 2 ? 0xfff876542ull : 0x876543210ull);
    const unsigned minus = k == 1 ? 0x01au : (k == 2 ? 0x032u : 0u);
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int d = (int)(order >> (4 * j)) & 15;
        const double v = __shfl_sync(kAll, mine, base + (d < 9 ? d : 0));
        const double w = __hiloint2double(__double2hiint(v) ^ (int)(((minus >> j) & 1u) << 31), __double2loint(v));
        const double sum = j == 0 ? w : A::add(acc, w);
        acc = d < 9 ? sum : acc;
    }
    const double rho = __shfl_sync(kAll, acc, base);
    bool slow = false;
    double u = quot64(acc, recip64(rho, slow), slow);
    if (slow) u = A::div(acc, rho);
    const double ux = __shfl_sync(kAll, u, base + 1), uy = __shfl_sync(kAll, u, base + 2);
    // f*_k as in feq9<double>
    const double usq = A::add(A::mul(ux, ux), A::mul(uy, uy));
    const double t3 = A::mul(3.0, usq);
    const double both = (k == 6 || k == 8) ? A::sub(uy, ux) : A::add(ux, uy);
    const double c = k == 0 ? 0.0 : ((k == 1 || k == 3) ? ux : ((k == 2 || k == 4) ? uy : both));
    const bool opp = k == 3 || k == 4 || k == 7 || k == 8;
    const double c3 = A::mul(3.0, c), s9 = A::mul(9.0, A::mul(c, c));
    const double poly = fma(t3, -0.5, fma(s9, 0.5, A::add(1.0, opp ? -c3 : c3)));
    const double fs = A::mul(A::mul(rho, Lat<9>::w(k)), poly);
    // collision and the dS term
    const double fp = A::add(fs, A::mul(a2b, A::sub(fs, mine)));
    const double d = A::sub(fp, fs), dd = A::mul(d, d);
    bool slow_t = false;
    double term = quot64(dd, recip64(fs, slow_t), slow_t);
    if (slow_t) term = A::div(dd, fs);
    const unsigned bad_lanes = __ballot_sync(kAll, !gt0(fs) || !finite64(mine));
    double s = __shfl_sync(kAll, term, base);
#pragma unroll
    for (int j = 1; j < 9; ++j) s = A::add(s, __shfl_sync(kAll, term, base + j));
    const bool bad = ((bad_lanes >> base) & 0x1ffu) != 0 || !gt0(rho) || !finite64(rho) || !finite64(ux) || !finite64(uy);
    return !bad && finite64(s) && s > delta_e ? s : -1.0;
}

template <typename S>
__device__ __noinline__ double key_dS9_group(const KeyGeom p, const S *src, int site, double delta_e)
{
    if (p.eq == 1) return key_ent9<S>(p, src, site, delta_e);
    const int lane = threadIdx.x & 31, k = lane < 27 ? lane % 9 : lane - 27;
    return key_dS9_core(pull_one_f64<S>(p, src, site % p.nx, site / p.nx, k), p.a, delta_e);
}

// The same key evaluated by one thread alone (lane-parallel keying of many
// candidates: each lane keys its own site).
template <typename S>
__device__ __noinline__ double key_dS9_lane(const KeyGeom p, const S *src, int site, double delta_e)
{
    if (p.eq == 1) return key_ent9<S>(p, src, site, delta_e);
    const int x = site % p.nx, y = site / p.nx;
    double fin[9], fs[9], fp[9], ds, dsin, rho;
#pragma unroll
    for (int k = 0; k < 9; ++k) fin[k] = pull_one_f64<S>(p, src, x, y, k);
    const bool bad = site_poly64<9>(fin, p.a, true, fs, fp, ds, dsin, rho, false);
    return !bad && ds > delta_e ? ds : -1.0;
}

// The key of a D1Q3 site (closed or periodic tube) by one thread.
template <typename S>
__device__ __noinline__ double key_dS3_lane(const KeyGeom p, const S *src, int x, double delta_e)
{
    const bool wrap = bc_wrap_x(p.boundary);
    int r = x + 1, l = x - 1;
    if (r >= p.nx) r = wrap ? 0 : -1;
    if (l < 0) l = wrap ? p.nx - 1 : -1;
    auto at = [&](int k, int xx) { return Ar<double>::add((double)s2f(src[(long long)k * p.plane + kLead + xx]), p.rw(k)); };
    double fin[3], fs[3], fp[3], ds, dsin, rho;
    fin[0] = at(0, x);
    fin[1] = at(r >= 0 ? 1 : 2, r >= 0 ? r : x);
    fin[2] = at(l >= 0 ? 2 : 1, l >= 0 ? l : x);
    const bool bad = site_collide<3, double>(fin, p.a, true, fs, fp, ds, dsin, rho, p.eq, false);
    return !bad && ds > delta_e ? ds : -1.0;
}

template <int Q, typename S>
__device__ __forceinline__ double key_dS_lane(const KeyGeom &p, const S *src, int site, double delta_e)
{
    if constexpr (Q == 9)
        return key_dS9_lane<S>(p, src, site, delta_e);
    else
        return key_dS3_lane<S>(p, src, site, delta_e);
}

}  // namespace lbm
