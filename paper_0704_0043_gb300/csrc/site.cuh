// site.cuh -- what a site of any lattice and boundary reads: free flight, the
// boundary-node rules, the median stencil (tiled and resident kernels).
#pragma once

#include <type_traits>

#include "internal.h"
#include "lattice.cuh"

namespace lbm {
namespace {

__device__ __forceinline__ long long fidx(long long plane, int pitch, int k, int y, int x)
{
    return (long long)k * plane + (long long)y * pitch + kLead + x;
}

// Stored value as a compute value: FP64 storage is f itself; FP32 / BF16 /
// FP16 storage is the deviation g, read as g in FP32 or as the absolute
// f = (double) g + rw_k in FP64.
template <typename S, typename T, typename P>
__device__ __forceinline__ T load_as(const P &p, S v, int k)
{
    if constexpr (std::is_same<S, double>::value)
        return T(v);
    else if constexpr (std::is_same<T, double>::value)
        return Ar<double>::add((double)s2f(v), p.rw[k]);
    else
        return s2f(v);
}

// (double) v and (float) v on integers (a conversion takes the FP64 unit as long as
// an addition does); subnormal and nonfinite values by the conversion itself, out
// of line (inline, the compiler runs it for every value and selects).
__device__ __noinline__ double widen_rare(float v) { return (double)v; }
__device__ __noinline__ float narrow_rare(double v) { return (float)v; }
__device__ __forceinline__ double widen(float v)
{
    const unsigned u = __float_as_uint(v), e = (u >> 23) & 0xffu;
    if (e - 1u >= 0xfeu && (u << 1) != 0) return widen_rare(v);
    const unsigned hi = (u << 1) != 0 ? ((u & 0x7fffffffu) >> 3) + (896u << 20) : 0u;
    return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ float narrow(double v)
{
    const unsigned h = (unsigned)__double2hiint(v), l = (unsigned)__double2loint(v);
    const unsigned e = (h >> 20) & 0x7ffu;
    if (e - 897u >= 253u) {  // zero, else below 2^-126, above 2^127 or nonfinite
        if (((h << 1) | l) == 0) return __uint_as_float(h);
        return narrow_rare(v);
    }
    unsigned m = (((h & 0x7fffffffu) << 3) | (l >> 29)) - (896u << 23);
    const unsigned rest = l & 0x1fffffffu;
    m += rest > 0x10000000u || (rest == 0x10000000u && (m & 1u));  // to nearest, ties to even
    return __uint_as_float(m | (h & 0x80000000u));
}

// v 2^e as a double, to nearest (ties to even); the result's exponent is normal.
__device__ __forceinline__ double fixed_value(long long v, int e)
{
    if (v == 0) return 0.0;
    unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)m);
    m <<= lz;
    unsigned long long t = m >> 11;
    const unsigned rest = (unsigned)m & 0x7ffu;
    t += rest > 0x400u || (rest == 0x400u && (t & 1ull));
    t += (unsigned long long)(63 - lz + e + 1022) << 52;
    return __longlong_as_double((long long)(t | ((unsigned long long)(v < 0) << 63)));
}

// rho, u of a site's stored populations (Eq. macro_dis; lbm_moments and the control
// point).  FP64 storage: the FP64 formula.  FP32 / 16-bit storage: the sums of the
// deviations in fixed point, in units of 2^(exponent of rho_ref - 58): a deviation below
// 2^exponent in size as a high part of 28 bits and a low part of 31, rounded once, so
// exact for deviations of at least 2^(exponent - 35) and off by at most half a unit
// below.  (The FP64 sum rounds a population to its own last place: half a unit on the
// diagonals of D2Q9 at rho_ref = 1, two units on the axes.)  The sums are exact and added
// to rho_ref sum W (every rho_ref W_k is a whole number of units); the quotients from one
// reciprocal, corrected by their residuals.  That is eight FP64 instructions (five for
// D1Q3), and no less exact than the FP64 sums, which round every sum too.
// A site with a deviation of rho_ref or more, or rho <= 0, takes the FP64 formula.
template <int Q, typename S, typename P>
__device__ __forceinline__ void site_moments(const P &p, const S raw[Q], double &rho, double &ux, double &uy)
{
    if constexpr (!std::is_same<S, double>::value) {
        int h[3] = {0, 0, 0};  // sums of g, c_x g, c_y g: at most nine of 2^27,
        long long l[3] = {0, 0, 0};  // and of 2^30
        bool plain = true;
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const float g = s2f(raw[k]);
            plain = plain && fabsf(g) < p.mfx.lim;
            const float x = __fmul_rn(g, p.mfx.scale);  // below 2^27, exact
            const int hi = __float2int_rn(x);
            const int lo = __float2int_rn(__fmul_rn(__fsub_rn(x, __int2float_rn(hi)), 2147483648.0f));
            h[0] += hi;
            l[0] += lo;
            h[1] += Lat<Q>::cx(k) * hi;
            l[1] += (long long)Lat<Q>::cx(k) * lo;
            h[2] += Lat<Q>::cy(k) * hi;
            l[2] += (long long)Lat<Q>::cy(k) * lo;
        }
        auto units = [&](int j) { return (long long)h[j] * (1ll << 31) + l[j]; };
        const long long r = p.mfx.rest + units(0), jx = units(1), jy = units(2);
        if (plain && r > 0) {
            bool slow = false;
            rho = fixed_value(r, p.mfx.exp);
            const Recip64 R = recip64(rho, slow);
            const double a = fixed_value(jx, p.mfx.exp), a0 = __dmul_rn(a, R.y);
            ux = fma(fma(-rho, a0, a), R.y, a0);
            uy = 0.0;
            if constexpr (Q == 9) {
                const double b = fixed_value(jy, p.mfx.exp), b0 = __dmul_rn(b, R.y);
                uy = fma(fma(-rho, b0, b), R.y, b0);
            }
            if (!slow) return;
        }
    }
    double f[Q];
#pragma unroll
    for (int k = 0; k < Q; ++k) f[k] = load_as<S, double>(p, raw[k], k);
    moments<Q, double>(f, rho, ux, uy);
}

// Free flight in pull form at site (x, y) (Sec. 2): f_in_k(x) = f_k(x - v_k);
// a link leaving the lattice is reflected, f_in_k(x) = f_opp(k)(x) (halfway
// bounce-back, Sec. 4.4.1), plus the moving-wall term for links through the lid.
// pull_raw reads storage type S: the address is selected, not the load, so all Q
// loads are in flight together also at the edges (one branch per link made them
// wait for one another, Q times the latency of L2).  `edge` = false: no link
// leaves the lattice; `wall`: a boundary node, whose links from outside read the
// node's own value of their direction.  pulled converts to compute type T (see
// load_as) and adds the lid terms.
template <int Q, typename S>
__device__ __forceinline__ void pull_raw(const StepParams &p, const S *f, int x, int y, bool edge, bool wall, S raw[Q])
{
    if (!edge) {
        const S *at = f + fidx(p.plane, p.pitch, 0, y, x);
#pragma unroll
        for (int k = 0; k < Q; ++k)
            raw[k] = at[(long long)k * p.plane - Lat<Q>::cy(k) * p.pitch - Lat<Q>::cx(k)];
        return;
    }
    const bool wrapx = bc_wrap_x(p.boundary);
    const bool wrapy = (Q == 9) && bc_wrap_y(p.boundary);
    const int xl = x > 0 ? x - 1 : (wrapx ? p.nx - 1 : -1), xr = x + 1 < p.nx ? x + 1 : (wrapx ? 0 : -1);
    const int yl = y > 0 ? y - 1 : (wrapy ? p.ny - 1 : -1), yr = y + 1 < p.ny ? y + 1 : (wrapy ? 0 : -1);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        const int sx = Lat<Q>::cx(k) > 0 ? xl : (Lat<Q>::cx(k) < 0 ? xr : x);
        const int sy = Lat<Q>::cy(k) > 0 ? yl : (Lat<Q>::cy(k) < 0 ? yr : y);
        const bool out = sx < 0 || sy < 0;
        raw[k] = f[fidx(p.plane, p.pitch, out && !wall ? Lat<Q>::opp(k) : k, out ? y : sy, out ? x : sx)];
    }
}

template <int Q, typename S, typename T>
__device__ __forceinline__ void pulled(const StepParams &p, int y, const S raw[Q], T fin[Q])
{
    using A = Ar<T>;
    const bool lid = Q == 9 && y + 1 == p.ny && !bc_wrap_y(p.boundary);
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        fin[k] = load_as<S, T>(p, raw[k], k);  // W_opp(k) = W_k
        if (Q == 9 && Lat<Q>::cy(k) < 0 && lid) {  // through the lid: a link that left
            if constexpr (std::is_same<T, double>::value)
                fin[k] = A::add(fin[k], p.lid[k]);
            else
                fin[k] = A::add(A::add(fin[k], p.lidf[k]), p.lidlo[k]);
        }
    }
}

template <int Q, typename S, typename T>
__device__ __forceinline__ void pull(const StepParams &p, const S *f, int x, int y, T fin[Q])
{
    S raw[Q];
    pull_raw<Q, S>(p, f, x, y, true, false, raw);
    pulled<Q, S, T>(p, y, raw, fin);
}

// Free flight and the wall rule at a boundary node (x, y) of a cavity whose
// outer ring of nodes lies on the walls (LBM_BC_NODE_WALLS, LBM_BC_DIFFUSIVE;
// Sec. 4.4): the populations whose source is on the lattice arrive; the others
// are supplied by the wall.  The lid is the top row without its corners and
// moves with (u_lid, 0); the other walls and the corners are at rest.
//   bounce-back (Sec. 4.4.1): f_k = f_opp(k) + 6 W_k rho_wall (v_k . u_wall);
//   diffusive (Sec. 4.4.2): f_k = gamma f*_k(1, u_wall), gamma = (sum of the
//     arrived f_opp(k)) / (sum of f*_k(1, u_wall)) over the returned
//     directions, evaluated in FP64 for every storage type; bounce-back in the
//     corners.
// A corner's two missing populations whose opposite is missing too point out
// of the lattice again; they keep their stored values.  fw: f*(1, u_wall) of the
// node's wall (wall_star), read by the diffusive rule only; raw: from pull_raw.
__device__ __forceinline__ void wall_star(const StepParams &p, bool lid, double fw[9])
{
    feq_any<9>(p.eq, 1.0, lid ? p.u_lid : 0.0, 0.0, fw);  // density is a linear factor of f*: take 1
}
__device__ __forceinline__ bool wall_corner(const StepParams &p, int x, int y)
{
    return (x == 0 || x == p.nx - 1) && (y == 0 || y == p.ny - 1);
}
__device__ __forceinline__ bool wall_lid(const StepParams &p, int x, int y)
{
    return y == p.ny - 1 && !wall_corner(p, x, y);
}

template <typename S, typename T>
__device__ __forceinline__ void wall_node(const StepParams &p, const S raw[9], int x, int y, const double *fw, T fin[9])
{
    using A = Ar<T>;
    bool known[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int sx = x - Lat<9>::cx(k), sy = y - Lat<9>::cy(k);
        known[k] = sx >= 0 && sx < p.nx && sy >= 0 && sy < p.ny;
        fin[k] = load_as<S, T>(p, raw[k], k);
    }
    const bool lid = wall_lid(p, x, y);
    if (p.boundary == 4 && !wall_corner(p, x, y)) {
        double arrived = 0.0, returned = 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k)
            if (!known[k]) {
                const int o = Lat<9>::opp(k);
                arrived = Ar<double>::add(arrived, load_as<S, double>(p, raw[o], o));
                returned = Ar<double>::add(returned, fw[k]);
            }
        const double gamma = Ar<double>::div(arrived, returned);
#pragma unroll
        for (int k = 0; k < 9; ++k)
            if (!known[k]) {
                const double v = Ar<double>::mul(gamma, fw[k]);
                if constexpr (std::is_same<T, double>::value)
                    fin[k] = v;
                else
                    fin[k] = (T)Ar<double>::sub(v, p.rw[k]);  // the deviation, rounded once
            }
    } else {
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            if (known[k]) continue;
            const int o = Lat<9>::opp(k);
            if (known[o]) {
                T v = fin[o];
                if (lid) {
                    if constexpr (std::is_same<T, double>::value)
                        v = A::add(v, p.lid[k]);
                    else
                        v = A::add(A::add(v, p.lidf[k]), p.lidlo[k]);
                }
                fin[k] = v;
            }  // else the stored value, already there
        }
    }
}

// Population k of a boundary node streams back onto the lattice, so the mass counts it.
__device__ __forceinline__ bool wall_counts(const StepParams &p, int x, int y, int k)
{
    const int dx = x + Lat<9>::cx(k), dy = y + Lat<9>::cy(k);
    return dx >= 0 && dx < p.nx && dy >= 0 && dy < p.ny;
}
// Their sum in k order: FP64 storage f itself, FP32 / 16-bit storage the absolute f.
template <typename T>
__device__ __forceinline__ double wall_mass(const StepParams &p, int x, int y, const T fin[9])
{
    double m = 0.0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        if (wall_counts(p, x, y, k)) {
            if constexpr (std::is_same<T, float>::value)
                m += (double)fin[k] + p.rw[k];
            else
                m = Ar<double>::add(m, fin[k]);
        }
    }
    return m;
}

__device__ __forceinline__ bool is_wall_node(const StepParams &p, int x, int y)
{
    return bc_node_walls(p.boundary) && (x == 0 || x == p.nx - 1 || y == 0 || y == p.ny - 1);
}

// Median of the dS stencil of site (x, y), tile-local position (tx, ty) in a
// shared array with row stride `ld` (Sec. 3.5; wall rules of Sec. 4.4, read for
// walls half a link outside the lattice: a node next to one wall uses itself
// and its two neighbours along that wall, a corner node itself and its inward
// x and y neighbours, every other node the 3x3 block; the two end sites of a
// closed D1Q3 tube are not filtered).  Returns false for sites the filter skips.
template <int Q, typename T>
__device__ __forceinline__ bool stencil_median(const StepParams &p, const T *s, int ld, int tx, int ty,
                                               int x, int y, T &med)
{
#define S_(dx, dy) s[(ty + (dy)) * ld + tx + (dx)]
    if constexpr (Q == 3) {
        if (p.boundary == 0 && (x == 0 || x == p.nx - 1)) return false;
        med = med3(S_(-1, 0), S_(0, 0), S_(1, 0));
        return true;
    } else {
        if (bc_node_walls(p.boundary)) {
            // boundary nodes are not filtered; their neighbours use stencils
            // along the wall (Sec. 4.4)
            if (x == 0 || x == p.nx - 1 || y == 0 || y == p.ny - 1) return false;
            const bool nx1 = x == 1 || x == p.nx - 2, ny1 = y == 1 || y == p.ny - 2;
            if (nx1 && ny1) {
                med = med3(S_(0, 0), S_(x == 1 ? 1 : -1, 0), S_(0, y == 1 ? 1 : -1));
            } else if (ny1) {
                med = med3(S_(-1, 0), S_(0, 0), S_(1, 0));
            } else if (nx1) {
                med = med3(S_(0, -1), S_(0, 0), S_(0, 1));
            } else {
                med = med9(S_(-1, -1), S_(-1, 0), S_(-1, 1), S_(0, -1), S_(0, 0), S_(0, 1), S_(1, -1), S_(1, 0),
                           S_(1, 1));
            }
            return true;
        }
        const bool wallx = p.boundary == 0, wally = p.boundary != 1;
        const bool nearx = wallx && (x == 0 || x == p.nx - 1);
        const bool neary = wally && (y == 0 || y == p.ny - 1);
        if (nearx && neary) {
            const int dx = x == 0 ? 1 : -1, dy = y == 0 ? 1 : -1;
            med = med3(S_(0, 0), S_(dx, 0), S_(0, dy));
        } else if (neary) {
            med = med3(S_(-1, 0), S_(0, 0), S_(1, 0));
        } else if (nearx) {
            med = med3(S_(0, -1), S_(0, 0), S_(0, 1));
        } else {
            med = med9(S_(-1, -1), S_(-1, 0), S_(-1, 1), S_(0, -1), S_(0, 0), S_(0, 1), S_(1, -1), S_(1, 0),
                       S_(1, 1));
        }
        return true;
    }
#undef S_
}

}  // namespace
}  // namespace lbm
