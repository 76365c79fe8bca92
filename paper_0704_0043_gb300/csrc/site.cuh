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
template <typename S, typename T>
__device__ __forceinline__ T load_as(const StepParams &p, S v, int k)
{
    if constexpr (std::is_same<S, double>::value)
        return T(v);
    else if constexpr (std::is_same<T, double>::value)
        return Ar<double>::add((double)s2f(v), p.rw[k]);
    else
        return s2f(v);
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

// The populations of a boundary node that stream back onto the lattice, summed in
// k order: FP64 storage f itself, FP32 / 16-bit storage the absolute f (W = true)
// or the deviations alone.
template <typename T, typename R, bool W>
__device__ __forceinline__ R wall_mass(const StepParams &p, int x, int y, const T fin[9])
{
    R m = R(0);
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        const int dx = x + Lat<9>::cx(k), dy = y + Lat<9>::cy(k);
        if (dx >= 0 && dx < p.nx && dy >= 0 && dy < p.ny) {
            if constexpr (W && std::is_same<T, float>::value)
                m += (R)fin[k] + p.rw[k];
            else
                m = Ar<R>::add(m, (R)fin[k]);
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
