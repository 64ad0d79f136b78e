// iblb_kernels.cu -- sm_103a kernels of one IBLB droplet step
// (arXiv:2403.01161, Sec. 3.1-3.3).
//
// Lattice: D3Q19 populations stored in place with the AA access pattern as
// deviations g_i = f_i - w_i (rho_0 = 1), structure of arrays [19][qs] with
// x fastest.  An even step reads slot i of node x and writes the
// post-collision value back to slot opp(i) of the same node; an odd step
// reads slot opp(i) of node x - c_i and writes slot i of node x + c_i.  Wet
// boundary nodes rebuild the populations whose source lies outside the box
// on both parities (Zou-He face rule, edge and corner rules), and skip the
// loads and stores that would leave the box, so no halo is needed.
//
// Immersed boundary: node positions and nodal forces in FP64; the Eulerian
// force and velocity live in full-size arrays of the population type, but
// only the droplet patch (bounding box of the 4x4x4 stencils) is ever
// touched: the spread adds into it, the lattice kernel reads and re-zeroes it
// and stores the velocity there, the interpolation reads it.
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <algorithm>
#include <mutex>
#include <set>
#include <type_traits>
#include <utility>

#include "iblb_internal.h"
#include "iblb_device.cuh"

namespace iblb {
namespace {

// Half of the moving-wall difference f_eq(c_j) - f_eq(-c_j) at rho0 = 1:
// 3 w_j (c_j.u_w).
template <typename T, int J>
__device__ __forceinline__ T buried_wall_share(const T (&uw)[3])
{
    T cu = T(0);
    if constexpr (cxf(J) != 0) cu += T(cxf(J)) * uw[0];
    if constexpr (cyf(J) != 0) cu += T(cyf(J)) * uw[1];
    if constexpr (czf(J) != 0) cu += T(czf(J)) * uw[2];
    return T(3.0 * wgt(J)) * cu;
}

template <typename T, int SX, int SY, int SZ>
__device__ __forceinline__ void bc_apply(T (&f)[19], const T (&uw)[3], int rule)
{
    constexpr int NB = (SX != 0) + (SY != 0) + (SZ != 0);
    if constexpr (NB == 1) {
        // Face, Eq. (ZH_bulk) with the Zou-He closure for the density.
        constexpr int A = SX != 0 ? 0 : (SY != 0 ? 1 : 2);
        constexpr int SA = SX != 0 ? SX : (SY != 0 ? SY : SZ);
        const T un = T(SA) * uw[A];
        T sum_tan = 0, sum_out = 0;
        T P[3] = {0, 0, 0};  // tangential momentum of the in-plane populations
        sfor<19>([&](auto K) {
            constexpr int k = decltype(K)::value;
            if constexpr (comp(k, A) == 0) {
                sum_tan += f[k];
                if constexpr (cxf(k) != 0) P[0] += T(cxf(k)) * f[k];
                if constexpr (cyf(k) != 0) P[1] += T(cyf(k)) * f[k];
                if constexpr (czf(k) != 0) P[2] += T(czf(k)) * f[k];
            } else if constexpr (comp(k, A) * SA > 0) {
                sum_out += f[k];
            }
        });
        const T drho = (sum_tan + T(2) * sum_out - un) / (T(1) + un);
        const T rho = T(1) + drho;
        sfor<19>([&](auto J) {
            constexpr int j = decltype(J)::value;
            if constexpr (comp(j, A) * SA < 0) {
                constexpr int i = opp(j);
                constexpr int tn = (c2(i) == 2) ? 1 : 0;  // |t_i| for t_i = c_i - (c_i.n)n
                T cu = T(0), tu = T(0), corr = T(0);
                if constexpr (cxf(i) != 0) cu += T(cxf(i)) * uw[0];
                if constexpr (cyf(i) != 0) cu += T(cyf(i)) * uw[1];
                if constexpr (czf(i) != 0) cu += T(czf(i)) * uw[2];
                if constexpr (A != 0 && cxf(i) != 0) { tu += T(cxf(i)) * uw[0]; corr += T(cxf(i)) * P[0]; }
                if constexpr (A != 1 && cyf(i) != 0) { tu += T(cyf(i)) * uw[1]; corr += T(cyf(i)) * P[1]; }
                if constexpr (A != 2 && czf(i) != 0) { tu += T(czf(i)) * uw[2]; corr += T(czf(i)) * P[2]; }
                f[j] = f[i] - T(2 - tn) * rho * T(1.0 / 6.0) * cu - rho * T(1.0 / 3.0) * tu + T(0.5) * corr;
            }
        });
    } else if constexpr (NB == 2) {
        // Edge, Eq. (ZH_edges) (t_i = projection of c_i on the edge line),
        // then the buried links, Eq. (zh-buried-links-edges), f_0 = 12 f_b.
        // Counter-slip reading (default): the tangential sum with the face
        // rule's sign, so that it cancels the edge-line momentum f_{+e} -
        // f_{-e}, moving-wall bounce-back, the wall's edge-line share
        // -(t_i.u_w)/12, and each buried link plus its half of the
        // moving-wall difference 3 w_j (c_j.u_w): the node then carries
        // exactly u_w (rho0 = 1).  The literal rule: the printed sign and no
        // wall terms.
        constexpr int E = SX == 0 ? 0 : (SY == 0 ? 1 : 2);
        constexpr int PE = E + 1, ME = E + 10;  // +e_E and -e_E in the library order
        static_assert(comp(PE, E) == 1 && comp(ME, E) == -1, "axis links");
        const T dE = f[PE] - f[ME];
        const bool slip = (rule == IBL_EDGE_COUNTER_SLIP);
        sfor<19>([&](auto J) {
            constexpr int j = decltype(J)::value;
            if constexpr (j != 0 && unknown_dir<SX, SY, SZ>(j) && !unknown_dir<SX, SY, SZ>(opp(j))) {
                constexpr int i = opp(j);
                T v = f[i];
                if constexpr (comp(i, E) != 0) v += (slip ? T(0.25) : T(-0.25)) * T(comp(i, E)) * dE;
                if (slip) {
                    T cu = T(0);
                    if constexpr (cxf(i) != 0) cu += T(cxf(i)) * uw[0];
                    if constexpr (cyf(i) != 0) cu += T(cyf(i)) * uw[1];
                    if constexpr (czf(i) != 0) cu += T(czf(i)) * uw[2];
                    v -= T(6.0 * wgt(i)) * cu;
                    if constexpr (comp(i, E) != 0) v -= T(1.0 / 12.0) * T(comp(i, E)) * uw[E];
                }
                f[j] = v;
            }
        });
        T sb = T(0);
        sfor<19>([&](auto I) {
            constexpr int i = decltype(I)::value;
            if constexpr (i != 0 && !(unknown_dir<SX, SY, SZ>(i) && unknown_dir<SX, SY, SZ>(opp(i)))) sb += f[i];
        });
        const T fb = sb * T(1.0 / 22.0);
        sfor<19>([&](auto J) {
            constexpr int j = decltype(J)::value;
            if constexpr (j != 0 && unknown_dir<SX, SY, SZ>(j) && unknown_dir<SX, SY, SZ>(opp(j)))
                f[j] = slip ? fb + buried_wall_share<T, j>(uw) : fb;
        });
        f[0] = T(12) * fb;
    } else if constexpr (NB == 3) {
        // Corner, Eq. (zh-buried-links-corners); non-buried unknowns take
        // (moving-wall) bounce-back, buried links (plus their moving-wall
        // share under the counter-slip reading); f_0 = 12 f_b.
        const bool wall = (rule == IBL_EDGE_COUNTER_SLIP);
        sfor<19>([&](auto J) {
            constexpr int j = decltype(J)::value;
            constexpr int cs = -(cxf(j) * SX + cyf(j) * SY + czf(j) * SZ);
            if constexpr (j != 0 && unknown_dir<SX, SY, SZ>(j) && cs != 0) {
                constexpr int i = opp(j);
                T v = f[i];
                if (wall) {
                    T cu = T(0);
                    if constexpr (cxf(i) != 0) cu += T(cxf(i)) * uw[0];
                    if constexpr (cyf(i) != 0) cu += T(cyf(i)) * uw[1];
                    if constexpr (czf(i) != 0) cu += T(czf(i)) * uw[2];
                    v -= T(6.0 * wgt(i)) * cu;
                }
                f[j] = v;
            }
        });
        T sb = T(0);
        sfor<19>([&](auto I) {
            constexpr int i = decltype(I)::value;
            constexpr int cs = cxf(i) * SX + cyf(i) * SY + czf(i) * SZ;
            if constexpr (i != 0 && cs != 0) sb += f[i];
        });
        const T fb = sb * T(1.0 / 18.0);
        sfor<19>([&](auto J) {
            constexpr int j = decltype(J)::value;
            constexpr int cs = cxf(j) * SX + cyf(j) * SY + czf(j) * SZ;
            if constexpr (j != 0 && cs == 0) f[j] = wall ? fb + buried_wall_share<T, j>(uw) : fb;
        });
        f[0] = T(12) * fb;
    }
}

// MIRRORED: no case on the x = nx - 1 wall.
template <typename T, bool MIRRORED>
__device__ __forceinline__ void bc_dispatch(T (&f)[19], const T (&uw)[3], int rule, int code)
{
#define IBL_BC_CASE(a, b, c)                                              \
    case (a + 1) + 3 * (b + 1) + 9 * (c + 1):                             \
        if constexpr (!(MIRRORED && a > 0)) bc_apply<T, a, b, c>(f, uw, rule); \
        break;
    switch (code) {
        IBL_BC_CASE(-1, 0, 0) IBL_BC_CASE(1, 0, 0) IBL_BC_CASE(0, -1, 0) IBL_BC_CASE(0, 1, 0)
        IBL_BC_CASE(0, 0, -1) IBL_BC_CASE(0, 0, 1)
        IBL_BC_CASE(-1, -1, 0) IBL_BC_CASE(1, -1, 0) IBL_BC_CASE(-1, 1, 0) IBL_BC_CASE(1, 1, 0)
        IBL_BC_CASE(-1, 0, -1) IBL_BC_CASE(1, 0, -1) IBL_BC_CASE(-1, 0, 1) IBL_BC_CASE(1, 0, 1)
        IBL_BC_CASE(0, -1, -1) IBL_BC_CASE(0, 1, -1) IBL_BC_CASE(0, -1, 1) IBL_BC_CASE(0, 1, 1)
        IBL_BC_CASE(-1, -1, -1) IBL_BC_CASE(1, -1, -1) IBL_BC_CASE(-1, 1, -1) IBL_BC_CASE(1, 1, -1)
        IBL_BC_CASE(-1, -1, 1) IBL_BC_CASE(1, -1, 1) IBL_BC_CASE(-1, 1, 1) IBL_BC_CASE(1, 1, 1)
        default: break;
    }
#undef IBL_BC_CASE
}

// ---------------------------------------------------------------------------
// Lattice update: streaming (AA pattern) + boundary rebuild + moments with
// half-force momentum + BGK + Guo source, Eqs. (LBMEQ)-(density_velocity_LB).
// One thread per node: outside the patch consecutive nodes of the flattened
// box, their coordinates by a division by constants (fast_div), in the patch
// the rows of its box.  Indices are 32-bit (19 * stride < 2^31 is checked on
// the host).  The collision works on opposite pairs (c_i, -c_i), whose
// equilibrium and source terms share their even parts.
// Node sets of one lattice launch: every node of a box without a droplet
// (FULL); only the nodes outside the droplet patch (FAR); only patch nodes
// (NEAR).  FAR and NEAR launches of the same step may run concurrently: in
// the AA pattern every population slot is read and written by one node only
// within a step.  Only patch nodes carry a force, so FULL and FAR compile
// without the Guo source.
enum { LAT_FULL = 0, LAT_FAR = 1, LAT_NEAR = 2 };

// 3 w_i, the weight of the odd (momentum) parts of the equilibrium and of
// the Guo source.  The exact values are 1/6 (|c_i|^2 = 1) and 1/12 (|c_i|^2
// = 2), and sum_i c_ia c_ia 3 w_i = 2/6 + 8/12 = 1 carries the momentum
// through the collision.  Rounded to nearest in FP32 both come out 2^-25
// relatively high, so that every collision would multiply the momentum by
// 1 + 3.0e-8 -- a bias that accumulates over the thousands of steps a
// velocity perturbation lives (L^2 / nu).  In FP32 1/6 is therefore rounded
// down instead (0x3E2AAAAA, 2^-24 relatively low), which makes
// 2 (3 w_1) + 8 (3 w_2) equal to 1 exactly; what remains of each product's
// error is its own rounding, without a common sign.
template <typename T, int i>
__device__ __forceinline__ T odd_weight()
{
    if constexpr (sizeof(T) == 4) return __int_as_float(c2(i) == 1 ? 0x3E2AAAAA : 0x3DAAAAAB);
    else return T(3.0 * wgt(i));
}

// Moments with half-force momentum, BGK and Guo source (FORCE) on the 19
// populations of a node, in place; returns whether it is unstable.  FP32: each
// population is relaxed from its own value, and the momentum terms keep the
// weights of odd_weight.
template <bool FORCE, typename T>
__device__ __forceinline__ bool collide(T (&g)[19], const T Fx, const T Fy, const T Fz, const T om, T &drho, T &ux, T &uy,
                                        T &uz)
{
    drho = T(0);
    T jx = T(0), jy = T(0), jz = T(0);
    sfor<19>([&](auto I) {
        constexpr int i = decltype(I)::value;
        drho += g[i];
        if constexpr (cxf(i) != 0) jx += T(cxf(i)) * g[i];
        if constexpr (cyf(i) != 0) jy += T(cyf(i)) * g[i];
        if constexpr (czf(i) != 0) jz += T(czf(i)) * g[i];
    });
    const T rho = T(1) + drho;
    const T ir = T(1) / rho;
    // rho u = j + F/2 (Eq. (density_velocity_LB)); the odd (momentum)
    // parts of the equilibrium are formed from it directly
    T mx = jx, my = jy, mz = jz;
    if constexpr (FORCE) {
        mx += T(0.5) * Fx;
        my += T(0.5) * Fy;
        mz += T(0.5) * Fz;
    }
    ux = mx * ir;
    uy = my * ir;
    uz = mz * ir;
    const T uu = ux * ux + uy * uy + uz * uz;
    const bool bad = !(uu <= T(0.09)) || !(drho == drho);
    [[maybe_unused]] T fpre, uF;
    if constexpr (FORCE) {
        fpre = T(1) - T(0.5) * om;
        uF = ux * Fx + uy * Fy + uz * Fz;
    }
    const T dmr = drho - rho * (T(1.5) * uu);  // drho - (3/2) rho u.u
    {
        constexpr double w0 = wgt(0);
        const T geq = T(w0) * dmr;
        g[0] = g[0] + om * (geq - g[0]);
        if constexpr (FORCE) g[0] += fpre * T(w0) * (T(-3) * uF);
    }
    sfor<9>([&](auto I) {
        constexpr int i = decltype(I)::value + 1;
        constexpr int j = opp(i);
        T cp = T(0);  // c_i . rho u
        if constexpr (cxf(i) != 0) cp += T(cxf(i)) * mx;
        if constexpr (cyf(i) != 0) cp += T(cyf(i)) * my;
        if constexpr (czf(i) != 0) cp += T(czf(i)) * mz;
        const T cu = cp * ir;
        constexpr double w = wgt(i);
        const T w3 = odd_weight<T, i>();
        const T even_eq = T(w) * (T(4.5) * cp * cu + dmr);
        const T odd_eq = w3 * cp;
        g[i] = g[i] + om * (even_eq + odd_eq - g[i]);
        g[j] = g[j] + om * (even_eq - odd_eq - g[j]);
        if constexpr (FORCE) {
            T cF = T(0);  // c_i . F
            if constexpr (cxf(i) != 0) cF += T(cxf(i)) * Fx;
            if constexpr (cyf(i) != 0) cF += T(cyf(i)) * Fy;
            if constexpr (czf(i) != 0) cF += T(czf(i)) * Fz;
            const T even_src = fpre * T(w) * (T(9) * cu * cF - T(3) * uF);
            const T odd_src = fpre * w3 * cF;
            g[i] += even_src + odd_src;
            g[j] += even_src - odd_src;
        }
    });
    return bad;
}

// FP64: the same on sums and differences of opposite populations, s = g_i +
// g_j and d = g_i - g_j: the moments need each once, and a pair relaxes as
//   g_i, g_j = [(1 - w)/2 s + w even_eq] +- [(1 - w)/2 d + w odd_eq]
// (w = omega), 143 FP64 instructions a node without force against 185: the
// FP64 pipe, one warp instruction per 16 cycles and SM, sets the FP64 step.
// (FP32 keeps `collide`: there this grouping rounds the momentum worse.)  u is
// formed only where it is stored (VEL).
template <bool FORCE, bool VEL, typename T>
__device__ __forceinline__ bool collide_pairs(T (&g)[19], const T Fx, const T Fy, const T Fz, const T om, T &drho, T &ux,
                                              T &uy, T &uz)
{
    drho = g[0];
    T mx = T(0), my = T(0), mz = T(0);  // rho u
    if constexpr (FORCE) {
        mx = T(0.5) * Fx;
        my = T(0.5) * Fy;
        mz = T(0.5) * Fz;
    }
    sfor<9>([&](auto I) {
        constexpr int i = decltype(I)::value + 1, j = opp(i);
        const T s = g[i] + g[j], d = g[i] - g[j];
        g[i] = s;
        g[j] = d;
        drho += s;
        if constexpr (cxf(i) != 0) mx += T(cxf(i)) * d;
        if constexpr (cyf(i) != 0) my += T(cyf(i)) * d;
        if constexpr (czf(i) != 0) mz += T(czf(i)) * d;
    });
    const T ir = T(1) / (T(1) + drho);
    const T ke = (mx * mx + my * my + mz * mz) * ir;  // rho u.u
    const bool bad = !(ke * ir <= T(0.09));           // NaN density included
    const T dmr = drho - T(1.5) * ke, q = T(4.5) * ir;
    const T keep = T(0.5) - T(0.5) * om;
    [[maybe_unused]] T fpre, uF;
    if constexpr (VEL) {
        ux = mx * ir;
        uy = my * ir;
        uz = mz * ir;
    }
    if constexpr (FORCE) {
        fpre = T(1) - T(0.5) * om;
        uF = ux * Fx + uy * Fy + uz * Fz;
    }
    g[0] = (keep + keep) * g[0] + (om * T(wgt(0))) * dmr;
    if constexpr (FORCE) g[0] -= (fpre * T(3.0 * wgt(0))) * uF;
    const T e1 = om * T(wgt(1)), e2 = om * T(wgt(4)), o1 = om * T(3.0 * wgt(1)), o2 = om * T(3.0 * wgt(4));
    sfor<9>([&](auto I) {
        constexpr int i = decltype(I)::value + 1, j = opp(i);
        constexpr bool axis = c2(i) == 1;
        T cp = T(0);  // c_i . rho u
        if constexpr (cxf(i) != 0) cp += T(cxf(i)) * mx;
        if constexpr (cyf(i) != 0) cp += T(cyf(i)) * my;
        if constexpr (czf(i) != 0) cp += T(czf(i)) * mz;
        T S = keep * g[i] + (axis ? e1 : e2) * (q * (cp * cp) + dmr);
        T D = keep * g[j] + (axis ? o1 : o2) * cp;
        if constexpr (FORCE) {
            T cF = T(0);  // c_i . F
            if constexpr (cxf(i) != 0) cF += T(cxf(i)) * Fx;
            if constexpr (cyf(i) != 0) cF += T(cyf(i)) * Fy;
            if constexpr (czf(i) != 0) cF += T(czf(i)) * Fz;
            S += fpre * T(wgt(i)) * (T(9) * (cp * ir) * cF - T(3) * uF);
            D += fpre * T(3.0 * wgt(i)) * cF;
        }
        g[i] = S + D;
        g[j] = S - D;
    });
    return bad;
}

// Population of the velocity c_i with its x component reversed.
__host__ __device__ constexpr int mirrored(int i)
{
    for (int j = 0; j < 19; ++j)
        if (cxf(j) == -cxf(i) && cyf(j) == cyf(i) && czf(j) == czf(i)) return j;
    return i;
}
template <typename T>
__device__ __forceinline__ void mirror_x(T (&g)[19], const bool on)
{
    sfor<19>([&](auto I) {
        constexpr int i = decltype(I)::value, j = mirrored(i);
        if constexpr (cxf(i) > 0) {
            const T a = g[i], b = g[j];
            g[i] = on ? b : a;
            g[j] = on ? a : b;
        }
    });
}

// Offsets to a node's neighbours along each axis (odd step), S to a node (its
// bytes, or 1).  Periodic axes wrap.  On a Zou-He axis a missing neighbour points back
// at the node itself: a population whose source lies outside the box is an
// unknown that the boundary rebuild overwrites before anything reads it, so
// its load only needs an address inside the array, while a store to a missing
// destination is left out: by the flags, or where an axis may be periodic by
// the bits of `miss` (six flags beside six run-time offsets made the periodic
// patch update of an ensemble spill 88 bytes, the bits 4).
struct Hops {
    int xm, xp, ym, yp, zm, zp;
    bool no_xm, no_xp, no_ym, no_yp, no_zm, no_zp;
    int miss;  // 1 x-1, 2 x+1, 4 y-1, 8 y+1, 16 z-1, 32 z+1
};
// Whether an odd update forms its addresses from element indices and its hops
// twice, before the loads and again for the stores, instead of byte offsets on
// common bases held across the collision.  Outside the patch of a box with a
// periodic axis, where the hops are selects at run time, that is fewer
// instructions and registers (FP32, us per step, byte offsets and indices:
// periodic 128^3 droplet 53.1 and 50.7, 160^3 100.4 and 97.3, 256^3 412.6 and
// 403.5, 64^3 12.37 and 12.45; channel without a droplet 64^3 6.06 and 5.59,
// 256^3 372.1 and 372.7; 32 periodic droplets 358.4 and 348.3).  FP64, set by
// its pipe, does not gain (64^3 droplet 94.0 and 94.7).
template <typename T, int MODE, bool PER>
constexpr bool kIndexed = sizeof(T) == 4 && PER && MODE != LAT_NEAR;
template <int S, bool PER>
__device__ __forceinline__ Hops make_hops(const LbView &L, const int x, const int y, const int z)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2], Sx = S * nx, Sxy = Sx * ny;
    const bool px = PER && L.bc[0] == IBL_BC_PERIODIC, py = PER && L.bc[1] == IBL_BC_PERIODIC,
               pz = PER && L.bc[2] == IBL_BC_PERIODIC;
    Hops h;
    h.no_xm = x == 0;
    h.no_xp = x == nx - 1;
    h.no_ym = y == 0;
    h.no_yp = y == ny - 1;
    h.no_zm = z == 0;
    h.no_zp = z == nz - 1;
    h.xm = h.no_xm ? (px ? Sx - S : 0) : -S;
    h.xp = h.no_xp ? (px ? S - Sx : 0) : S;
    h.ym = h.no_ym ? (py ? Sxy - Sx : 0) : -Sx;
    h.yp = h.no_yp ? (py ? Sx - Sxy : 0) : Sx;
    h.zm = h.no_zm ? (pz ? Sxy * (nz - 1) : 0) : -Sxy;
    h.zp = h.no_zp ? (pz ? -Sxy * (nz - 1) : 0) : Sxy;
    if (PER) {
        h.no_xm = h.no_xm && !px;
        h.no_xp = h.no_xp && !px;
        h.no_ym = h.no_ym && !py;
        h.no_yp = h.no_yp && !py;
        h.no_zm = h.no_zm && !pz;
        h.no_zp = h.no_zp && !pz;
    }
    h.miss = (h.no_xm ? 1 : 0) | (h.no_xp ? 2 : 0) | (h.no_ym ? 4 : 0) | (h.no_yp ? 8 : 0) | (h.no_zm ? 16 : 0) |
             (h.no_zp ? 32 : 0);
    return h;
}
// Offset of the neighbour along (CX, CY, CZ), and whether it exists.
template <int CX, int CY, int CZ>
__device__ __forceinline__ unsigned hop(const Hops &h)
{
    unsigned o = 0;
    if constexpr (CX != 0) o += (unsigned)(CX > 0 ? h.xp : h.xm);
    if constexpr (CY != 0) o += (unsigned)(CY > 0 ? h.yp : h.ym);
    if constexpr (CZ != 0) o += (unsigned)(CZ > 0 ? h.zp : h.zm);
    return o;
}
template <bool PER, int CX, int CY, int CZ>
__device__ __forceinline__ bool hop_exists(const Hops &h)
{
    if constexpr (PER) {
        constexpr int need = (CX > 0 ? 2 : (CX < 0 ? 1 : 0)) | (CY > 0 ? 8 : (CY < 0 ? 4 : 0)) |
                             (CZ > 0 ? 32 : (CZ < 0 ? 16 : 0));
        return (h.miss & need) == 0;
    }
    bool no = false;
    if constexpr (CX != 0) no = no || (CX > 0 ? h.no_xp : h.no_xm);
    if constexpr (CY != 0) no = no || (CY > 0 ? h.no_yp : h.no_ym);
    if constexpr (CZ != 0) no = no || (CZ > 0 ? h.no_zp : h.no_zm);
    return !no;
}

// The part of a node update after its 19 incoming populations g are in
// registers: boundary rebuild (sx, sy, sz: -1 / 0 / +1 where the node lies on
// a wall of that axis), patch force, moments, BGK + Guo, stores (AA pattern:
// even step own slots opp(i), odd step slot i at x + c_i), velocity record.
// Returns whether the node is unstable.
// CEN: the boundary field may be centred on the droplet (L.recentre); false
// where the host knows it is not, since the offset's FP64 arithmetic would
// otherwise be issued by every warp with a wall node, predicated off or not
// (nine FP64 instructions, 16 cycles each per SM).
template <typename T, bool ODD, bool REC, int MODE, bool PER, bool CEN, class P = L2Keep>
__device__ __forceinline__ bool lattice_finish(const LbView &L, T (&g)[19], const int x, const int y, const int z,
                                               const int node, const int pbuf, const int sx, const int sy, const int sz,
                                               [[maybe_unused]] const Hops &h_)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    constexpr bool FORCE = MODE == LAT_NEAR;
    bool bad = false;
    {
        T *__restrict__ f = static_cast<T *>(L.f);
        struct NoKeep {};
        [[maybe_unused]] const std::conditional_t<MODE == LAT_NEAR, P, NoKeep> K;
        const long long qs = L.qs;
        [[maybe_unused]] const unsigned noff = (unsigned)node * (unsigned)sizeof(T);
        if (sx | sy | sz) {
            // Eq. (velo_facce_cubo_da_gradiente) in the storage precision,
            // about the box centre or, with re-centring, about the droplet's
            // centre of mass at the start of the step (the offset in FP64)
            const T *A = static_cast<const T *>(L.frames_t) + 9 * L.ctl->frame_par[ODD ? 1 : 0];
            T lx, ly, lz;
            if (CEN && L.recentre) {
                const double *c = L.ctl->centre[pbuf];
                lx = T(double(x) - c[0]);
                ly = T(double(y) - c[1]);
                lz = T(double(z) - c[2]);
            } else {
                lx = T(x) - T(0.5) * T(nx - 1);
                ly = T(y) - T(0.5) * T(ny - 1);
                lz = T(z) - T(0.5) * T(nz - 1);
            }
            const T uw[3] = {A[0] * lx + A[1] * ly + A[2] * lz, A[3] * lx + A[4] * ly + A[5] * lz,
                             A[6] * lx + A[7] * ly + A[8] * lz};
            if constexpr (sizeof(T) == 4) {
                bc_dispatch<T, false>(g, uw, L.rule, (sx + 1) + 3 * (sy + 1) + 9 * (sz + 1));
            } else {
                // both x walls through one rebuild, the far one mirrored: a
                // warp that holds both (rows of 32 nodes and fewer, or rows
                // that are no multiple of 32) issues its FP64 instructions
                // once; the exchange is selects
                const bool mir = sx > 0;
                const T vw[3] = {mir ? -uw[0] : uw[0], uw[1], uw[2]};
                mirror_x(g, mir);
                bc_dispatch<T, true>(g, vw, L.rule, (mir ? 0 : sx + 1) + 3 * (sy + 1) + 9 * (sz + 1));
                mirror_x(g, mir);
            }
        }

        // droplet patch: read the spread force (and clear it), store u below;
        // both fields hold a 4-wide record (x, y, z, 0) per node
        T Fx = T(0), Fy = T(0), Fz = T(0);
        [[maybe_unused]] T *__restrict__ force = static_cast<T *>(L.force);
        if constexpr (FORCE) {
            K.ld3(force + 4 * node, Fx, Fy, Fz);
            K.st3(force + 4 * node, T(0), T(0), T(0));
        }

        T om = sizeof(T) == 4 ? T(L.omega_f) : T(L.omega);
        if constexpr (MODE == LAT_NEAR) {
            // viscosity ratio: relaxation of the inside nodes (flags read and cleared)
            if (L.visc) {
                unsigned char *flag = reinterpret_cast<unsigned char *>(L.ind) + node;
                if (*flag) om = sizeof(T) == 4 ? T(L.omega_in_f) : T(L.omega_in);
                *flag = 0;
            }
        }
        T drho, ux, uy, uz;
        if constexpr (sizeof(T) == 4) bad = collide<FORCE>(g, Fx, Fy, Fz, om, drho, ux, uy, uz);
        else bad = collide_pairs<FORCE, FORCE || REC>(g, Fx, Fy, Fz, om, drho, ux, uy, uz);

        if constexpr (!ODD) {
            sfor<19>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if constexpr (MODE == LAT_NEAR) K.st(slot_at(f, opp(i), qs, noff), g[i]);
                else *slot_at(f, opp(i), qs, noff) = g[i];
            });
        } else {
            // destination x + c_i, slot i.  The node's own offset passes
            // through an opaque move, so the neighbour offsets are summed
            // again here instead of being held in registers across the
            // collision; the patch-node update, which holds more, and the
            // indexed one form them anew from the coordinates (either way the
            // kernel spilled).
            constexpr bool IDX = kIndexed<T, MODE, PER>;
            unsigned here = noff;
            Hops h = h_;
            if constexpr (MODE == LAT_NEAR || IDX) {
                int xs = x, ys = y, zs = z;
                asm volatile("mov.b32 %0, %0;" : "+r"(xs));
                asm volatile("mov.b32 %0, %0;" : "+r"(ys));
                asm volatile("mov.b32 %0, %0;" : "+r"(zs));
                h = make_hops<IDX ? 1 : (int)sizeof(T), PER>(L, xs, ys, zs);
                if constexpr (IDX) here = (unsigned)(xs + nx * (ys + ny * zs));
            }
            if constexpr (!IDX) asm volatile("mov.b32 %0, %0;" : "+r"(here));
            sfor<19>([&](auto I) {
                constexpr int i = decltype(I)::value;
                if (hop_exists<PER, cxf(i), cyf(i), czf(i)>(h)) {
                    const unsigned o = here + hop<cxf(i), cyf(i), czf(i)>(h);
                    T *a = IDX ? f + (i * (int)qs + (int)o) : slot_at(f, i, qs, o);
                    if constexpr (MODE == LAT_NEAR) K.st(a, g[i]);
                    else *a = g[i];
                }
            });
        }
        if constexpr (MODE == LAT_NEAR) K.st3(static_cast<T *>(L.vel) + 4 * node, ux, uy, uz);
        if constexpr (REC) {
            const int nodes = L.nodes;
            T *__restrict__ rec = static_cast<T *>(L.rec);
            rec[node] = drho;
            rec[nodes + node] = ux;
            rec[2 * nodes + node] = uy;
            rec[3 * nodes + node] = uz;
            rec[4 * nodes + node] = Fx;
            rec[5 * nodes + node] = Fy;
            rec[6 * nodes + node] = Fz;
        }
    }
    return bad;
}

// One node update with its loads from global memory.
// PER: some axis may be periodic (false: every axis has Zou-He walls, so
// the neighbour offsets are fixed and only the boundary tests remain).
// P: L2 policy of the patch nodes' accesses (LAT_NEAR).
template <typename T, bool ODD, bool REC, int MODE, bool PER, bool CEN, class P = L2Keep>
__device__ __forceinline__ bool lattice_node(const LbView &L, const int x, const int y, const int z, const int node,
                                             const int pbuf)
{
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    // the patch of this step lives in buffer pbuf (step % 3)
    if constexpr (MODE == LAT_FAR) {
        if (node_in_patch<PER>(L, L.ctl, pbuf, x, y, z)) return false;
    }
    {
        T *__restrict__ f = static_cast<T *>(L.f);
        // the patch nodes keep their lines in L2 between steps (see L2Keep)
        struct NoKeep {};
        [[maybe_unused]] const std::conditional_t<MODE == LAT_NEAR, P, NoKeep> K;
        const long long qs = L.qs;
        const bool px = PER && L.bc[0] == IBL_BC_PERIODIC, py = PER && L.bc[1] == IBL_BC_PERIODIC,
                   pz = PER && L.bc[2] == IBL_BC_PERIODIC;
        const int sx = px ? 0 : (x == 0 ? -1 : (x == nx - 1 ? 1 : 0));
        const int sy = py ? 0 : (y == 0 ? -1 : (y == ny - 1 ? 1 : 0));
        const int sz = pz ? 0 : (z == 0 ? -1 : (z == nz - 1 ? 1 : 0));
        // the patch-node update guards its loads too, which measured faster there
        [[maybe_unused]] Hops h{};
        constexpr bool IDX = kIndexed<T, MODE, PER>;
        if constexpr (ODD) h = make_hops<IDX ? 1 : (int)sizeof(T), PER>(L, x, y, z);
        [[maybe_unused]] const unsigned noff = (unsigned)node * (unsigned)sizeof(T);

        T g[19];
        if constexpr (!ODD) {
            sfor<19>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const T *a = slot_at(f, i, qs, noff);
                if constexpr (MODE == LAT_NEAR) g[i] = K.ld(a);
                else g[i] = *a;
            });
        } else {
            // source x - c_i, slot opp(i)
            sfor<19>([&](auto I) {
                constexpr int i = decltype(I)::value;
                const unsigned o = hop<-cxf(i), -cyf(i), -czf(i)>(h);
                const T *a = IDX ? f + (opp(i) * (int)qs + node + (int)o) : slot_at(f, opp(i), qs, noff + o);
                if constexpr (MODE == LAT_NEAR)
                    g[i] = hop_exists<PER, -cxf(i), -cyf(i), -czf(i)>(h) ? K.ld(a) : T(0);
                else g[i] = *a;
            });
        }

        return lattice_finish<T, ODD, REC, MODE, PER, CEN, P>(L, g, x, y, z, node, pbuf, sx, sy, sz, h);
    }
}

// Sets the sticky instability flag.  Once it is set, further warps only look
// (a line their SM has cached): a box that has gone unstable has every warp
// here at every step, all on one address.
__device__ __forceinline__ void flag_unstable(const LbView &L)
{
    if ((L.ctl->err & IBL_ERRBIT_UNSTABLE) == 0) atomicOr(&L.ctl->err, IBL_ERRBIT_UNSTABLE);
}

// Closes step t: the step counter becomes t + 1 and the frame of step t + 1
// goes to its parity's slot.  The lattice kernel of step t and the patch
// update of step t read the other slot, and the kernels of step t - 1, the
// last readers of this one, have finished (both are ordered before the
// lattice kernel of step t), so one thread of that kernel can do it while the
// rest of the step runs: no separate launch sits between two lattice updates.
__device__ __forceinline__ void close_step(const LbView &L)
{
    const long long s = L.ctl->step + 1;
    L.ctl->step = s;
    const long long k = s / L.n_hold;
    L.ctl->frame_par[s & 1] = (int)(k < L.n_frames - 1 ? k : L.n_frames - 1);
}

// One node per thread, 128 consecutive nodes of the flattened box per block,
// so that every lane works in a box of any size (rows of 200 nodes left 22% of
// the lanes of row-aligned blocks idle) and every warp's run starts on a
// 128-byte line of each population array.  Co-limited by HBM and instruction
// issue: without the force terms where there is no force, and with 32-bit
// offsets on common bases, a 64^3 far launch issues 536 (even) / 730 (odd)
// instructions per warp against 643 / 765 before.  Per step: 97 x 75 x 61
// channel 16.5 -> 12.3 us, 200^3 regularised 228 -> 212 us, 128^3 droplet
// 57.1 -> 55.0 us, 256^3 within 0.3%.
// TILES: blocks take that many tiles in turn.
template <typename T, bool ODD, bool REC, int MODE, bool PER, bool CEN, int TILES>
__global__ void __launch_bounds__(128, sizeof(T) == 4 ? 8 : 4) k_lattice(LbView L, int pbuf, int ahead)
{
    int node = (int)(blockIdx.x * (128u * TILES) + threadIdx.x);
    if (node == 0) close_step(L);
    bool bad = false;
#pragma unroll 1
    for (int k = 0; k < TILES; ++k, node += 128) {
        // L2 prefetch of the node `ahead` nodes on, which a block of about one
        // resident wave later updates: its loads then find the lines in L2
        // instead of waiting on DRAM behind the stream (ahead = 0: none, see
        // prefetch_distance)
        if (ahead > 0 && node + ahead < L.nodes) {
            T *f = static_cast<T *>(L.f);
            const unsigned off = (unsigned)(node + ahead) * (unsigned)sizeof(T);
#pragma unroll
            for (int i = 0; i < 19; ++i) asm volatile("prefetch.global.L2 [%0];" ::"l"(slot_at(f, i, L.qs, off)));
        }
        if (node < L.nodes) {
            const int z = fast_div(node, L.div_nxy), p = node - z * L.n[0] * L.n[1];
            const int y = fast_div(p, L.div_nx), x = p - y * L.n[0];
            bad |= lattice_node<T, ODD, REC, MODE, PER, CEN>(L, x, y, z, node, pbuf);
        }
    }
    // sticky instability flag, one atomic per warp at most
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if (m != 0u && (threadIdx.x & 31) == 0) flag_unstable(L);
}

// Outside update (FAR) or whole-box update (FULL) through a shared-memory
// pipeline, for FP32 populations in a box with Zou-He walls on every axis.
// The one-thread-per-node kernel above holds its 19 loads in registers, so
// the bytes it keeps in flight are capped by the resident threads (8 blocks
// of 128 at 64 registers fill the register file), and a droplet-kernel
// block that takes a slot on an SM cuts that SM's share of the stream.
// Here each block is persistent (B per SM) and walks tiles of NT
// consecutive nodes of the flattened box; warp 0 stages the 19 source runs
// of a tile (one lane per run) with bulk asynchronous copies (cp.async.bulk,
// completion counted in bytes on an mbarrier) S tiles ahead, so the bytes in
// flight do not depend on registers.  On GB300 it measures slower than the
// direct kernel in every launch shape (the update is co-limited by
// instruction issue, and the pipeline adds instructions and holds its SM
// resources for the whole launch); it is selected by ibl_set_outside_update.
// Source runs: even step, slot i of the tile's own nodes; odd step, slot
// opp(i) of the nodes n - o_i, o_i = c_ix + c_iy nx + c_iz nx ny (the
// source x - c_i).  A run [n0 - o_i, n0 - o_i + NT) is widened down to the
// 16-byte boundary u_i = (n0 - o_i) & ~3 and up to the next one, and placed
// in its stage slot as if it started at u_i, so that node n0 + t reads
// element t + d_i with d_i = (n0 - o_i) - u_i = (-o_i) & 3 (n0 is a multiple
// of 4), the same for every tile.  The part of a widened run outside its
// array is not copied: those elements, like any other element of a source
// outside the box (a row, plane or array end crossed), are unknowns the
// boundary rebuild overwrites.  Stores go straight from registers
// (lattice_finish).
constexpr unsigned long long kStageWaitNs = 1000000000ull;  // a stage that has not arrived after 1 s is lost
constexpr unsigned long long kDrainWaitNs = 200000000ull;  // then each copy still in flight gets 0.2 s

template <int NT>
__host__ __device__ constexpr int stage_run()
{
    return NT + 8;  // floats per population per stage: NT plus the widening to 16-byte boundaries
}

template <int NT, int S>
__host__ __device__ constexpr size_t stage_bytes()
{
    return sizeof(float) * (size_t)S * 19 * stage_run<NT>();
}

template <bool ODD, int i>
__device__ __forceinline__ int src_offset(const int nx, const int nxy)
{
    return ODD ? cxf(i) + cyf(i) * nx + czf(i) * nxy : 0;
}

// a / b for 0 <= a < 2^26 and b >= 1 from a float reciprocal, corrected to
// the exact quotient
__device__ __forceinline__ int div_by(const int a, const int b, const float inv_b)
{
    int q = __float2int_rz(__int2float_rn(a) * inv_b);
    const int r = a - q * b;
    q += (r >= b) - (r < 0);
    return q;
}

// Registers are capped near 80 per thread whatever the resident blocks B (the
// bound is 6 blocks of 128 threads, or 3 of 256), leaving part of the
// register file free for the droplet kernels beside this one.
template <int NT, int S, int B, bool ODD, int MODE>
__global__ void __launch_bounds__(NT, (B > 768 / NT ? B : 768 / NT)) k_lattice_staged(LbView L, int pbuf)
{
    constexpr int RUN = stage_run<NT>();
    extern __shared__ __align__(128) float stage[];  // [S][19][RUN]
    __shared__ __align__(8) unsigned long long full[S];
    const int tid = threadIdx.x;
    const int nodes = L.nodes, nx = L.n[0], ny = L.n[1], nz = L.n[2], nxy = nx * ny;
    const int qs = (int)L.qs;
    const float *__restrict__ f = static_cast<const float *>(L.f);
    const int ntiles = (nodes + NT - 1) / NT;
    const float inv_nx = 1.0f / (float)nx, inv_nxy = 1.0f / (float)nxy;
    if ((blockIdx.x | tid) == 0) close_step(L);
    if (tid == 0) {
        for (int k = 0; k < S; ++k) mbar_init(&full[k], 1);
        fence_mbar_init();
    }
    __syncthreads();
    // d_i of every population, two bits each
    unsigned long long dpack = 0;
    if constexpr (ODD)
        sfor<19>([&](auto I) {
            constexpr int i = decltype(I)::value;
            dpack |= (unsigned long long)((-src_offset<ODD, i>(nx, nxy)) & 3) << (2 * i);
        });
    // warp 0: the 19 source runs of `tile` into stage `s`, lane i copying
    // run i.  Lane 0's single arrival, which also announces the bytes of all
    // 19 copies, comes after the copies are issued: until it arrives the
    // phase cannot complete, whatever the copies have delivered by then.
    const int lane = tid & 31;
    int off_l = 0, arr_l = 0;  // lane i < 19: source offset and array of population i
    sfor<19>([&](auto I) {
        constexpr int i = decltype(I)::value;
        if (lane == i) {
            off_l = src_offset<ODD, i>(nx, nxy);
            arr_l = ODD ? opp(i) : i;
        }
    });
    auto issue = [&](const int tile, const int s) {
        const int n0 = tile * NT, len = min(NT, nodes - n0);
        unsigned nb = 0;
        if (lane < 19) {
            const int u = (n0 - off_l) & ~3;  // widened start, may lie before the array
            const int a = max(u, 0), b = min((n0 - off_l + len + 3) & ~3, qs);
            if (b > a) {
                nb = 4u * (unsigned)(b - a);
                bulk_g2s(stage + (s * 19 + lane) * RUN + (a - u), f + (size_t)arr_l * qs + a, nb, &full[s]);
            }
        }
        const unsigned total = __reduce_add_sync(0xffffffffu, nb);
        // L.stage_fault (tests of the timeout path only): announce 16 bytes
        // more than the copies deliver, so that the phase never completes
        if (lane == 0) mbar_arrive_expect_tx(&full[s], total + (L.stage_fault ? 16u : 0u));
    };
    if (tid < 32)
        for (int k = 0; k < S; ++k) {
            const int t = blockIdx.x + k * gridDim.x;
            if (t < ntiles) issue(t, k);
        }
    int k = 0;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++k) {
        const int s = k % S;
        const bool arrived = mbar_wait(&full[s], (unsigned)(k / S) & 1u, kStageWaitNs);
        if (!__syncthreads_and(arrived)) {
            // a stage that never completes: report it, let the copies still
            // in flight land (bounded), and leave without touching memory
            if (tid == 0) {
                atomicOr(&L.ctl->err, IBL_ERRBIT_TIMEOUT);
                for (int j = 0; j < S; ++j) {
                    const int kk = k + j;
                    if (blockIdx.x + kk * (int)gridDim.x < ntiles)
                        mbar_wait(&full[kk % S], (unsigned)(kk / S) & 1u, kDrainWaitNs);
                }
            }
            return;
        }
        const int n = tile * NT + tid;
        bool bad = false;
        if (n < nodes) {
            const int z = div_by(n, nxy, inv_nxy), rem = n - z * nxy, y = div_by(rem, nx, inv_nx), x = rem - y * nx;
            if (MODE != LAT_FAR || !node_in_patch<false>(L, L.ctl, pbuf, x, y, z)) {
                const int sx = x == 0 ? -1 : (x == nx - 1 ? 1 : 0);
                const int sy = y == 0 ? -1 : (y == ny - 1 ? 1 : 0);
                const int sz = z == 0 ? -1 : (z == nz - 1 ? 1 : 0);
                const float *src = stage + s * 19 * RUN + tid;
                float g[19];
                sfor<19>([&](auto I) {
                    constexpr int i = decltype(I)::value;
                    if constexpr (ODD) g[i] = src[i * RUN + (int)((dpack >> (2 * i)) & 3u)];
                    else g[i] = src[i * RUN];
                });
                Hops h{};
                if constexpr (ODD) h = make_hops<(int)sizeof(float), false>(L, x, y, z);
                bad = lattice_finish<float, ODD, false, MODE, false, true>(L, g, x, y, z, n, pbuf, sx, sy, sz, h);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, bad);
        if (m != 0u && (tid & 31) == 0) flag_unstable(L);
        __syncthreads();  // every thread is done with stage s
        if (tid < 32) {
            const int t = tile + S * (int)gridDim.x;
            if (t < ntiles) issue(t, s);
        }
    }
}

// The patch nodes of the step: one warp per row (y, z) of the patch box,
// its lanes along x (32 at a time), so that each access of a warp is one
// contiguous run of a row.  Rows go round the blocks before a block gets its
// second one: a patch of fewer rows than the grid has warps (324 of 2432 for a
// 32^3 box) otherwise runs on the SMs of the first blocks alone, eight warps
// deep in each SM's FP64 pipe.
template <typename T, bool ODD, bool REC, bool PER, class P>
__device__ __forceinline__ void patch_rows(const LbView &L, const int buf, const int warp0, const int nwarps)
{
    const Ctl *c = L.ctl;
    const int ex = c->patch_ext[buf][0] + 1, ey = c->patch_ext[buf][1] + 1, ez = c->patch_ext[buf][2] + 1;
    const int lx = c->patch_lo[buf][0], ly = c->patch_lo[buf][1], lz = c->patch_lo[buf][2];
    const int rows = (ex > 0 && ey > 0 && ez > 0) ? ey * ez : 0;
    const int lane = threadIdx.x & 31;
    for (int row = warp0; row < rows; row += nwarps) {
        const int pz = row / ey, py = row - pz * ey;
        int y = ly + py, z = lz + pz;
        if (y >= L.n[1]) y -= L.n[1];  // a periodic patch may wrap once
        if (z >= L.n[2]) z -= L.n[2];
        for (int x0 = 0; x0 < ex; x0 += 32) {
            bool bad = false;
            if (x0 + lane < ex) {
                int x = lx + x0 + lane;
                if (x >= L.n[0]) x -= L.n[0];
                bad = lattice_node<T, ODD, REC, LAT_NEAR, PER, true, P>(L, x, y, z, x + L.n[0] * (y + L.n[1] * z), buf);
            }
            const unsigned m = __ballot_sync(0xffffffffu, bad);
            if (m != 0u && lane == 0) flag_unstable(L);
        }
    }
}

template <typename T, bool ODD, bool REC, bool PER>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_lattice_near(LbView L, int buf)
{
    const int wpb = blockDim.x >> 5;
    patch_rows<T, ODD, REC, PER, L2Keep>(L, buf, (threadIdx.x >> 5) * gridDim.x + blockIdx.x, gridDim.x * wpb);
}

// Ensemble: the nodes outside each member's droplet patch, one launch over
// the lattices of a group of members (the patches are updated concurrently
// by k_lattice_near_batched on the helper stream).  Block b works for member
// blk_member[b0 + b] (view G.v[member - m0], read from the kernel
// parameters) as its local block l = b0 + b - blk_start[member]: `tiles`
// tiles of NT consecutive nodes of the flattened box, from node l tiles NT
// on.  The first thread of a member's first block closes that member's step,
// as the single-droplet far kernel does.  With prefetch each thread fetches
// into L2 the node `ahead_nodes` further.
// Several tiles per block because a block starts with a chain of its own, the
// member from the table and then its view from the parameters (64 views do not
// stay in the constant cache), before its first population load: four tiles
// took the step of 32 droplets from 508 to 470 us (two 489, eight 474).  Where
// a member is re-centred (CEN, for the whole ensemble) the droplet chain is as
// long as the outside update, and its blocks wait for the outside update's to
// end: there one tile is faster (16 regularised, centred droplets 232 against
// 239 us with four).
template <typename T, bool ODD, int NT, bool PER, bool CEN>
__global__ void __launch_bounds__(NT, (sizeof(T) == 4 ? 1024 : 512) / NT)
    k_lattice_batched(const __grid_constant__ LbGroup G, const int m0, const int b0,
                      const int *__restrict__ blk_member, const int *__restrict__ blk_start, const int pbuf,
                      const int ahead_nodes)
{
    constexpr int tiles = CEN ? kEnsTilesCentred : kEnsTiles;
    const int mi = blk_member[b0 + blockIdx.x];
    const LbView &L = G.v[mi - m0];
    const int lb = b0 + (int)blockIdx.x - blk_start[mi];
    int node = lb * (tiles * NT) + (int)threadIdx.x;
    if (node == 0) close_step(L);
    bool bad = false;
#pragma unroll 1
    for (int k = 0; k < tiles; ++k, node += NT) {
        if (ahead_nodes > 0 && node + ahead_nodes < L.nodes) {
            T *f = static_cast<T *>(L.f);
            const unsigned off = (unsigned)(node + ahead_nodes) * (unsigned)sizeof(T);
#pragma unroll
            for (int i = 0; i < 19; ++i) asm volatile("prefetch.global.L2 [%0];" ::"l"(slot_at(f, i, L.qs, off)));
        }
        if (node < L.nodes) {
            const int z = fast_div(node, L.div_nxy), p = node - z * L.n[0] * L.n[1];
            const int y = fast_div(p, L.div_nx), x = p - y * L.n[0];
            bad |= lattice_node<T, ODD, false, LAT_FAR, PER, CEN>(L, x, y, z, node, pbuf);
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, bad);
    if (m != 0u && (threadIdx.x & 31) == 0) flag_unstable(L);
}

// Ensemble: the patch nodes of every member of a group (blockIdx.y is the
// member within the group), a warp per patch row as in k_lattice_near.  Capped
// at 64 registers: at 80 its two blocks per SM held 62% of the register file
// from the concurrent outside update for as long as they ran (step of 32
// droplets 478 -> 457 us, of 16 centred ones 234 -> 223; 32 periodic ones 375
// at 80, 358 at 64).  The odd form spills 16 bytes for it, 4 in periodic boxes.
template <typename T, bool ODD, bool PER, class P>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) k_lattice_near_batched(const __grid_constant__ LbGroup G,
                                                                                    const int buf)
{
    const int wpb = blockDim.x >> 5;
    patch_rows<T, ODD, false, PER, P>(G.v[blockIdx.y], buf, (threadIdx.x >> 5) * gridDim.x + blockIdx.x, gridDim.x * wpb);
}


template <typename T>
__global__ void __launch_bounds__(256) k_init(LbView L)
{
    const int node = blockIdx.x * blockDim.x + threadIdx.x;
    if (node >= L.nodes) return;
    const int nx = L.n[0], ny = L.n[1], nz = L.n[2];
    const int z = node / (nx * ny);
    const int rem = node - z * nx * ny;
    const int y = rem / nx;
    const int x = rem - y * nx;
    const double *A = L.frames;
    const double lx = x - 0.5 * (nx - 1), ly = y - 0.5 * (ny - 1), lz = z - 0.5 * (nz - 1);
    const double u[3] = {A[0] * lx + A[1] * ly + A[2] * lz, A[3] * lx + A[4] * ly + A[5] * lz,
                         A[6] * lx + A[7] * ly + A[8] * lz};
    const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    T *f = static_cast<T *>(L.f);
    sfor<19>([&](auto I) {
        constexpr int i = decltype(I)::value;
        const double cu = cxf(i) * u[0] + cyf(i) * u[1] + czf(i) * u[2];
        f[i * L.qs + node] = T(wgt(i) * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu));
    });
}

// ---------------------------------------------------------------------------
// Immersed boundary.
// One block beside the force/spread kernel of step t: reduce the bounding-box
// rows of r_t left by the previous interpolation (or regularisation) into the
// patch of step t + 1, grown by one node, in buffer `buf` (the parity of step
// t + 1).  Minima and maxima are integer ones on order-preserving keys: in
// FP64, by one warp before its share of the nodes, they were the longest chain
// of the kernel (a warp's FP64 instruction takes 64 cycles).
template <class P>
__device__ __forceinline__ void patch_from_rows(const LbView &L, const MeshView &M, const int buf)
{
    __shared__ unsigned long long box[4][6];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = L.ctl->n_part;
    const P K;
    unsigned long long v[6] = {0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
    for (int k = threadIdx.x; k < rows; k += kIbThreads)
        for (int a = 0; a < 6; ++a) {
            // minima as maxima of the negated value (sign bit)
            const double x = K.ld(M.part + 6 * k + a);
            const double y = a < 3 ? __longlong_as_double(__double_as_longlong(x) ^ 0x8000000000000000ull) : x;
            v[a] = max(v[a], order_key(y));
        }
    for (int a = 0; a < 6; ++a) {
        const unsigned long long m = warp_max(v[a]);
        if (lane == 0) box[warp][a] = m;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        unsigned long long lo = 0ull, hi = 0ull;
        for (int w = 0; w < kIbThreads / 32; ++w) {
            lo = max(lo, box[w][a]);
            hi = max(hi, box[w][3 + a]);
        }
        write_patch_axis(L, a, lo ? -key_value(lo) : 1e300, hi ? key_value(hi) : -1e300, buf, 1);
    }
    if (M.rec_ctl && threadIdx.x == 32) {
        // this step's patch buffer, for the adjoint
        const int pb = (buf + 2) % 3;
        for (int a = 0; a < 4; ++a) {
            M.rec_ctl->patch_lo[pb][a] = L.ctl->patch_lo[pb][a];
            M.rec_ctl->patch_ext[pb][a] = L.ctl->patch_ext[pb][a];
        }
    }
    __syncthreads();  // the block's next unit of work may reuse the rows
}

// Nodal force F_i = -sigma dA/dx_i (Eq. (pi_drop)) gathered over the
// triangles around node i, then spread with the 4-point delta
// (Eq. (ibm_force_d)(a)) by atomic adds into the Eulerian force.  LANES
// lanes per node: the lanes split the incident triangles (reduced with
// shuffles), then each lane adds 16 / LANES x-rows of four stencil points.
// STORED: m_t comes from M.tm (written by k_tri_moment_batched just before);
// otherwise each lane evaluates it for its triangle, from the edges out of its
// node (three times per triangle in all, but one kernel boundary fewer on the
// droplet chain of a single droplet, which is latency bound).
template <typename T, bool STORED, int LANES, class P = L2Keep>
__device__ __forceinline__ void spread_body(const LbView &L, const MeshView &M, const int blk)
{
    const int gid = blk * (kIbThreads / LANES) + threadIdx.x / LANES;
    const int lane = threadIdx.x % LANES;
    const bool valid = gid < M.nv;
    const int i = valid ? gid : M.nv - 1;
    const P K;
    const int k0 = K.ld(M.n2t_ptr + i), k1 = K.ld(M.n2t_ptr + i + 1);
    double ra;
    const NodeStencil<T> S = node_stencil<T, LANES, false>(L, M.r + 3 * i, lane, K, ra);
    double xi[3];
    if constexpr (!STORED)
        for (int a = 0; a < 3; ++a) xi[a] = K.ld(M.r + 3 * i + a);
    // force of the incidence k: triangle t with the node in position `slot`
    auto term = [&](const int k, double (&g)[3]) {
        const int e = K.ld(M.n2t + k);
        const int t = e / 3, slot = e - 3 * t;
        const int vp = K.ld(M.tris + (slot == 2 ? e - 2 : e + 1)), vq = K.ld(M.tris + (slot == 0 ? e + 2 : e - 1));
        double p[3], q[3];
        for (int a = 0; a < 3; ++a) p[a] = K.ld(M.r + 3 * vp + a);
        for (int a = 0; a < 3; ++a) q[a] = K.ld(M.r + 3 * vq + a);
        double m[3];
        if constexpr (STORED) {
            for (int a = 0; a < 3; ++a) m[a] = K.ld(M.tm + 3 * t + a);
        } else {
            const double e1[3] = {p[0] - xi[0], p[1] - xi[1], p[2] - xi[2]};
            const double e2[3] = {q[0] - xi[0], q[1] - xi[1], q[2] - xi[2]};
            double N[3];
            cross3(e1, e2, N);
            const double s = -0.5 * M.sigma * rsqrt(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
            for (int a = 0; a < 3; ++a) m[a] = s * N[a];
        }
        const double dd[3] = {q[0] - p[0], q[1] - p[1], q[2] - p[2]};
        cross3(m, dd, g);
    };
    double F[4] = {0.0, 0.0, 0.0, 0.0};
    int k = k0 + lane;
    if (k < k1) {
        double g[3];
        term(k, g);
        for (int a = 0; a < 3; ++a) F[a] = g[a];
    }
    while ((k += LANES) < k1) {  // valences above LANES
        double g[3];
        term(k, g);
        for (int a = 0; a < 3; ++a) F[a] += g[a];
    }
    const double Fa = group_sum4<LANES>(F);  // component lane / (LANES / 4)
    const int comp = lane / (LANES / 4);
    if (valid && lane % (LANES / 4) == 0 && comp < 3) M.fn[3 * i + comp] = Fa;
    if (M.rec_r && valid && lane < 3) M.rec_r[3 * i + lane] = ra;
    const int w0 = (threadIdx.x & 31) & ~(LANES - 1);
    const T Ft = T(Fa);
    const T Fx = __shfl_sync(0xffffffffu, Ft, w0), Fy = __shfl_sync(0xffffffffu, Ft, w0 + LANES / 4),
            Fz = __shfl_sync(0xffffffffu, Ft, w0 + LANES / 2);
    if (valid && !S.ok && lane == 0) atomicOr(&L.ctl->err, IBL_ERRBIT_WALL);
    if (!valid || !S.ok) return;
    const int nx = L.n[0], nxy = L.n[0] * L.n[1];
    T *force = static_cast<T *>(L.force);  // [nodes][4]
    T w[4];
    int x[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        w[a] = stencil_w(S.f[0], S.s[0], a);
        x[a] = stencil_at(S.base[0], a, nx);
    }
    // the lane's (y, z) rows r = lane, lane + LANES, ...: (b, c) = (r & 3, r >> 2)
    const int b = lane & 3;
    const T wy = stencil_w(S.f[1], S.s[1], b);
    const int y = stencil_at(S.base[1], b, L.n[1]) * nx;
#pragma unroll
    for (int j = 0; j < 16 / LANES; ++j) {
        const int c = (lane >> 2) + (LANES / 4) * j;
        const T wz = stencil_w(S.f[2], S.s[2], c);
        const int row = y + stencil_at(S.base[2], c, L.n[2]) * nxy;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const T dl = w[a] * wy * wz;
            K.red_add3(slot_at(force, 0, 0, (unsigned)(row + x[a]) * (unsigned)(4 * sizeof(T))), Fx * dl, Fy * dl, Fz * dl);
        }
    }
}

// Re-centring (Sec. 3.2: the linearisation is centred on the droplet's
// centre of mass).  `nblk` blocks per droplet sum six times the volume V and
// twenty-four times its first moment m over the signed tetrahedra (box centre,
// a, b, c) of the triangles.  Each block writes its sums to a row of M.obs_part
// (the shape record, its other user, runs on the same stream); the last block
// to finish adds the rows in a fixed order and stores the step's centre, box
// centre + m / V, in buffer `buf`.  Runs after the interpolation of the
// previous step and before any lattice update of this step.
constexpr int kCentreBlocksMax = 128;
static_assert(kCentreBlocksMax <= kObsBlocksMax, "rows of obs_part");

// A triangle's share: 6 V and 24 m about the box centre.
__device__ __forceinline__ void centre_term(const double (&p)[3][3], double (&v)[4])
{
    double bc[3];
    cross3(p[1], p[2], bc);
    const double vt = p[0][0] * bc[0] + p[0][1] * bc[1] + p[0][2] * bc[2];
    v[0] += vt;
    for (int a = 0; a < 3; ++a) v[1 + a] += vt * (p[0][a] + p[1][a] + p[2][a]);
}
__device__ __forceinline__ void centre_ref(const LbView &L, double (&ref)[3])
{
    for (int a = 0; a < 3; ++a) ref[a] = 0.5 * (L.n[a] - 1);
}
__device__ __forceinline__ void centre_finish(const LbView &L, const MeshView &M, const double (&v)[4], const int blk,
                                              const int nblk, const int buf)
{
    __shared__ double sh[kIbThreads / 32][4];
    __shared__ int last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double w[4] = {v[0], v[1], v[2], v[3]};
    const double s = group_sum4<32>(w);
    if ((lane & 7) == 0) sh[warp][lane >> 3] = s;
    __syncthreads();
    if (threadIdx.x < 4) {
        double t = sh[0][threadIdx.x];
        for (int k = 1; k < kIbThreads / 32; ++k) t += sh[k][threadIdx.x];
        M.obs_part[4 * blk + threadIdx.x] = t;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&L.ctl->cen_ticket, 1u) == (unsigned)(nblk - 1) ? 1 : 0;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // warp 0: lane sums component lane / 8 of every eighth row
    if (warp == 0) {
        double t = 0.0;
        for (int b = lane & 7; b < nblk; b += 8) t += __ldcg(M.obs_part + 4 * b + (lane >> 3));
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        const double V = __shfl_sync(0xffffffffu, t, 0);
        if ((lane & 7) == 0 && lane > 0) {
            const int a = (lane >> 3) - 1;
            L.ctl->centre[buf][a] = 0.5 * ((a == 0 ? L.n[0] : (a == 1 ? L.n[1] : L.n[2])) - 1) + t / (4.0 * V);
        }
        if (lane == 0) L.ctl->cen_ticket = 0u;
    }
}
__device__ __forceinline__ void centre_unit(const LbView &L, const MeshView &M, const int blk, const int nblk,
                                            const int buf)
{
    const L2Keep K;
    double ref[3], v[4] = {0.0, 0.0, 0.0, 0.0};
    centre_ref(L, ref);
    for (int t = blk * kIbThreads + (int)threadIdx.x; t < M.nt; t += nblk * kIbThreads) {
        double p[3][3];
        for (int c = 0; c < 3; ++c) {
            const int q = K.ld(M.tris + 3 * t + c);
            for (int a = 0; a < 3; ++a) p[c][a] = K.ld(M.r + 3 * q + a) - ref[a];
        }
        centre_term(p, v);
    }
    centre_finish(L, M, v, blk, nblk, buf);
}

// Ensemble: m_t of every triangle of every member at the current positions
// (Eq. (pi_drop)), once per step, for the batched force kernel that follows
// on the same stream, and with re-centring the centre of mass from the same
// positions; blockIdx.y is the member within the group.
template <class P>
__global__ void __launch_bounds__(128)
    k_tri_moment_batched(const __grid_constant__ LbGroup LG, const __grid_constant__ MeshGroup MG, const int buf)
{
    const LbView &L = LG.v[blockIdx.y];
    const MeshView &M = MG.v[blockIdx.y];
    const P K;
    const bool centre = L.recentre != 0;
    double ref[3], v[4] = {0.0, 0.0, 0.0, 0.0};
    if (centre) centre_ref(L, ref);
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < M.nt; t += gridDim.x * blockDim.x) {
        double x[3][3], m[3];
        tri_moment(M, t, m, x, K);
        for (int a = 0; a < 3; ++a) K.st(M.tm + 3 * t + a, m[a]);
        if (centre) {
            for (int c = 0; c < 3; ++c)
                for (int a = 0; a < 3; ++a) x[c][a] -= ref[a];
            centre_term(x, v);
        }
    }
    if (centre) centre_finish(L, M, v, blockIdx.x, gridDim.x, buf);
}

// Viscosity ratio (Sec. 2: droplet viscosity chi mu): the inside flags of the
// patch nodes of step `buf` by the even-odd rule on vertical rays.  One
// thread per triangle (a, b, c): for every lattice column (x, y) of the patch
// whose point q = (x + kRayDx, y + kRayDy) lies strictly inside the
// triangle's xy projection (three edge functions of one sign), the height
// z_c of the triangle over q comes from the barycentric weights, and the
// flags of the patch nodes with z < z_c flip.  A node is inside when an odd
// number of triangles lie above it.  The sub-lattice offsets keep the rays
// off mesh vertices and edges; every operation is a separately rounded IEEE
// one (no contraction), so the flags do not depend on the compiler.  The
// patch covers the droplet, so every inside node is a patch node; the patch
// update reads and clears the flags.
constexpr double kRayDx = 1.4142135623730951e-7, kRayDy = 1.7320508075688772e-7;

__device__ __forceinline__ double edge_fn(double ax, double ay, double bx, double by, double qx, double qy)
{
    return __dsub_rn(__dmul_rn(__dsub_rn(bx, ax), __dsub_rn(qy, ay)), __dmul_rn(__dsub_rn(by, ay), __dsub_rn(qx, ax)));
}

__device__ __forceinline__ void indicator_unit(const LbView &L, const MeshView &M, const int blk, const int buf)
{
    const int t = blk * kIbThreads + (int)threadIdx.x;
    if (t >= M.nt) return;
    const Ctl *c = L.ctl;
    if (c->patch_ext[buf][0] < 0 || c->patch_ext[buf][1] < 0 || c->patch_ext[buf][2] < 0) return;
    const int lo[3] = {c->patch_lo[buf][0], c->patch_lo[buf][1], c->patch_lo[buf][2]};
    const int hi[3] = {lo[0] + c->patch_ext[buf][0], lo[1] + c->patch_ext[buf][1], lo[2] + c->patch_ext[buf][2]};
    double p[3][3];
    for (int k = 0; k < 3; ++k) {
        const int v = M.tris[3 * t + k];
        for (int a = 0; a < 3; ++a) p[k][a] = M.r[3 * v + a];
    }
    const double xmin = fmin(p[0][0], fmin(p[1][0], p[2][0])), xmax = fmax(p[0][0], fmax(p[1][0], p[2][0]));
    const double ymin = fmin(p[0][1], fmin(p[1][1], p[2][1])), ymax = fmax(p[0][1], fmax(p[1][1], p[2][1]));
    int x0 = (int)ceil(__dsub_rn(xmin, kRayDx)), x1 = (int)floor(__dsub_rn(xmax, kRayDx));
    int y0 = (int)ceil(__dsub_rn(ymin, kRayDy)), y1 = (int)floor(__dsub_rn(ymax, kRayDy));
    x0 = max(x0, max(lo[0], 0));
    y0 = max(y0, max(lo[1], 0));
    x1 = min(x1, min(hi[0], L.n[0] - 1));
    y1 = min(y1, min(hi[1], L.n[1] - 1));
    const int z_lo = max(lo[2], 0), z_hi = min(hi[2], L.n[2] - 1);
    for (int y = y0; y <= y1; ++y)
        for (int x = x0; x <= x1; ++x) {
            const double qx = __dadd_rn((double)x, kRayDx), qy = __dadd_rn((double)y, kRayDy);
            const double e0 = edge_fn(p[0][0], p[0][1], p[1][0], p[1][1], qx, qy);
            const double e1 = edge_fn(p[1][0], p[1][1], p[2][0], p[2][1], qx, qy);
            const double e2 = edge_fn(p[2][0], p[2][1], p[0][0], p[0][1], qx, qy);
            const bool inside = (e0 > 0.0 && e1 > 0.0 && e2 > 0.0) || (e0 < 0.0 && e1 < 0.0 && e2 < 0.0);
            if (!inside) continue;
            const double num = __dadd_rn(__dadd_rn(__dmul_rn(e1, p[0][2]), __dmul_rn(e2, p[1][2])), __dmul_rn(e0, p[2][2]));
            const double zc = __ddiv_rn(num, __dadd_rn(__dadd_rn(e0, e1), e2));
            for (int z = z_lo; z <= z_hi && (double)z < zc; ++z) {
                const int node = x + L.n[0] * (y + L.n[1] * z);
                atomicXor(L.ind + (node >> 2), 1u << (8 * (node & 3)));
            }
        }
}

// Blocks of one launch: the patch of the next step (block 0), then, where the
// step needs them, nc blocks for its centre of mass and ni for its inside
// flags, then the node groups.  All of them only read the positions, so none
// waits for another: as launches of their own, centre and flags put 16 and 10
// us (cold) ahead of the forces on the droplet chain.
template <typename T, int LANES, bool EXTRA>
__global__ void __launch_bounds__(128) k_spread(LbView L, MeshView M, int next_buf, int nc, int ni)
{
    int b = (int)blockIdx.x;
    if (b == 0) {
        patch_from_rows<L2Keep>(L, M, next_buf);
        return;
    }
    b -= 1;
    if constexpr (EXTRA) {
        const int buf = next_buf == 0 ? 2 : next_buf - 1;  // this step's
        if (b < nc) {
            centre_unit(L, M, b, nc, buf);
            return;
        }
        b -= nc;
        if (b < ni) {
            indicator_unit(L, M, b, buf);
            return;
        }
        b -= ni;
    }
    spread_body<T, false, LANES>(L, M, b);
}

template <typename T, int LANES, class P = L2Keep>
__device__ __forceinline__ void interp_body(const LbView &L, const MeshView &M, const int blk, const int nblk)
{
    const int gid = blk * (kIbThreads / LANES) + threadIdx.x / LANES;
    const int lane = threadIdx.x % LANES;
    const bool valid = gid < M.nv;
    const int i = valid ? gid : M.nv - 1;
    const P K;
    double r;  // the lane's coordinate (lanes 0..2)
    const NodeStencil<T> S = node_stencil<T, LANES, false>(L, M.r + 3 * i, lane, K, r);
    T v[3] = {T(0), T(0), T(0)};
    if (S.ok) {
        const int nx = L.n[0], nxy = L.n[0] * L.n[1];
        T *vel = static_cast<T *>(L.vel);  // [nodes][4]
        T w[4];
        int x[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            w[a] = stencil_w(S.f[0], S.s[0], a);
            x[a] = stencil_at(S.base[0], a, nx);
        }
        // the lane's (y, z) rows r = lane, lane + LANES, ...: (b, c) = (r & 3, r >> 2)
        const int b = lane & 3;
        const T wy = stencil_w(S.f[1], S.s[1], b);
        const int y = stencil_at(S.base[1], b, L.n[1]) * nx;
#pragma unroll
        for (int k = 0; k < 16 / LANES; ++k) {
            const int c = (lane >> 2) + (LANES / 4) * k;
            const T wz = stencil_w(S.f[2], S.s[2], c);
            const int row = y + stencil_at(S.base[2], c, L.n[2]) * nxy;
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const T dl = w[a] * wy * wz;
                T ua, ub, uc;
                K.ld3(slot_at(vel, 0, 0, (unsigned)(row + x[a]) * (unsigned)(4 * sizeof(T))), ua, ub, uc);
                v[0] += ua * dl;
                v[1] += ub * dl;
                v[2] += uc * dl;
            }
        }
    }
    for (int o = LANES / 2; o > 0; o >>= 1)
        for (int a = 0; a < 3; ++a) v[a] += __shfl_xor_sync(0xffffffffu, v[a], o, LANES);
    // forward Euler, one component a lane; floor of the new coordinate for
    // the bounding box, whose patch only needs floors (conversion saturates:
    // a coordinate beyond 2^31 makes the patch the whole axis, as any beyond
    // 1e8 does; NaN is left out)
    constexpr int kHigh = 2147483647, kLow = -2147483647 - 1;
    int lo = kHigh, hi = kLow;
    if (valid && lane < 3) {
        if (S.ok) {
            r += (double)(lane == 0 ? v[0] : (lane == 1 ? v[1] : v[2]));
            K.st(M.r + 3 * i + lane, r);
        } else if (lane == 0) {
            atomicOr(&L.ctl->err, IBL_ERRBIT_WALL);
        }
        if (r == r) lo = hi = __double2int_rd(r);
    }
    // block min / max -> one partial row per block; the next force/spread
    // kernel reduces the rows into the patch (no tail here)
    __shared__ int box[kIbThreads / 32][6];
    const int wlane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int a = 0; a < 3; ++a) {
        const int mn = __reduce_min_sync(0xffffffffu, lane == a ? lo : kHigh);
        const int mx = __reduce_max_sync(0xffffffffu, lane == a ? hi : kLow);
        if (wlane == 0) {
            box[warp][a] = mn;
            box[warp][3 + a] = mx;
        }
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        const int a = threadIdx.x;
        int m = box[0][a];
        for (int w = 1; w < kIbThreads / 32; ++w) m = a < 3 ? min(m, box[w][a]) : max(m, box[w][a]);
        K.st(M.part + 6 * blk + a, (double)m);
    }
    if (blk == 0 && threadIdx.x == 0) L.ctl->n_part = nblk;
}

template <typename T, int LANES>
__global__ void __launch_bounds__(128) k_interp(LbView L, MeshView M, int nblk)
{
    // The grid is one block per node group, so that this turns once; written
    // straight, the same body compiled to a kernel that was slower in more
    // boxes than it was faster (us per step, loop and straight: 24^3 FP64 21.7
    // and 22.9, 96^3 regularised every tenth step 22.8 and 23.7, 128^3
    // regularised every step 66.8 and 68.8; 32^3 FP64 32.7 and 32.1, 64^3 12.5
    // and 12.3).
    for (int b = blockIdx.x; b < nblk; b += (int)gridDim.x) {
        interp_body<T, LANES>(L, M, b, nblk);
        __syncthreads();
    }
}

// Ensemble versions: block b works for member blk_member[b0 + b] as its
// local block b0 + b - blk_start[member]; node-group kernels use ceil(nv /
// kFwdNodesPerBlock) blocks per member.

// The node groups b0 .. b0 + nb - 1 of a group of members, block-strided so
// that a grid capped below nb leaves most SM slots to the concurrent
// lattice update.
template <typename T, class P>
__global__ void __launch_bounds__(128)
    k_spread_batched(const __grid_constant__ LbGroup LG, const __grid_constant__ MeshGroup MG, const int m0,
                     const int nm, const int b0, const int nb, const int *__restrict__ blk_member,
                     const int *__restrict__ blk_start, const int next_buf)
{
    // first the patches of the group's nm members, then the node groups
    for (int u = (int)blockIdx.x; u < nm + nb; u += (int)gridDim.x) {
        if (u < nm) {
            patch_from_rows<P>(LG.v[u], MG.v[u], next_buf);
            continue;
        }
        const int bb = b0 + u - nm;
        const int mi = blk_member[bb];
        spread_body<T, true, kFwdLanes, P>(LG.v[mi - m0], MG.v[mi - m0], bb - blk_start[mi]);
    }
}

template <typename T, class P>
__global__ void __launch_bounds__(128)
    k_interp_batched(const __grid_constant__ LbGroup LG, const __grid_constant__ MeshGroup MG, const int m0,
                     const int b0, const int nb, const int *__restrict__ blk_member,
                     const int *__restrict__ blk_start)
{
    for (int bb = b0 + (int)blockIdx.x; bb < b0 + nb; bb += (int)gridDim.x) {
        const int mi = blk_member[bb];
        interp_body<T, kFwdLanes, P>(LG.v[mi - m0], MG.v[mi - m0], bb - blk_start[mi],
                                     blk_start[mi + 1] - blk_start[mi]);
        __syncthreads();  // the next pass reuses the body's shared rows
    }
}

__global__ void __launch_bounds__(256) k_patch(LbView L, MeshView M, int buf)
{
    block_bbox_patch(L, M, M.r, M.nv, buf);
}

// Shape record (Sec. 2): enclosed volume, centroid and second moment by
// signed tetrahedra (ref, a, b, c), S = (5/V) M, eigen-decomposition, Taylor
// D and beta of Eq. (beta).  Block blk of nblk sums its share of the
// triangles; the last block to finish (a ticket in the control block) adds
// the partial sums in block order and writes the record.
__device__ __forceinline__ void observables_body(const LbView &L, const MeshView &M, const unsigned blk,
                                                 const unsigned nblk)
{
    __shared__ double sh11[8][11];
    __shared__ bool last;
    // volume integrals relative to node 0 (any point near the droplet will
    // do; this one needs no prior reduction)
    const double ref[3] = {M.r[0], M.r[1], M.r[2]};
    double acc[11];
    for (int k = 0; k < 11; ++k) acc[k] = 0.0;
    for (int t = blk * blockDim.x + threadIdx.x; t < M.nt; t += nblk * blockDim.x) {
        double p[3][3];
        for (int v = 0; v < 3; ++v) {
            const int id = M.tris[3 * t + v];
            for (int a = 0; a < 3; ++a) p[v][a] = M.r[3 * id + a] - ref[a];
        }
        double bc[3];
        cross3(p[1], p[2], bc);
        const double vt = (p[0][0] * bc[0] + p[0][1] * bc[1] + p[0][2] * bc[2]) / 6.0;
        const double s[3] = {p[0][0] + p[1][0] + p[2][0], p[0][1] + p[1][1] + p[2][1],
                             p[0][2] + p[1][2] + p[2][2]};
        acc[0] += vt;
        for (int a = 0; a < 3; ++a) acc[1 + a] += vt * s[a];
        // second moments xx, yy, zz, xy, xz, yz of a, b, c and s
        double m[6] = {0, 0, 0, 0, 0, 0};
        for (int v = 0; v < 4; ++v) {
            const double *q = v < 3 ? p[v] : s;
            m[0] += q[0] * q[0];
            m[1] += q[1] * q[1];
            m[2] += q[2] * q[2];
            m[3] += q[0] * q[1];
            m[4] += q[0] * q[2];
            m[5] += q[1] * q[2];
        }
        for (int k = 0; k < 6; ++k) acc[4 + k] += vt * m[k];
        double e1[3], e2[3], nn[3];
        for (int a = 0; a < 3; ++a) { e1[a] = p[1][a] - p[0][a]; e2[a] = p[2][a] - p[0][a]; }
        cross3(e1, e2, nn);
        acc[10] += 0.5 * sqrt(nn[0] * nn[0] + nn[1] * nn[1] + nn[2] * nn[2]);
    }
    // per-block partial sums; the last block adds them in block order
    block_sum<11>(acc, sh11);
    if (threadIdx.x == 0) {
        for (int k = 0; k < 11; ++k) M.obs_part[11 * blk + k] = acc[k];
        __threadfence();
        const unsigned t = atomicAdd(&L.ctl->obs_blocks_done, 1u);
        last = (t == nblk - 1);
    }
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    __threadfence();
    for (int k = 0; k < 11; ++k) acc[k] = 0.0;
    for (unsigned b = 0; b < nblk; ++b)
        for (int k = 0; k < 11; ++k) acc[k] += __ldcg(M.obs_part + 11 * b + k);
    L.ctl->obs_blocks_done = 0u;
    const double V = acc[0];
    double xc[3];
    for (int a = 0; a < 3; ++a) xc[a] = acc[1 + a] / 4.0 / V;
    double S6[6];
    for (int k = 0; k < 6; ++k) S6[k] = acc[4 + k] / 20.0;
    S6[0] -= V * xc[0] * xc[0];
    S6[1] -= V * xc[1] * xc[1];
    S6[2] -= V * xc[2] * xc[2];
    S6[3] -= V * xc[0] * xc[1];
    S6[4] -= V * xc[0] * xc[2];
    S6[5] -= V * xc[1] * xc[2];
    for (int k = 0; k < 6; ++k) S6[k] *= 5.0 / V;
    double a[3][3] = {{S6[0], S6[3], S6[4]}, {S6[3], S6[1], S6[5]}, {S6[4], S6[5], S6[2]}};
    double lam[3], vec[3][3];
    jacobi3(a, lam, vec);
    int order[3] = {0, 1, 2};
    for (int i = 0; i < 3; ++i)
        for (int j = i + 1; j < 3; ++j)
            if (lam[order[j]] < lam[order[i]]) {
                const int t = order[i];
                order[i] = order[j];
                order[j] = t;
            }
    ibl_observables o;
    const long long step = L.ctl->step;
    const long long used = step > 0 ? step - 1 : 0;
    long long kf = used / L.n_hold;
    if (kf > L.n_frames - 1) kf = L.n_frames - 1;
    const double *A = L.frames + 9 * kf;
    o.step = step;
    o.frame = (int)kf;
    o.reg_iters = L.ctl->reg_iters;
    o.err = L.ctl->err;
    o.pad_ = 0;
    o.volume = V;
    o.area = acc[10];
    for (int k = 0; k < 3; ++k) o.centroid[k] = xc[k] + ref[k];
    for (int k = 0; k < 6; ++k) o.S[k] = S6[k];
    for (int k = 0; k < 3; ++k) o.lam[k] = lam[order[k]];
    for (int k = 0; k < 3; ++k) o.vmax[k] = vec[k][order[2]];
    const double sl = sqrt(fmax(o.lam[2], 0.0)), ss = sqrt(fmax(o.lam[0], 0.0));
    o.D = (sl - ss) / (sl + ss);
    double E[3][3], nE = 0.0;
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            E[r][c] = 0.5 * (A[3 * r + c] + A[3 * c + r]);
            nE += E[r][c] * E[r][c];
        }
    nE = sqrt(nE);
    double vEv = 0.0;
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) vEv += o.vmax[r] * E[r][c] * o.vmax[c];
    o.beta = nE > 0.0 ? vEv / nE : __longlong_as_double(0x7ff8000000000000ll);
    const int slot = L.ctl->n_records % M.ring_cap;
    M.ring[slot] = o;
    L.ctl->n_records += 1;
}

__global__ void __launch_bounds__(256) k_observables(LbView L, MeshView M)
{
    observables_body(L, M, blockIdx.x, gridDim.x);
}

// Ensemble: the shape records of the members of a group whose bit is set in
// `due` (blockIdx.y is the member within the group), all in one launch.
__global__ void __launch_bounds__(256) k_observables_batched(const __grid_constant__ LbGroup LG,
                                                             const __grid_constant__ MeshGroup MG,
                                                             const unsigned long long due)
{
    if (!((due >> blockIdx.y) & 1ull)) return;
    observables_body(LG.v[blockIdx.y], MG.v[blockIdx.y], blockIdx.x, gridDim.x);
}

}  // namespace

// ---------------------------------------------------------------------------
// launchers
static inline unsigned blocks_for(long long n, int b) { return (unsigned)((n + b - 1) / b); }

// Multiprocessors of the current device (read once; launch shapes and
// prefetch distances are sized by it).
static int sm_count()
{
    static int sms = 0;
    if (sms == 0 && cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, 0) != cudaSuccess) sms = 1;
    return sms;
}

cudaError_t launch_init(const LbView &L, cudaStream_t s)
{
    const unsigned g = blocks_for(L.nodes, 256);
    if (L.precision == IBL_FP64) k_init<double><<<g, 256, 0, s>>>(L);
    else k_init<float><<<g, 256, 0, s>>>(L);
    return cudaGetLastError();
}

static bool any_periodic(const LbView &L)
{
    return L.bc[0] == IBL_BC_PERIODIC || L.bc[1] == IBL_BC_PERIODIC || L.bc[2] == IBL_BC_PERIODIC;
}

// Prefetch distance in nodes: one wave of resident blocks; none where the host
// left it out beside a large droplet patch (L.prefetch), nor for populations
// that stay in L2 between steps (up to 96 MB of its 129), where the 19
// prefetches only cost issue slots (97 x 75 x 61 channel 12.3 -> 11.7 us a
// step; 128^3, 159 MB, keeps them: 51.8 us with, 53.7 without).
template <typename T>
static int prefetch_distance(const LbView &L)
{
    if (!L.prefetch || 19 * L.qs * (long long)sizeof(T) <= (96ll << 20)) return 0;
    return sm_count() * (sizeof(T) == 4 ? 8 : 4) * 128;
}

// Tiles per block of the update outside a droplet patch.  Beside a droplet in
// a small FP32 box the chain of droplet kernels sets the step, and it waits
// for SM slots: a quarter of the blocks leaves every SM slots free (us per
// step with one and four tiles: 48^3 12.8 and 11.4, 56^3 14.9 and 11.9, 64^3
// 17.0 and 15.0, 72^3 17.9 and 15.9, 80^3 19.0 and 18.1, 88^3 20.0 and 21.0,
// 128^3 55.0 and 57.8).  Without a droplet one tile is faster at every size,
// and FP64 needs every SM's FP64 pipe.
constexpr int kFarTiles = 4, kFarTilesNodes = 80 * 80 * 80;

// Variants: a recording launch takes the general (periodic) form, and CEN
// (re-centring) exists only where a droplet does.
template <typename T, bool ODD>
static void lattice_launch_t(const LbView &L, bool rec, int mode, int pbuf, cudaStream_t s)
{
    const int ahead = prefetch_distance<T>(L);
    const bool per = any_periodic(L), cen = L.recentre != 0;
    const bool tiled = sizeof(T) == 4 && L.nodes <= kFarTilesNodes;
#define IBL_LAUNCH(R, M, P, C, K) \
    k_lattice<T, ODD, R, M, P, C, K><<<blocks_for(L.nodes, 128 * K), 128, 0, s>>>(L, pbuf, ahead)
#define IBL_LAUNCH_FAR(P, C)                                                    \
    do {                                                                        \
        if (rec) IBL_LAUNCH(true, LAT_FAR, true, C, 1);                         \
        else if (sizeof(T) == 4 && tiled) IBL_LAUNCH(false, LAT_FAR, P, C, (sizeof(T) == 4 ? kFarTiles : 1)); \
        else IBL_LAUNCH(false, LAT_FAR, P, C, 1);                               \
    } while (0)
    if (mode != LAT_FAR) {
        if (rec) IBL_LAUNCH(true, LAT_FULL, true, false, 1);
        else if (per) IBL_LAUNCH(false, LAT_FULL, true, false, 1);
        else IBL_LAUNCH(false, LAT_FULL, false, false, 1);
    } else if (cen) {
        if (per) IBL_LAUNCH_FAR(true, true);
        else IBL_LAUNCH_FAR(false, true);
    } else {
        if (per) IBL_LAUNCH_FAR(true, false);
        else IBL_LAUNCH_FAR(false, false);
    }
#undef IBL_LAUNCH_FAR
#undef IBL_LAUNCH
}

// Opts a kernel into its dynamic shared memory and the largest shared-memory
// carveout, once per kernel and device.
static cudaError_t prefer_shared(const void *kernel, size_t dyn)
{
    static std::mutex mu;
    static std::set<std::pair<const void *, int>> done;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(mu);
    if (done.count({kernel, dev})) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    if (e == cudaSuccess) done.insert({kernel, dev});
    return e;
}

// Launch shapes of the staged outside update: nodes per tile (= threads per
// block), pipeline stages, resident blocks per SM.
template <int V>
struct StagedShape;
template <>
struct StagedShape<1> {
    static constexpr int NT = 128, S = 2, B = 8;
};
template <>
struct StagedShape<2> {
    static constexpr int NT = 128, S = 3, B = 6;
};

template <int V, bool ODD>
static cudaError_t staged_launch(const LbView &L, int mode, int pbuf, cudaStream_t s)
{
    constexpr int NT = StagedShape<V>::NT, S = StagedShape<V>::S, B = StagedShape<V>::B;
    constexpr size_t smem = stage_bytes<NT, S>();
    void (*k)(LbView, int) = mode == LAT_FAR ? k_lattice_staged<NT, S, B, ODD, LAT_FAR>
                                             : k_lattice_staged<NT, S, B, ODD, LAT_FULL>;
    cudaError_t e = prefer_shared(reinterpret_cast<const void *>(k), smem);
    if (e != cudaSuccess) return e;
    const long long tiles = ((long long)L.nodes + NT - 1) / NT;
    const unsigned g = (unsigned)std::min<long long>(tiles, (long long)sm_count() * B);
    k<<<g, NT, smem, s>>>(L, pbuf);
    return cudaGetLastError();
}

template <bool ODD>
static cudaError_t staged_dispatch(const LbView &L, int mode, int pbuf, cudaStream_t s)
{
    switch (L.staged) {
    case 1: return staged_launch<1, ODD>(L, mode, pbuf, s);
    default: return staged_launch<2, ODD>(L, mode, pbuf, s);
    }
}

template <int V>
static cudaError_t staged_prepare_v()
{
    constexpr int NT = StagedShape<V>::NT, S = StagedShape<V>::S, B = StagedShape<V>::B;
    constexpr size_t smem = stage_bytes<NT, S>();
    cudaError_t e = cudaSuccess;
    for (void (*k)(LbView, int) : {k_lattice_staged<NT, S, B, false, LAT_FAR>, k_lattice_staged<NT, S, B, false, LAT_FULL>,
                                   k_lattice_staged<NT, S, B, true, LAT_FAR>, k_lattice_staged<NT, S, B, true, LAT_FULL>})
        if (e == cudaSuccess) e = prefer_shared(reinterpret_cast<const void *>(k), smem);
    return e;
}

cudaError_t staged_prepare(int kind)
{
    switch (kind) {
    case 1: return staged_prepare_v<1>();
    case 2: return staged_prepare_v<2>();
    default: return cudaSuccess;
    }
}

bool staged_ok(const LbView &L)
{
    return L.precision == IBL_FP32_DEV && !any_periodic(L) && (reinterpret_cast<uintptr_t>(L.f) & 15u) == 0 &&
           (L.qs & 3) == 0 && L.nodes < (1 << 26);
}

cudaError_t launch_lattice(const LbView &L, bool odd, bool record, int mode, int pbuf, cudaStream_t s)
{
    if (L.staged > 0 && !record && staged_ok(L))
        return odd ? staged_dispatch<true>(L, mode, pbuf, s) : staged_dispatch<false>(L, mode, pbuf, s);
    if (L.precision == IBL_FP64) {
        if (odd) lattice_launch_t<double, true>(L, record, mode, pbuf, s);
        else lattice_launch_t<double, false>(L, record, mode, pbuf, s);
    } else {
        if (odd) lattice_launch_t<float, true>(L, record, mode, pbuf, s);
        else lattice_launch_t<float, false>(L, record, mode, pbuf, s);
    }
    return cudaGetLastError();
}

template <typename T, bool PER>
static cudaError_t near_t(const LbView &L, bool odd, bool record, int pbuf, cudaStream_t s, int prio)
{
    const dim3 g(2 * sm_count()), b(256);  // grid-stride over the patch box
    if (odd) {
        if (record) return launch_p(k_lattice_near<T, true, true, PER>, g, b, s, prio, L, pbuf);
        return launch_p(k_lattice_near<T, true, false, PER>, g, b, s, prio, L, pbuf);
    }
    if (record) return launch_p(k_lattice_near<T, false, true, PER>, g, b, s, prio, L, pbuf);
    return launch_p(k_lattice_near<T, false, false, PER>, g, b, s, prio, L, pbuf);
}

cudaError_t launch_near(const LbView &L, bool odd, bool record, int pbuf, cudaStream_t s, int prio)
{
    const bool per = any_periodic(L);
    if (L.precision == IBL_FP64)
        return per ? near_t<double, true>(L, odd, record, pbuf, s, prio) : near_t<double, false>(L, odd, record, pbuf, s, prio);
    return per ? near_t<float, true>(L, odd, record, pbuf, s, prio) : near_t<float, false>(L, odd, record, pbuf, s, prio);
}

template <typename T>
__global__ void k_convert_frames(LbView L, int k0, int k1)
{
    const int i = 9 * k0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 9 * k1) static_cast<T *>(const_cast<void *>(L.frames_t))[i] = T(L.frames[i]);
}

cudaError_t launch_convert_frames(const LbView &L, int k0, int k1, cudaStream_t s)
{
    const unsigned g = blocks_for(9LL * (k1 - k0), 256);
    if (L.precision == IBL_FP64) k_convert_frames<double><<<g, 256, 0, s>>>(L, k0, k1);
    else k_convert_frames<float><<<g, 256, 0, s>>>(L, k0, k1);
    return cudaGetLastError();
}

// Lanes per mesh node of a single droplet's force/spread and interpolation
// kernels.  A small mesh (one 16-lane block per SM or fewer) takes 16 lanes:
// its step is the droplet chain's latency, and more, shorter threads shorten
// it.  A larger mesh takes kFwdLanes: there the lattice update sets the step,
// and half the threads hold half the SM slots the chain takes from it.
static int fwd_lanes(const MeshView &M)
{
    return (long long)M.nv * 16 <= (long long)sm_count() * kIbThreads ? 16 : kFwdLanes;
}

template <typename T, int LANES>
static cudaError_t spread_t(const LbView &L, const MeshView &M, int next_buf, cudaStream_t s, int prio)
{
    const int nblk = (int)blocks_for((long long)M.nv * LANES, kIbThreads), nt = (int)blocks_for(M.nt, kIbThreads);
    const int nc = L.recentre ? (nt < kCentreBlocksMax ? nt : kCentreBlocksMax) : 0, ni = L.visc ? nt : 0;
    const dim3 g(1 + nc + ni + nblk), b(kIbThreads);
    if (nc + ni > 0) return launch_p(k_spread<T, LANES, true>, g, b, s, prio, L, M, next_buf, nc, ni);
    return launch_p(k_spread<T, LANES, false>, g, b, s, prio, L, M, next_buf, 0, 0);
}

cudaError_t launch_spread(const LbView &L, const MeshView &M, int next_buf, cudaStream_t s, int prio)
{
    if (fwd_lanes(M) == 16)
        return L.precision == IBL_FP64 ? spread_t<double, 16>(L, M, next_buf, s, prio)
                                       : spread_t<float, 16>(L, M, next_buf, s, prio);
    return L.precision == IBL_FP64 ? spread_t<double, kFwdLanes>(L, M, next_buf, s, prio)
                                   : spread_t<float, kFwdLanes>(L, M, next_buf, s, prio);
}

cudaError_t launch_interp(const LbView &L, const MeshView &M, cudaStream_t s, int prio)
{
    const int lanes = fwd_lanes(M);
    const int nblk = (int)blocks_for((long long)M.nv * lanes, kIbThreads);
    const dim3 g(nblk), b(kIbThreads);
    if (lanes == 16) {
        if (L.precision == IBL_FP64) return launch_p(k_interp<double, 16>, g, b, s, prio, L, M, nblk);
        return launch_p(k_interp<float, 16>, g, b, s, prio, L, M, nblk);
    }
    if (L.precision == IBL_FP64) return launch_p(k_interp<double, kFwdLanes>, g, b, s, prio, L, M, nblk);
    return launch_p(k_interp<float, kFwdLanes>, g, b, s, prio, L, M, nblk);
}

cudaError_t launch_observables(const LbView &L, const MeshView &M, cudaStream_t s, int prio)
{
    int g = (M.nt + 255) / 256;
    if (g > kObsBlocksMax) g = kObsBlocksMax;
    return launch_p(k_observables, dim3(g), dim3(256), s, prio, L, M);
}

cudaError_t launch_patch_from_mesh(const LbView &L, const MeshView &M, int buf, cudaStream_t s)
{
    k_patch<<<1, 256, 0, s>>>(L, M, buf);
    return cudaGetLastError();
}

// Ensemble phases.  Each launches one kernel per group of up to kGroup
// members; the group's views travel in the kernel parameters.
namespace {
struct Groups {
    // parameter blocks are large: kept off the stack
    LbGroup lg;
    MeshGroup mg;
};
Groups &groups()
{
    static thread_local Groups g;
    return g;
}
void fill_group(const EnsembleView &E, int m0, int m1)
{
    Groups &G = groups();
    for (int k = m0; k < m1; ++k) {
        G.lg.v[k - m0] = E.lv[k];
        G.mg.v[k - m0] = E.mv[k];
    }
}
}  // namespace

static int ens_shape(const EnsembleView &E) { return E.shape >= 0 && E.shape < kEnsShapes ? E.shape : kEnsDefaultShape; }

// Blocks of a batched droplet-side kernel over nb node groups: all of them,
// or, in the capped shapes, at most the shape's cap per SM (the kernels then
// stride over the node groups).
static int chain_grid(const EnsembleView &E, int nb)
{
    if (!ens_shape_capped(ens_shape(E))) return nb;
    const int cap = ens_shape_cap(ens_shape(E)) * sm_count();
    return nb < cap ? nb : cap;
}

cudaError_t launch_ensemble_tri(const EnsembleView &E, long long step, cudaStream_t s, int prio)
{
    const int pbuf = (int)(step % 3), n = (int)E.lv.size();
    const bool keep = ens_shape_keep(ens_shape(E));
    Groups &G = groups();
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        fill_group(E, m0, m1);
        int nt_max = 0;
        for (int k = m0; k < m1; ++k) nt_max = E.mv[k].nt > nt_max ? E.mv[k].nt : nt_max;
        int tb = (nt_max + 127) / 128;
        if (ens_shape_capped(ens_shape(E))) {
            const int cap = ens_shape_cap(ens_shape(E)) * sm_count() / (m1 - m0);
            tb = tb < cap ? tb : (cap < 1 ? 1 : cap);
        }
        tb = tb < kCentreBlocksMax ? tb : kCentreBlocksMax;
        const dim3 g(tb, m1 - m0), b(kIbThreads);
        const cudaError_t e = keep ? launch_p(k_tri_moment_batched<L2Keep>, g, b, s, prio, G.lg, G.mg, pbuf)
                                   : launch_p(k_tri_moment_batched<L2Plain>, g, b, s, prio, G.lg, G.mg, pbuf);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T, class P>
static cudaError_t ensemble_spread_t(const EnsembleView &E, int m0, int m1, int nxt, cudaStream_t s, int prio)
{
    Groups &G = groups();
    const int nb0 = E.node_start[m0], nb = E.node_start[m1] - nb0;
    return launch_p(k_spread_batched<T, P>, dim3(chain_grid(E, nb + m1 - m0)), dim3(kIbThreads), s, prio, G.lg, G.mg, m0,
                    m1 - m0, nb0, nb, E.node_member, E.node_start_d, nxt);
}

cudaError_t launch_ensemble_spread(const EnsembleView &E, long long step, cudaStream_t s, int prio)
{
    const int nxt = (int)((step + 1) % 3), n = (int)E.lv.size();
    const bool keep = ens_shape_keep(ens_shape(E));
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        fill_group(E, m0, m1);
        cudaError_t e;
        if (E.precision == IBL_FP64)
            e = keep ? ensemble_spread_t<double, L2Keep>(E, m0, m1, nxt, s, prio)
                     : ensemble_spread_t<double, L2Plain>(E, m0, m1, nxt, s, prio);
        else
            e = keep ? ensemble_spread_t<float, L2Keep>(E, m0, m1, nxt, s, prio)
                     : ensemble_spread_t<float, L2Plain>(E, m0, m1, nxt, s, prio);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T, bool PER, class P>
static cudaError_t ensemble_near_t(const EnsembleView &E, bool odd, int m0, int m1, int pbuf, cudaStream_t s, int prio)
{
    Groups &G = groups();
    // blocks per member: kEnsNearBlocks, or in the capped shapes about the
    // shape's cap per SM over the whole group
    int per = kEnsNearBlocks;
    if (ens_shape_capped(ens_shape(E))) {
        per = ens_shape_cap(ens_shape(E)) * sm_count() / (m1 - m0);
        per = per < 1 ? 1 : (per > kEnsNearBlocks ? kEnsNearBlocks : per);
    }
    const dim3 g(per, m1 - m0), b(256);
    return odd ? launch_p(k_lattice_near_batched<T, true, PER, P>, g, b, s, prio, G.lg, pbuf)
               : launch_p(k_lattice_near_batched<T, false, PER, P>, g, b, s, prio, G.lg, pbuf);
}

template <class P>
static cudaError_t ensemble_near_p(const EnsembleView &E, bool odd, int m0, int m1, int pbuf, cudaStream_t s,
                                   int prio)
{
    bool per = false;
    for (int k = m0; k < m1; ++k) per = per || any_periodic(E.lv[k]);
    if (E.precision == IBL_FP64)
        return per ? ensemble_near_t<double, true, P>(E, odd, m0, m1, pbuf, s, prio)
                   : ensemble_near_t<double, false, P>(E, odd, m0, m1, pbuf, s, prio);
    return per ? ensemble_near_t<float, true, P>(E, odd, m0, m1, pbuf, s, prio)
               : ensemble_near_t<float, false, P>(E, odd, m0, m1, pbuf, s, prio);
}

cudaError_t launch_ensemble_near(const EnsembleView &E, long long step, cudaStream_t s, int prio)
{
    const bool odd = (step & 1) != 0;
    const int pbuf = (int)(step % 3);
    const int n = (int)E.lv.size();
    const bool keep = ens_shape_keep(ens_shape(E));
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        fill_group(E, m0, m1);
        const cudaError_t e = keep ? ensemble_near_p<L2Keep>(E, odd, m0, m1, pbuf, s, prio)
                                   : ensemble_near_p<L2Plain>(E, odd, m0, m1, pbuf, s, prio);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

template <typename T, bool ODD, bool PER, bool CEN>
static void far_batched_t(const EnsembleView &E, int m0, int pbuf, int waves, int ti, cudaStream_t s)
{
    const int m1 = m0 + kGroup < (int)E.lv.size() ? m0 + kGroup : (int)E.lv.size();
    const int lb0 = E.lat_start[ti][m0], lbn = E.lat_start[ti][m1] - lb0;
    const int nt = ti == 0 ? 128 : 256;
    const int per_sm = (sizeof(T) == 4 ? 1024 : 512) / nt;
    const int ahead = waves * sm_count() * per_sm * nt;
    Groups &G = groups();
    if (nt == 128)
        k_lattice_batched<T, ODD, 128, PER, CEN><<<lbn, 128, 0, s>>>(G.lg, m0, lb0, E.lat_member[ti], E.lat_start_d[ti], pbuf, ahead);
    else
        k_lattice_batched<T, ODD, 256, PER, CEN><<<lbn, 256, 0, s>>>(G.lg, m0, lb0, E.lat_member[ti], E.lat_start_d[ti], pbuf, ahead);
}

template <typename T>
static void far_batched_p(const EnsembleView &E, bool odd, bool per, bool cen, int m0, int pbuf, int waves, int ti,
                          cudaStream_t s)
{
#define IBL_LAUNCH(P, C)                                                   \
    do {                                                                   \
        if (odd) far_batched_t<T, true, P, C>(E, m0, pbuf, waves, ti, s);  \
        else far_batched_t<T, false, P, C>(E, m0, pbuf, waves, ti, s);     \
    } while (0)
    if (per && cen) IBL_LAUNCH(true, true);
    else if (per) IBL_LAUNCH(true, false);
    else if (cen) IBL_LAUNCH(false, true);
    else IBL_LAUNCH(false, false);
#undef IBL_LAUNCH
}

cudaError_t launch_ensemble_far(const EnsembleView &E, long long step, cudaStream_t s)
{
    const bool odd = (step & 1) != 0;
    const int pbuf = (int)(step % 3);
    const int n = (int)E.lv.size();
    const int shape = ens_shape(E);
    const int ti = ens_shape_threads(shape) == 128 ? 0 : 1, waves = ens_shape_waves(shape);
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        fill_group(E, m0, m1);
        bool per = false;
        for (int k = m0; k < m1; ++k) per = per || any_periodic(E.lv[k]);
        if (E.precision == IBL_FP64) far_batched_p<double>(E, odd, per, E.recentre, m0, pbuf, waves, ti, s);
        else far_batched_p<float>(E, odd, per, E.recentre, m0, pbuf, waves, ti, s);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_ensemble_interp(const EnsembleView &E, cudaStream_t s, int prio)
{
    const int n = (int)E.lv.size();
    const bool keep = ens_shape_keep(ens_shape(E));
    Groups &G = groups();
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        fill_group(E, m0, m1);
        const int nb0 = E.node_start[m0], nb = E.node_start[m1] - nb0;
        const dim3 g(chain_grid(E, nb)), b(kIbThreads);
        cudaError_t e;
        if (E.precision == IBL_FP64)
            e = keep ? launch_p(k_interp_batched<double, L2Keep>, g, b, s, prio, G.lg, G.mg, m0, nb0, nb,
                                E.node_member, E.node_start_d)
                     : launch_p(k_interp_batched<double, L2Plain>, g, b, s, prio, G.lg, G.mg, m0, nb0, nb,
                                E.node_member, E.node_start_d);
        else
            e = keep ? launch_p(k_interp_batched<float, L2Keep>, g, b, s, prio, G.lg, G.mg, m0, nb0, nb,
                                E.node_member, E.node_start_d)
                     : launch_p(k_interp_batched<float, L2Plain>, g, b, s, prio, G.lg, G.mg, m0, nb0, nb,
                                E.node_member, E.node_start_d);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_observables_batched(const EnsembleView &E, const std::vector<char> &due, cudaStream_t s, int prio)
{
    const int n = (int)E.lv.size();
    Groups &G = groups();
    for (int m0 = 0; m0 < n; m0 += kGroup) {
        const int m1 = m0 + kGroup < n ? m0 + kGroup : n;
        unsigned long long mask = 0;
        int nt_max = 0;
        for (int k = m0; k < m1; ++k)
            if (due[k]) {
                mask |= 1ull << (k - m0);
                nt_max = E.mv[k].nt > nt_max ? E.mv[k].nt : nt_max;
            }
        if (!mask) continue;
        fill_group(E, m0, m1);
        int g = (nt_max + 255) / 256;
        if (g > kObsBlocksMax) g = kObsBlocksMax;
        const cudaError_t e =
            launch_p(k_observables_batched, dim3(g, m1 - m0), dim3(256), s, prio, G.lg, G.mg, mask);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

void velocity_table(int c[19][3], double w[19])
{
    for (int i = 0; i < 19; ++i) {
        c[i][0] = cxf(i);
        c[i][1] = cyf(i);
        c[i][2] = czf(i);
        w[i] = wgt(i);
    }
}

}  // namespace iblb
