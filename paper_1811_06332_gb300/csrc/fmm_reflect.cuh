// M2L over the uniform interaction lists by reflections: what the generated
// kernels (_gen/rf_P<p>_<type>.cu) share.
//
// D_k(s r) = s^k D_k(r) for a vector s of signs, so the sources at the
// offsets (+-a, +-b, +-c) of a target share one D-tensor once their multipoles are
// combined by the parities of the three axes:
//   L_n += sum_m D_{n+m}(a, b, c) T_m^par(n+m),  T_m^pi = sum_s s^pi c_m^(s),
// c the folded multipoles (components with nz <= 1, weights 1/m! included) and
// s over the signs that the target's list has: both for magnitudes 1 and 2, one
// for 3 (the far side of the parent's neighbour) and one, trivially, for 0.  The
// 189 offsets of a target become 56 magnitude triples; the combination is a
// butterfly per axis with both signs (24 sums for 8 sources).  At p = 8 a target
// takes 56 x 1365 products and 30618 sums instead of 189 x 1365 products,
// and components of D that vanish (odd in an axis of magnitude 0) are left out:
// 54 000 products.
#pragma once
#include "fmm_device.cuh"
#include "fmm_internal.h"

namespace fmm {

constexpr int RF_NORB = 56;
constexpr int RF_PAD = 32;   // zero cells after each component's row: the source of a missing neighbour

// one warp's share of the lists: 32 cells of one class, the orbits grp, grp + g, ...
struct RfUnit {
    int l, g, grp, cls;
    int64_t ncell, F, L, part;   // cells; element offsets of the level in F, Lt and part
    int64_t t, tg;               // position in the class (may pass its end), cell
    bool act;
};
__device__ __forceinline__ bool rf_unit(const RfLevels& lv, int unit, int lane, RfUnit& u) {
    int i = 0;
    while (i < lv.n && unit >= lv.v[i].end) ++i;
    if (i >= lv.n) return false;
    const RfLevel& v = lv.v[i];
    const int local = unit - (i ? lv.v[i - 1].end : 0);
    u.l = v.l;
    u.g = v.g;
    u.ncell = (int64_t)1 << (3 * v.l);
    u.F = v.F; u.L = v.L; u.part = v.part;
    // consecutive units: other cells, the same orbits (warps that run side by
    // side run the same code)
    const int64_t h3 = u.ncell >> 3, wpc = (h3 + 31) / 32, cb = local % (8 * wpc);
    u.grp = (int)(local / (8 * wpc));
    u.cls = (int)(cb / wpc);
    u.t = (cb % wpc) * 32 + lane;
    u.act = u.t < h3;
    u.tg = u.cls * h3 + u.t;
    return true;
}

// Cells of the sources of one orbit: i[s], s bit d set: the negative side of
// axis d (axes with both signs only); the pad where there is no such cell.
__device__ __forceinline__ void rf_sources(const RfUnit& u, int a, int b, int c, int (&i)[8]) {
    const int hs = 1 << (u.l - 1), side = 1 << u.l, h3 = hs * hs * hs;
    const int cl[3] = {u.cls & 1, (u.cls >> 1) & 1, u.cls >> 2};
    const int t = (int)u.t;
    const int x[3] = {2 * (t % hs) + cl[0], 2 * ((t / hs) % hs) + cl[1], 2 * (t / (hs * hs)) + cl[2]};
    const int mag[3] = {a, b, c}, st[3] = {1, hs, hs * hs};
    int f[3][2];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // r = target - source; magnitude 3 lies on the side away from the parent's centre
        const int r0 = mag[d] == 3 && cl[d] == 0 ? -3 : mag[d];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            const int j = x[d] - (s ? -mag[d] : r0);
            f[d][s] = j >= 0 && j < side ? ((j & 1) << d) * h3 + (j >> 1) * st[d] : -(1 << 30);
        }
    }
#pragma unroll
    for (int s = 0; s < 8; ++s) {
        const int64_t k = (int64_t)f[0][s & 1] + f[1][(s >> 1) & 1] + f[2][s >> 2];
        i[s] = u.act && k >= 0 ? (int)k : (int)u.ncell;
    }
}

// this lane's share of the orbit's D components (those with nz <= 1 + 1 of
// ranks <= p) into the warp's sD, signs of the one-sided axes included
template <typename T>
__device__ __forceinline__ void rf_stage(int nd, int ns, const double* __restrict__ Dtab, const RfUnit& u, int a, int b,
                                         int c, int lane, T* sD) {
    // odd powers change sign on an axis of magnitude 3 seen from the even side
    const int neg = (a == 3 && !(u.cls & 1) ? 1 : 0) | (b == 3 && !(u.cls & 2) ? 2 : 0) |
                    (c == 3 && !(u.cls & 4) ? 4 : 0);
    const double* D = Dtab + (int64_t)((3 + c) * 49 + (3 + b) * 7 + 3 + a) * ns;
    __syncwarp();
    for (int k = lane; k < nd; k += 32) {
        const double v = D[d_rf_pos[k]];
        sD[k] = T(__popc(neg & d_rf_par[k]) & 1 ? -v : v);
    }
    __syncwarp();
}

__device__ __forceinline__ void rf_orbit(int u, int& a, int& b, int& c) {
    const int o = d_rf_orb[u];
    a = o & 3; b = (o >> 2) & 3; c = o >> 4;
}

// Entry K of the warp's D components at shared address sa.  volatile: the
// compiler knows nothing of the memory that is read, and a plain asm could be
// moved past the barriers and stores of the next orbit's rf_stage.
template <typename T, int K>
__device__ __forceinline__ T rf_lds(unsigned sa) {
    T v;
    if constexpr (sizeof(T) == 4) asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(sa), "n"(4 * K));
    else asm volatile("ld.shared.f64 %0, [%1+%2];" : "=d"(v) : "r"(sa), "n"(8 * K));
    return v;
}

template <typename T>
__device__ __forceinline__ void rf_bf(T& a, T& b) {   // both signs: (sum, difference)
    const T s = a + b;
    b = a - b;
    a = s;
}

}  // namespace fmm
