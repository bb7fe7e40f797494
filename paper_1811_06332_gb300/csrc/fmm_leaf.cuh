// What the leaf kernels of the uniform and the adaptive tree share: the columns
// (nx, ny) of a P2M warp, a leaf's local expansion as columns in shared memory,
// and its evaluation at a point.
#pragma once
#include "fmm_internal.h"

namespace fmm {

// Column c in order of nx + ny, the longest first (z powers 0 .. P - nx - ny): at
// p = 8 lanes 0..31 hold columns of 9 to 2 components and the 13 columns of the
// second turn have at most 2, so that turn takes 2 products per particle instead
// of the 9 of an order by nx, and the columns of a z power >= k are the first ones.
template <int P>
__device__ __forceinline__ void p2m_column(int c, int& nx, int& ny) {
    int s = 0;
    while (s < P && (s + 1) * (s + 2) / 2 <= c) ++s;   // (past the last column: anything)
    ny = c - s * (s + 1) / 2;
    nx = s - ny;
}
// the highest z power of turn k's columns
template <int P>
__device__ __forceinline__ constexpr int p2m_longest(int k) {
    int s = 0;
    while ((s + 1) * (s + 2) / 2 <= 32 * k) ++s;
    return P - s;
}

// length padded to a multiple of 16 bytes
template <typename T>
__host__ __device__ constexpr int pad16(int len) {
    return (len + (int)(16 / sizeof(T)) - 1) / (int)(16 / sizeof(T)) * (int)(16 / sizeof(T));
}
// offset of the column (kx, ky), s = kx + ky, in a symmetric tensor of rank <= P
// stored as columns in the order above, each from a 16-byte aligned offset;
// leaf_col(P + 1, 0) is the whole size
template <int P, typename T>
__host__ __device__ constexpr int leaf_col(int s, int ky) {
    int off = 0;
#pragma unroll
    for (int u = 0; u <= P; ++u)
        if (u < s) off += (u + 1) * pad16<T>(P + 1 - u);
    return off + ky * pad16<T>(P + 1 - s);
}
// loads N consecutive coefficients from a 16-byte aligned shared address
template <typename T, int N>
__device__ __forceinline__ void load16(const T* __restrict__ src, T (&dst)[N]) {
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int q = 0; q < (N + 3) / 4; ++q) {
            const float4 v = reinterpret_cast<const float4*>(src)[q];
            if (4 * q + 0 < N) dst[4 * q + 0] = v.x;
            if (4 * q + 1 < N) dst[4 * q + 1] = v.y;
            if (4 * q + 2 < N) dst[4 * q + 2] = v.z;
            if (4 * q + 3 < N) dst[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < (N + 1) / 2; ++q) {
            const double2 v = reinterpret_cast<const double2*>(src)[q];
            if (2 * q + 0 < N) dst[2 * q + 0] = v.x;
            if (2 * q + 1 < N) dst[2 * q + 1] = v.y;
        }
    }
}

// A leaf's local expansion as columns in shared memory, by LANES lanes of a warp
// (all 32 lanes call; valid: this part of the warp has a leaf).  ld(t) is
// component t of the stored form.  Traceless: the stored components of rank j are
// those with nz = 0, then those with nz = 1, from j^2 on by rising ny; the others
// follow from the trace, L[x, y, z+2] = -L[x+2, y, z] - L[x, y+2, z], one z at a
// time: 2 reads and an addition per component instead of a dot product of up to
// 2p + 1 with a row of the expansion matrix.  (Ls not __restrict__: the lanes read
// what other lanes wrote between the warp barriers.)
template <int P, int LANES, typename T, typename F>
__device__ __forceinline__ void local_columns(int basis, int lane, bool valid, T* Ls, F ld) {
    constexpr int NCOL = (P + 1) * (P + 2) / 2;
    constexpr int KC = (NCOL + LANES - 1) / LANES;
    int o0[KC], ox[KC], oy[KC];   // the columns (nx, ny), (nx + 2, ny), (nx, ny + 2)
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        const int col = lane + LANES * k;
        o0[k] = ox[k] = oy[k] = 0;
        if (col < NCOL) {
            int nx, ny;
            p2m_column<P>(col, nx, ny);
            const int s = nx + ny;
            o0[k] = leaf_col<P, T>(s, ny);
            if (s + 2 <= P) {
                ox[k] = leaf_col<P, T>(s + 2, ny);
                oy[k] = leaf_col<P, T>(s + 2, ny + 2);
            }
            if (valid) {
                if (basis) {
                    Ls[o0[k]] = ld(s * s + ny);
                    if (s < P) Ls[o0[k] + 1] = ld((s + 1) * (s + 1) + s + 2 + ny);
                } else {
                    T v[P + 1];   // all loads of the column in flight together
#pragma unroll
                    for (int z = 0; z <= P; ++z)
                        if (z <= P - s) v[z] = ld(pos_sym(nx, ny, z));
#pragma unroll
                    for (int z = 0; z <= P; ++z)
                        if (z <= P - s) Ls[o0[k] + z] = v[z];
                }
            }
        }
    }
    __syncwarp();
    if (!basis) return;
#pragma unroll
    for (int z = 2; z <= P; ++z) {
        const int nc = (P - z + 1) * (P - z + 2) / 2;   // columns with nx + ny <= P - z
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (LANES * k < nc && lane + LANES * k < nc && valid)
                Ls[o0[k] + z] = -(Ls[ox[k] + z - 2] + Ls[oy[k] + z - 2]);
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Phi = sum_k fx[kx] fy[ky] fz[kz] L[k] (f[j] = r^j / j!) and its gradient from
// the columns above, each read once by 16-byte loads.  With
//   Y = sum_z fz[z] L[kx,ky,z],  Yz = sum_z fz[z] L[kx,ky,z+1]  per column,
//   X = sum_y fy[y] Y,  Xy = sum_y fy[y-1] Y,  Xz = sum_y fy[y] Yz  per kx:
// Phi = sum fx[x] X, d/dx = sum fx[x-1] X, d/dy = sum fx[x] Xy, d/dz = sum fx[x] Xz.
// The x and y derivatives are the inner sums again under shifted powers, so a
// point takes 2 products per component (at p = 8, 460 with the outer sums)
// instead of the 4 of four separate sums (740) and a third of the shared reads.
// ---------------------------------------------------------------------------
template <int P, typename T, int KX, int KY, bool COLS>
__device__ __forceinline__ void l2p_row(const T* __restrict__ Ln, const T (&fy)[P + 1], const T (&fz)[P + 1],
                                        T& xp, T& xy, T& xz) {
    if constexpr (KY <= P - KX) {
        constexpr int LEN = P + 1 - KX - KY;
        T c[LEN];
        if constexpr (COLS) {
            load16<T, LEN>(Ln + leaf_col<P, T>(KX + KY, KY), c);
        } else {
#pragma unroll
            for (int z = 0; z < LEN; ++z) c[z] = Ln[pos_sym(KX, KY, z)];
        }
        T y = T(0), yz = T(0);
#pragma unroll
        for (int z = 0; z < LEN; ++z) {
            y = fma(fz[z], c[z], y);
            if (z + 1 < LEN) yz = fma(fz[z], c[z + 1], yz);
        }
        xp = fma(fy[KY], y, xp);
        if constexpr (KY > 0) xy = fma(fy[KY - 1], y, xy);
        if constexpr (LEN > 1) xz = fma(fy[KY], yz, xz);
        l2p_row<P, T, KX, KY + 1, COLS>(Ln, fy, fz, xp, xy, xz);
    }
}
// COLS: Ln as columns (local_columns); else in the order of symmetric storage
template <int P, typename T, int KX, bool COLS = true>
__device__ __forceinline__ void l2p_all(const T* __restrict__ Ln, const T (&fx)[P + 1], const T (&fy)[P + 1],
                                        const T (&fz)[P + 1], T& ph, T& gx, T& gy, T& gz) {
    if constexpr (KX <= P) {
        T xp = T(0), xy = T(0), xz = T(0);
        l2p_row<P, T, KX, 0, COLS>(Ln, fy, fz, xp, xy, xz);
        ph = fma(fx[KX], xp, ph);
        if constexpr (KX > 0) gx = fma(fx[KX - 1], xp, gx);
        gy = fma(fx[KX], xy, gy);
        gz = fma(fx[KX], xz, gz);
        l2p_all<P, T, KX + 1, COLS>(Ln, fx, fy, fz, ph, gx, gy, gz);
    }
}

}  // namespace fmm
