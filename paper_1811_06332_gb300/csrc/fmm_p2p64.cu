// FP64 near field (App. C direct sum over adjacent leaves, Eq. PhiAB), on the
// uniform octree and over the interaction lists of the adaptive trees.
//
// Bound: this part's FP64 pipe takes 17 cycles per warp instruction and SM,
// whatever the number of active lanes, so the time is the number of FP64
// warp instructions.  Hence:
//   - 18 FP64 instructions per pair: 3 differences, 3 for r^2, 5 for 1/r
//     (rsqrt_or0, below), 3 for the weights, 4 sums; the self test is an
//     integer test of r^2's exponent instead of an FP64 compare, and the
//     differences are taken of the stored coordinates (no leaf centre);
//   - lanes filled whatever the leaf size: NT targets per lane on groups of
//     ceil(tn / NT) lanes, as many groups as fit the warp splitting the
//     staged sources (0.75 to 1 of the lane slots in use, 0.9 on average for
//     leaves of 8 to 24; the power-of-two groups used before: 0.5 to 1);
//   - sources of up to 32 leaves staged as one sequence, so that every
//     chunk but the last holds 32 whatever the leaf sizes;
//   - lists cut into segments (adaptive) or shared by the warps of a block
//     (small uniform trees), so that no warp walks a list of thousands of
//     leaves alone while the others are done.  Partial sums are added in a
//     fixed order: results do not depend on scheduling.
// Measured (one-sided; kernel before -> here): uniform 524,288 particles at depth 5
// 11.3 -> 8.2 ms (2.2e8 pairs: 27 Gpairs/s of the 33 that 18 instructions at
// 17 cycles allow), 4,096 at depth 3 0.20 -> 0.08 ms, Plummer 100,003 with
// lists of up to thousands of leaves (AP variant) 133.6 -> 9.3 ms, binary tree
// of 150,000 29.7 -> 4.6 ms.
#include "fmm_adaptive.h"
#include "fmm_internal.h"

namespace fmm {

// 1/sqrt(v) for v > 0, and 0 for v = 0 (and NaN): the hardware's approximate
// reciprocal square root y (relative error below 2^-19) and one step of the
// binomial series of (1 - e)^(-1/2) about it, e = 1 - v y^2:
// y (1 + e/2 + 3 e^2 / 8), whose remainder 5 e^3 / 16 is below 2^-55.  The
// approximation flushes subnormal arguments, which are scaled first.
__device__ __forceinline__ double rsqrt_step(double v) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
    const double e = fma(-(v * y), y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double rsqrt_or0(double v) {
    double y = rsqrt_step(v);
    // zero, subnormal, infinite or NaN: an integer test of the high word
    if ((unsigned)(__double2hiint(v) - 0x00100000) >= 0x7fe00000u) {
        if (!(v > 0.0) || v > 1.7976931348623157e308) y = 0.0;
        else y = rsqrt_step(v * 0x1p+108) * 0x1p+54;
    }
    return y;
}

// targets per lane (1..3) for a block of tn = 1..32 targets: the value with
// the fewest steps NT / floor(32 / ceil(tn / NT)) per source
__device__ __forceinline__ int p2p64_nt(int tn) { return 1 + (int)((0xaa5a00a20820ull >> (2 * (tn - 1))) & 3ull); }

struct P2P64In {
    const double *x, *y, *z, *q;   // sorted particles
};
struct P2P64Out {
    double *pot, *ax, *ay, *az;    // caller order
};

// Sums of the block's targets [t0, t0 + tn) over one batch of up to 32 source
// leaves (lane l: leaf l's first particle sb, exclusive and inclusive prefix
// of the counts), chunks c0, c0 + cstep, ...
template <int NT>
__device__ __forceinline__ void p2p64_batch(int lane, int grp, int G, bool act, const double (&xt)[NT],
                                            const double (&yt)[NT], const double (&zt)[NT], double (&ph)[NT],
                                            double (&gx)[NT], double (&gy)[NT], double (&gz)[NT], int c0, int cstep,
                                            int total, int sb, int excl, int incl, const P2P64In& P,
                                            double2* __restrict__ sXY, double2* __restrict__ sZQ) {
    for (; c0 < total; c0 += cstep) {
        const int g = min(c0 + lane, total - 1);
        int i = 0;
#pragma unroll
        for (int step = 16; step >= 1; step >>= 1) {
            const int v = __shfl_sync(0xffffffffu, incl, i + step - 1);
            if (v <= g) i += step;
        }
        const int sj = __shfl_sync(0xffffffffu, sb, i) + (g - __shfl_sync(0xffffffffu, excl, i));
        const double2 xy = make_double2(P.x[sj], P.y[sj]), zq = make_double2(P.z[sj], P.q[sj]);
        __syncwarp();
        sXY[lane] = xy;
        sZQ[lane] = zq;
        __syncwarp();
        const int cnt = act ? min(32, total - c0) : 0;
        for (int k = grp; k < cnt; k += G) {
            const double2 a = sXY[k], b = sZQ[k];
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                const double dx = a.x - xt[j], dy = a.y - yt[j], dz = b.x - zt[j];
                const double ir = rsqrt_or0(fma(dx, dx, fma(dy, dy, dz * dz)));   // self, coincident: 0
                const double qir = b.y * ir, w = qir * ir * ir;   // ir * ir alone may overflow
                ph[j] += qir;
                gx[j] = fma(w, dx, gx[j]);
                gy[j] = fma(w, dy, gy[j]);
                gz[j] = fma(w, dz, gz[j]);
            }
        }
    }
}

// One block of up to 32 targets against the leaves given by meta(kb, sb, cnt)
// for lane l of batch kb (k0 <= kb + l < k1); the sums of target tl + gw j end
// in the lanes of group 0 and are handed to put(k, ph, gx, gy, gz).
template <int NT, typename Meta, typename Put>
__device__ __forceinline__ void p2p64_block(int lane, int t0, int tn, int k0, int k1, int part, int parts,
                                            const P2P64In& P, double2* sXY, double2* sZQ, Meta meta, Put put) {
    const int gw = (tn + NT - 1) / NT, G = 32 / gw, grp = lane / gw, tl = lane - grp * gw;
    const bool act = grp < G;
    double xt[NT], yt[NT], zt[NT], ph[NT], gx[NT], gy[NT], gz[NT];
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int k = t0 + min(tl + gw * j, tn - 1);
        xt[j] = P.x[k]; yt[j] = P.y[k]; zt[j] = P.z[k];
        ph[j] = gx[j] = gy[j] = gz[j] = 0.0;
    }
    for (int kb = k0; kb < k1; kb += 32) {
        int sb = 0, cnt = 0;
        if (kb + lane < k1) meta(kb + lane, sb, cnt);
        int incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        p2p64_batch<NT>(lane, grp, G, act, xt, yt, zt, ph, gx, gy, gz, 32 * part, 32 * parts, total, sb, incl - cnt,
                        incl, P, sXY, sZQ);
    }
    // the groups' sums, halving the groups (an order fixed by their number): a leaf
    // of one particle has 32 of them
    for (int h = G > 1 ? 1 << (31 - __clz(G - 1)) : 0; h; h >>= 1) {
        const int src = min(31, lane + h * gw);
        const bool take = grp + h < G && grp < h;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const double p0 = __shfl_sync(0xffffffffu, ph[j], src), x0 = __shfl_sync(0xffffffffu, gx[j], src),
                         y0 = __shfl_sync(0xffffffffu, gy[j], src), z0 = __shfl_sync(0xffffffffu, gz[j], src);
            if (take) { ph[j] += p0; gx[j] += x0; gy[j] += y0; gz[j] += z0; }
        }
    }
#pragma unroll
    for (int j = 0; j < NT; ++j) {
        const int k = tl + gw * j;
        if (grp == 0 && k < tn) put(k, ph[j], gx[j], gy[j], gz[j]);
    }
}

template <typename Meta, typename Put>
__device__ __forceinline__ void p2p64_any(int lane, int t0, int tn, int k0, int k1, int part, int parts,
                                          const P2P64In& P, double2* sXY, double2* sZQ, Meta meta, Put put) {
    const int nt = p2p64_nt(tn);
    if (nt == 1) p2p64_block<1>(lane, t0, tn, k0, k1, part, parts, P, sXY, sZQ, meta, put);
    else if (nt == 2) p2p64_block<2>(lane, t0, tn, k0, k1, part, parts, P, sXY, sZQ, meta, put);
    else p2p64_block<3>(lane, t0, tn, k0, k1, part, parts, P, sXY, sZQ, meta, put);
}

// ---------------------------------------------------------------------------
// uniform octree: WPL warps per leaf (1, or the 4 of a block, each taking
// every fourth chunk of the leaf's sources; their sums added in warp order)
// ---------------------------------------------------------------------------
template <int WPL>
__global__ void __launch_bounds__(128)
k_p2p64_uniform(int depth, int64_t nleaf, const int* __restrict__ start, P2P64In P, const int* __restrict__ perm,
                P2P64Out O) {
    __shared__ double2 sXY[4][32], sZQ[4][32];
    __shared__ double sR[WPL == 1 ? 1 : 4][4][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, part = w % WPL;
    const int64_t c = (int64_t)blockIdx.x * (4 / WPL) + w / WPL;
    if (c >= nleaf) return;   // WPL 4: the whole block
    const int b = start[c], e = start[c + 1];
    if (b == e) return;
    const int side = 1 << depth;
    int ix, iy, iz;
    cell_coords(depth, c, ix, iy, iz);
    auto meta = [&](int d, int& sb, int& cnt) {
        const int jx = ix - 1 + d % 3, jy = iy - 1 + (d / 3) % 3, jz = iz - 1 + d / 9;
        if (jx < 0 || jy < 0 || jz < 0 || jx >= side || jy >= side || jz >= side) return;
        const int64_t S = cell_index(depth, jx, jy, jz);
        sb = start[S];
        cnt = start[S + 1] - sb;
    };
    for (int t0 = b; t0 < e; t0 += 32) {
        const int tn = min(32, e - t0);
        p2p64_any(lane, t0, tn, 0, 27, part, WPL, P, sXY[w], sZQ[w], meta,
                  [&](int k, double ph, double gx, double gy, double gz) {
                      if (WPL == 1) {
                          const int o = perm[t0 + k];
                          O.pot[o] -= ph; O.ax[o] += gx; O.ay[o] += gy; O.az[o] += gz;
                      } else {
                          sR[w][0][k] = ph; sR[w][1][k] = gx; sR[w][2][k] = gy; sR[w][3][k] = gz;
                      }
                  });
        if constexpr (WPL > 1) {
            __syncthreads();
            // warp w adds component w of every target
            if (lane < tn) {
                const double v = sR[0][w][lane] + sR[1][w][lane] + sR[2][w][lane] + sR[3][w][lane];
                const int o = perm[t0 + lane];
                if (w == 0) O.pot[o] -= v;
                else if (w == 1) O.ax[o] += v;
                else if (w == 2) O.ay[o] += v;
                else O.az[o] += v;
            }
            __syncthreads();
        }
    }
}

// ---------------------------------------------------------------------------
// uniform octree, mutual form: every pair of particles of two adjacent leaves
// is evaluated once, 23 FP64 instructions for both directions instead of 2 x 18.
// A leaf's warp takes the sources of the leaf's 13 forward neighbours (the
// half of its 26 neighbours that follows it), 32 at a time, one per lane, and
// walks the targets: lane l meets target (l + r) mod tn in step r, so the lanes
// hold different targets; the source's sums stay in the lane's registers, the
// targets' in shared memory (a copy per group of tn lanes).  The sources' sums go
// to a slot of their own per direction, slots[13][4][n], which k_p2p64_back adds
// to the particles afterwards: no two warps write one word, and the sums run
// in a fixed order.  The leaf's own pairs take the one-sided form.  (1/r)^3 does
// not overflow: points of the unit cube in different leaves differ by at least
// 2^-63 along some axis, and points outside it by as much.
// Measured, 524,288 particles at depth 5: 8.2 -> 5.4 ms; 120,011 at depth 4: 3.2 ->
// 2.2 ms; but 4,096 at depth 3: 84 -> 99 us (see launch_p2p64).
// ---------------------------------------------------------------------------
constexpr int P2P64_DIRS = 13;

// neighbour d (0..26) of leaf (ix, iy, iz): false outside the grid
__device__ __forceinline__ bool p2p64_neighbour(int depth, int ix, int iy, int iz, int d, int64_t& S) {
    const int side = 1 << depth, jx = ix - 1 + d % 3, jy = iy - 1 + (d / 3) % 3, jz = iz - 1 + d / 9;
    if (jx < 0 || jy < 0 || jz < 0 || jx >= side || jy >= side || jz >= side) return false;
    S = cell_index(depth, jx, jy, jz);
    return true;
}

template <int WPL>
__global__ void __launch_bounds__(128)
k_p2p64_mutual(int depth, int64_t nleaf, const int* __restrict__ start, P2P64In P, const int* __restrict__ perm,
               P2P64Out O, double* __restrict__ slots, int64_t n) {
    __shared__ double2 sXY[4][32], sZQ[4][32];     // targets of the block
    __shared__ double2 sA[4][64], sB[4][64];       // their sums (potential, x | y, z); first the self sources
    __shared__ double sS[4][4][32];                // sums over the leaf's own particles
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, part = w % WPL;
    const int64_t c = (int64_t)blockIdx.x * (4 / WPL) + w / WPL;
    if (c >= nleaf) return;   // WPL 4: the whole block
    const int b = start[c], e = start[c + 1];
    if (b == e) return;
    int ix, iy, iz;
    cell_coords(depth, c, ix, iy, iz);
    // forward neighbours, one per lane
    int sb = 0, cnt = 0;
    if (lane < P2P64_DIRS) {
        int64_t S;
        if (p2p64_neighbour(depth, ix, iy, iz, 14 + lane, S)) { sb = start[S]; cnt = start[S + 1] - sb; }
    }
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31), excl = incl - cnt;
    for (int t0 = b; t0 < e; t0 += 32) {
        const int tn = min(32, e - t0);
        p2p64_any(
            lane, t0, tn, 0, 1, part, WPL, P, sA[w], sB[w],
            [&](int, int& s0, int& c0) { s0 = b; c0 = e - b; },
            [&](int k, double ph, double gx, double gy, double gz) {
                sS[w][0][k] = ph; sS[w][1][k] = gx; sS[w][2][k] = gy; sS[w][3][k] = gz;
            });
        __syncwarp();
        if (lane < tn) {
            sXY[w][lane] = make_double2(P.x[t0 + lane], P.y[t0 + lane]);
            sZQ[w][lane] = make_double2(P.z[t0 + lane], P.q[t0 + lane]);
        }
        sA[w][lane] = sA[w][lane + 32] = sB[w][lane] = sB[w][lane + 32] = make_double2(0.0, 0.0);
        __syncwarp();
        const int slot0 = (lane / tn) * tn;   // this lane group's copy of the targets' sums
        for (int c0 = 32 * part; c0 < total; c0 += 32 * WPL) {
            const int g = min(c0 + lane, total - 1);
            int i = 0;
#pragma unroll
            for (int step = 16; step >= 1; step >>= 1) {
                const int v = __shfl_sync(0xffffffffu, incl, i + step - 1);
                if (v <= g) i += step;
            }
            const int sj = __shfl_sync(0xffffffffu, sb, i) + (g - __shfl_sync(0xffffffffu, excl, i));
            const bool act = c0 + lane < total;
            const double x = P.x[sj], y = P.y[sj], z = P.z[sj], q = act ? P.q[sj] : 0.0;
            double ph = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
            int t = lane - slot0;
            for (int r = 0; r < tn; r += 2) {
                // two targets at a time (independent chains), their sums updated in turn:
                // in the next step another lane holds the same target
                double dx[2], dy[2], dz[2], ir[2], i3[2], qt[2];
                int tt[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    tt[u] = t;
                    t = t + 1 == tn ? 0 : t + 1;
                    const double2 a = sXY[w][tt[u]], d = sZQ[w][tt[u]];
                    dx[u] = x - a.x; dy[u] = y - a.y; dz[u] = z - d.x;
                    qt[u] = d.y;
                    ir[u] = rsqrt_or0(fma(dx[u], dx[u], fma(dy[u], dy[u], dz[u] * dz[u])));
                    i3[u] = ir[u] * (ir[u] * ir[u]);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (r + u < tn) {   // the same for the whole warp
                        const double ws = q * i3[u], wt = qt[u] * i3[u];
                        double2 A = sA[w][slot0 + tt[u]], B = sB[w][slot0 + tt[u]];
                        A.x = fma(q, ir[u], A.x);
                        A.y = fma(ws, dx[u], A.y);
                        B.x = fma(ws, dy[u], B.x);
                        B.y = fma(ws, dz[u], B.y);
                        sA[w][slot0 + tt[u]] = A;
                        sB[w][slot0 + tt[u]] = B;
                        ph = fma(qt[u], ir[u], ph);
                        gx = fma(-wt, dx[u], gx);
                        gy = fma(-wt, dy[u], gy);
                        gz = fma(-wt, dz[u], gz);
                        __syncwarp();
                    }
                }
            }
            if (act) {
                double* o = slots + (int64_t)i * 4 * n + sj;
                if (t0 != b) { ph += o[0]; gx += o[n]; gy += o[2 * n]; gz += o[3 * n]; }   // earlier targets of the leaf
                o[0] = ph; o[n] = gx; o[2 * n] = gy; o[3 * n] = gz;
            }
        }
        __syncwarp();
        double v[4] = {0.0, 0.0, 0.0, 0.0};
        if (lane < tn) {
            for (int k = lane; k < 64; k += tn) {   // the copies in order (those past the last group are zero)
                const double2 A = sA[w][k], B = sB[w][k];
                v[0] += A.x; v[1] += A.y; v[2] += B.x; v[3] += B.y;
            }
            for (int d = 0; d < 4; ++d) v[d] += sS[w][d][lane];
        }
        if constexpr (WPL == 1) {
            if (lane < tn) {
                const int o = perm[t0 + lane];
                O.pot[o] -= v[0]; O.ax[o] += v[1]; O.ay[o] += v[2]; O.az[o] += v[3];
            }
            __syncwarp();
        } else {
            __syncwarp();
            if (lane < tn)
                for (int d = 0; d < 4; ++d) sS[w][d][lane] = v[d];
            __syncthreads();
            if (lane < tn) {   // warp w adds component w of every target
                const double u = sS[0][w][lane] + sS[1][w][lane] + sS[2][w][lane] + sS[3][w][lane];
                const int o = perm[t0 + lane];
                if (w == 0) O.pot[o] -= u;
                else if (w == 1) O.ax[o] += u;
                else if (w == 2) O.ay[o] += u;
                else O.az[o] += u;
            }
            __syncthreads();
        }
    }
}

// the sums that the leaf's particles received as sources, over the 13 leaves before it
__global__ void __launch_bounds__(128)
k_p2p64_back(int depth, int64_t nleaf, const int* __restrict__ start, const int* __restrict__ perm, P2P64Out O,
             const double* __restrict__ slots, int64_t n) {
    const int lane = threadIdx.x & 31;
    const int64_t c = (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5);
    if (c >= nleaf) return;
    const int b = start[c], e = start[c + 1];
    if (b == e) return;
    int ix, iy, iz;
    cell_coords(depth, c, ix, iy, iz);
    // direction i of the leaf before: neighbour 14 + i of it is this leaf
    bool has = false;
    if (lane < P2P64_DIRS) {
        int64_t S;
        has = p2p64_neighbour(depth, ix, iy, iz, 12 - lane, S) && start[S + 1] > start[S];
    }
    const unsigned m = __ballot_sync(0xffffffffu, has);
    for (int a = b + lane; a < e; a += 32) {
        double ph = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
#pragma unroll
        for (int i = 0; i < P2P64_DIRS; ++i)
            if (m >> i & 1) {
                const double* s = slots + (int64_t)i * 4 * n + a;
                ph += s[0]; gx += s[n]; gy += s[2 * n]; gz += s[3 * n];
            }
        const int o = perm[a];
        O.pot[o] -= ph; O.ax[o] += gx; O.ay[o] += gy; O.az[o] += gz;
    }
}

// Bytes of slots for the mutual form where it is the faster one, else 0: from 4
// million pairs, about 27 n^2 / nleaf, on; below, the time is the latency of a leaf's
// chain and a second launch (one-sided against mutual: 0.9 million pairs 84 and 99
// us; 95 million 3.2 and 2.2 ms).  Up to 2^24 particles (7 GB of slots).
int64_t p2p64_slot_bytes(int64_t n, int64_t nleaf) {
    const bool mutual = n <= ((int64_t)1 << 24) && 27.0 * (double)n * (double)n / (double)nleaf >= 4e6;
    return mutual ? P2P64_DIRS * 4 * 8 * n : 0;
}

// The mutual form where slots (p2p64_slot_bytes) are given, else the one-sided.
int launch_p2p64(int depth, int64_t nleaf, const int* start, const double* xs, const double* ys, const double* zs,
                 const double* qs, const int* perm, double* pot, double* ax, double* ay, double* az, double* slots,
                 int64_t n, cudaStream_t s) {
    if (nleaf <= 0 || n <= 0) return 0;
    const P2P64In P{xs, ys, zs, qs};
    const P2P64Out O{pot, ax, ay, az};
    // four warps per leaf up to 8^4 leaves: with one warp each, 4096 leaves
    // are 27 warps per SM, and the last, fullest leaf sets the time
    const bool four = nleaf <= 4096;
    const unsigned g = (unsigned)(four ? nleaf : (nleaf + 3) / 4);
    if (slots) {
        if (four) k_p2p64_mutual<4><<<g, 128, 0, s>>>(depth, nleaf, start, P, perm, O, slots, n);
        else k_p2p64_mutual<1><<<g, 128, 0, s>>>(depth, nleaf, start, P, perm, O, slots, n);
        k_p2p64_back<<<(unsigned)((nleaf + 3) / 4), 128, 0, s>>>(depth, nleaf, start, perm, O, slots, n);
        count_launch();
    } else {
        if (four) k_p2p64_uniform<4><<<g, 128, 0, s>>>(depth, nleaf, start, P, perm, O);
        else k_p2p64_uniform<1><<<g, 128, 0, s>>>(depth, nleaf, start, P, perm, O);
    }
    count_launch();
    return 0;
}

// ---------------------------------------------------------------------------
// adaptive trees: work items (target block of a leaf, segment of its list)
// ---------------------------------------------------------------------------
// items and partial-sum slots of each leaf of the work list: ceil(n / 32)
// target blocks times ceil(len / seg) segments; slots only where a list has
// several segments (the others write their result directly)
__global__ void k_p2p64_items(int nn, const int* __restrict__ leaf, const int* __restrict__ nchild,
                              const int* __restrict__ nb, const int* __restrict__ ne, const int* __restrict__ off,
                              int seg, int* __restrict__ items, int* __restrict__ slots) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const int c = leaf[i];
    if (nchild[c]) { items[i] = slots[i] = 0; return; }   // the work list's tail: cells
    const int nblk = (ne[c] - nb[c] + 31) / 32, nseg = (off[c + 1] - off[c] + seg - 1) / seg;
    items[i] = nblk * nseg;
    slots[i] = nseg > 1 ? nblk * nseg : 0;
}

__global__ void __launch_bounds__(128)
k_p2p64_list(int nleaf, const int* __restrict__ leaf, const int* __restrict__ ioff, const int* __restrict__ soff,
             const int* __restrict__ off, const int* __restrict__ src, int seg, const int* __restrict__ nb,
             const int* __restrict__ ne, P2P64In P, const int* __restrict__ perm, P2P64Out O,
             double* __restrict__ part, int* __restrict__ counter) {
    __shared__ double2 sXY[4][32], sZQ[4][32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nitem = ioff[nleaf];
    for (;;) {
        int item = 0;
        if (lane == 0) item = atomicAdd(counter, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= nitem) break;
        // the last leaf i with ioff[i] <= item (every leaf has an item), 32 probes at a time
        int i = 0, len = nleaf;
        while (len > 1) {
            const int step = (len + 31) / 32, at = lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, at < len && ioff[i + at] <= item);
            const int hit = __popc(m) - 1;
            i += hit * step;
            len = min(step, len - hit * step);
        }
        const int c = leaf[i], b = nb[c], e = ne[c], k0 = off[c], k1 = off[c + 1];
        const int nblk = (e - b + 31) / 32, nseg = (k1 - k0 + seg - 1) / seg, local = item - ioff[i];
        const int t0 = b + 32 * (local % nblk), sg = local / nblk, slot = soff[i] + local;
        const int ka = k0 + sg * seg, ke = min(k1, ka + seg);
        p2p64_any(
            lane, t0, min(32, e - t0), ka, ke, 0, 1, P, sXY[w], sZQ[w],
            [&](int k, int& sb, int& cnt) {
                const int S = src[k];
                sb = nb[S];
                cnt = ne[S] - sb;
            },
            [&](int k, double ph, double gx, double gy, double gz) {
                if (nseg == 1) {
                    const int o = perm[t0 + k];
                    O.pot[o] -= ph; O.ax[o] += gx; O.ay[o] += gy; O.az[o] += gz;
                } else {
                    double* p = part + (int64_t)slot * 128 + k;
                    p[0] = ph; p[32] = gx; p[64] = gy; p[96] = gz;
                }
            });
    }
}

// the segments' sums of each target, in list order (one warp per leaf)
__global__ void __launch_bounds__(128)
k_p2p64_sum(int nleaf, const int* __restrict__ leaf, const int* __restrict__ soff, const int* __restrict__ nb,
            const int* __restrict__ ne, const int* __restrict__ perm, P2P64Out O, const double* __restrict__ part) {
    const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (i >= nleaf) return;
    const int s0 = soff[i], ns = soff[i + 1] - s0;
    if (ns == 0) return;
    const int c = leaf[i], b = nb[c], e = ne[c], nblk = (e - b + 31) / 32;
    for (int blk = 0; blk < nblk; ++blk) {
        const int t = b + 32 * blk + lane;
        if (t >= e) continue;
        double ph = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
        for (int s = blk; s < ns; s += nblk) {
            const double* p = part + (int64_t)(s0 + s) * 128 + lane;
            ph += p[0]; gx += p[32]; gy += p[64]; gz += p[96];
        }
        const int o = perm[t];
        O.pot[o] -= ph; O.ax[o] += gx; O.ay[o] += gy; O.az[o] += gz;
    }
}

int ad_p2p64_items(int nn, const int* leaf, const int* nchild, const int* nb, const int* ne, const int* off, int seg,
                   int* items, int* slots, cudaStream_t s) {
    if (nn <= 0) return 0;
    k_p2p64_items<<<(unsigned)((nn + 255) / 256), 256, 0, s>>>(nn, leaf, nchild, nb, ne, off, seg, items, slots);
    count_launch();
    return 0;
}

int ad_p2p64(int nleaf, const int* leaf, const int* ioff, const int* soff, const int* off, const int* src, int seg,
             const int* nb, const int* ne, const double* xs, const double* ys, const double* zs, const double* qs,
             const int* perm, double* pot, double* ax, double* ay, double* az, double* part, bool split, int* counter,
             int blocks, cudaStream_t s) {
    if (nleaf <= 0) return 0;
    const P2P64In P{xs, ys, zs, qs};
    const P2P64Out O{pot, ax, ay, az};
    k_p2p64_list<<<(unsigned)blocks, 128, 0, s>>>(nleaf, leaf, ioff, soff, off, src, seg, nb, ne, P, perm, O, part,
                                                  counter);
    count_launch();
    if (split) {
        k_p2p64_sum<<<(unsigned)((nleaf + 3) / 4), 128, 0, s>>>(nleaf, leaf, soff, nb, ne, perm, O, part);
        count_launch();
    }
    return 0;
}

}  // namespace fmm
