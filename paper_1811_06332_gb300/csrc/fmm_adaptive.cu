// Adaptive-octree FMM (App. C with an octree): tree construction from Morton
// keys, enclosing radii, directed dual-tree traversal with the multipole
// acceptance criterion theta |z_A - z_B| > r_A + r_B, interaction lists in
// CSR form, and the folded multipoles of the list M2L.  Expansions are kept
// node-major ([node][ncoef]) in public storage (full symmetric, or independent
// traceless components).
//
// Geometry (bounding cube, centres, radii, MAC) is evaluated with explicitly
// rounded FP64 operations (no fused multiply-add) in the same order as the
// plain C formulation, so the tree and the lists do not depend on the
// compiler's contraction choices.
#include "fmm_internal.h"
#include "_gen/fmm_fold.cuh"

namespace fmm {

// ---------------------------------------------------------------------------
// bounding cube: lo[3], side, scale = 2^21 / side
// ---------------------------------------------------------------------------
__global__ void k_bbox_partial(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                               const double* __restrict__ z, double* __restrict__ part) {
    __shared__ double s[6][256];
    double lo[3] = {1e308, 1e308, 1e308}, hi[3] = {-1e308, -1e308, -1e308};
    for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
        const double v[3] = {x[i], y[i], z[i]};
        for (int d = 0; d < 3; ++d) { lo[d] = fmin(lo[d], v[d]); hi[d] = fmax(hi[d], v[d]); }
    }
    for (int d = 0; d < 3; ++d) { s[d][threadIdx.x] = lo[d]; s[3 + d][threadIdx.x] = hi[d]; }
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o)
            for (int d = 0; d < 3; ++d) {
                s[d][threadIdx.x] = fmin(s[d][threadIdx.x], s[d][threadIdx.x + o]);
                s[3 + d][threadIdx.x] = fmax(s[3 + d][threadIdx.x], s[3 + d][threadIdx.x + o]);
            }
        __syncthreads();
    }
    if (threadIdx.x < 6) part[blockIdx.x * 6 + threadIdx.x] = s[threadIdx.x][0];
}

// one block of 256: the partial boxes of up to 256 blocks
__global__ void __launch_bounds__(256) k_bbox_final(int nblk, const double* __restrict__ part, double* __restrict__ box) {
    __shared__ double s[6][256];
    for (int d = 0; d < 6; ++d)
        s[d][threadIdx.x] = threadIdx.x < nblk ? part[threadIdx.x * 6 + d] : d < 3 ? 1e308 : -1e308;
    __syncthreads();
    for (int o = 128; o; o >>= 1) {
        if (threadIdx.x < o)
            for (int d = 0; d < 3; ++d) {
                s[d][threadIdx.x] = fmin(s[d][threadIdx.x], s[d][threadIdx.x + o]);
                s[3 + d][threadIdx.x] = fmax(s[3 + d][threadIdx.x], s[3 + d][threadIdx.x + o]);
            }
        __syncthreads();
    }
    if (threadIdx.x) return;
    const double lo[3] = {s[0][0], s[1][0], s[2][0]}, hi[3] = {s[3][0], s[4][0], s[5][0]};
    double side = 0.0;
    for (int d = 0; d < 3; ++d) {
        const double e = __dsub_rn(hi[d], lo[d]);
        if (e > side) side = e;
    }
    if (side == 0.0) side = 1.0;
    side = __dmul_rn(side, 1.0 + 1e-12);
    box[0] = lo[0]; box[1] = lo[1]; box[2] = lo[2];
    box[3] = side;
    box[4] = __ddiv_rn(2097152.0, side);
}

__device__ __forceinline__ uint64_t spread21(uint64_t v) {
    v &= 0x1fffffull;
    v = (v | (v << 32)) & 0x1f00000000ffffull;
    v = (v | (v << 16)) & 0x1f0000ff0000ffull;
    v = (v | (v << 8)) & 0x100f00f00f00f00full;
    v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
    v = (v | (v << 2)) & 0x1249249249249249ull;
    return v;
}

__global__ void k_morton(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                         const double* __restrict__ z, const double* __restrict__ q, const double* __restrict__ box,
                         uint64_t* __restrict__ key, double2* __restrict__ rec) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v[3] = {x[i], y[i], z[i]};
    uint64_t k = 0;
    for (int d = 0; d < 3; ++d) {
        int64_t c = (int64_t)floor(__dmul_rn(__dsub_rn(v[d], box[d]), box[4]));
        c = c < 0 ? 0 : (c > 2097151 ? 2097151 : c);
        k |= spread21((uint64_t)c) << d;
    }
    key[i] = k;
    rec[2 * i] = make_double2(v[0], v[1]);
    rec[2 * i + 1] = make_double2(v[2], q[i]);
}

// ---------------------------------------------------------------------------
// tree construction, level by level
// ---------------------------------------------------------------------------
// For each node of the level with more than max_leaf particles (and level
// below 21): the octant ranges, 8 lanes per node, each finding the first
// position of its octant by binary search on the sorted keys (one search deep
// instead of seven after another).
__global__ void __launch_bounds__(256)
k_split_count(int lb, int le, int max_leaf, const int* __restrict__ lev, const int* __restrict__ nb,
              const int* __restrict__ ne, const uint64_t* __restrict__ key, int* __restrict__ bounds,
              int* __restrict__ nch) {
    const int c = lb + blockIdx.x * 32 + (threadIdx.x >> 3), o = threadIdx.x & 7;
    int lo = 0, hi = 0, e = 0;
    bool split = false;
    if (c < le) {
        const int b = nb[c], L = lev[c];
        e = ne[c];
        split = e - b > max_leaf && L < 21;
        if (split) {
            const int shift = 3 * (20 - L);
            lo = b;
            hi = o ? e : b;
            while (lo < hi) {   // first position whose octant digit is >= o
                const int mid = (lo + hi) >> 1;
                if ((int)((key[mid] >> shift) & 7ull) < o) lo = mid + 1; else hi = mid;
            }
            bounds[9 * (c - lb) + o] = lo;
            if (o == 7) bounds[9 * (c - lb) + 8] = e;
        }
    }
    const int up = __shfl_down_sync(0xffffffffu, lo, 1);
    const bool has = split && (o == 7 ? e : up) > lo;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    if (c < le && o == 0) nch[c - lb] = __popc((m >> (threadIdx.x & 24)) & 255u);
}

__global__ void k_split_write(int lb, int le, const int* __restrict__ bounds, const int* __restrict__ nch,
                              const int* __restrict__ choff, int* __restrict__ lev, int* __restrict__ ix,
                              int* __restrict__ iy, int* __restrict__ iz, int* __restrict__ nb, int* __restrict__ ne,
                              int* __restrict__ child0, int* __restrict__ nchild, int* __restrict__ parent) {
    const int c = lb + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    const int k = nch[c - lb];
    nchild[c] = k;
    if (!k) { child0[c] = -1; return; }
    const int base = le + choff[c - lb];
    child0[c] = base;
    const int* bd = bounds + 9 * (c - lb);
    int j = 0;
    for (int o = 0; o < 8; ++o) {
        if (bd[o + 1] <= bd[o]) continue;
        const int ch = base + j++;
        lev[ch] = lev[c] + 1;
        ix[ch] = 2 * ix[c] + (o & 1);
        iy[ch] = 2 * iy[c] + ((o >> 1) & 1);
        iz[ch] = 2 * iz[c] + ((o >> 2) & 1);
        nb[ch] = bd[o];
        ne[ch] = bd[o + 1];
        parent[ch] = c;
        child0[ch] = -1;
        nchild[ch] = 0;
    }
}

__device__ __forceinline__ double dist3_rn(const double* a, const double* b) {
    const double dx = __dsub_rn(a[0], b[0]), dy = __dsub_rn(a[1], b[1]), dz = __dsub_rn(a[2], b[2]);
    return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)));
}

__global__ void k_centres(int nn, const int* __restrict__ lev, const int* __restrict__ ix, const int* __restrict__ iy,
                          const int* __restrict__ iz, const double* __restrict__ box, double* __restrict__ zc) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nn) return;
    const double h = __ddiv_rn(box[3], (double)(1ull << lev[c]));
    zc[3 * c] = __dadd_rn(box[0], __dmul_rn((double)ix[c] + 0.5, h));
    zc[3 * c + 1] = __dadd_rn(box[1], __dmul_rn((double)iy[c] + 0.5, h));
    zc[3 * c + 2] = __dadd_rn(box[2], __dmul_rn((double)iz[c] + 0.5, h));
}

// Centres of mass of the nodes [lb, lb + n) (one level, children done), the
// AP variant's expansion centres: a leaf sums q_a x_a and q_a over its
// particles in sorted order, a cell sums Q_c z_c and Q_c over its children
// in octant order, z = S / Q; explicitly rounded FP64 in the oracle's order,
// so both trees have the same centres, radii and lists.  A node of zero
// total charge keeps its geometric centre.
__global__ void k_com(int lb, int le, const int* __restrict__ nb, const int* __restrict__ ne,
                      const int* __restrict__ child0, const int* __restrict__ nchild, const double* __restrict__ xs,
                      const double* __restrict__ ys, const double* __restrict__ zs, const double* __restrict__ qs,
                      double* __restrict__ Q, double* __restrict__ zc) {
    const int c = lb + blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= le) return;
    double q = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    if (nchild[c] == 0) {
        for (int a = nb[c]; a < ne[c]; ++a) {
            q = __dadd_rn(q, qs[a]);
            sx = __dadd_rn(sx, __dmul_rn(qs[a], xs[a]));
            sy = __dadd_rn(sy, __dmul_rn(qs[a], ys[a]));
            sz = __dadd_rn(sz, __dmul_rn(qs[a], zs[a]));
        }
    } else {
        for (int k = 0; k < nchild[c]; ++k) {
            const int ch = child0[c] + k;
            q = __dadd_rn(q, Q[ch]);
            sx = __dadd_rn(sx, __dmul_rn(Q[ch], zc[3 * ch]));
            sy = __dadd_rn(sy, __dmul_rn(Q[ch], zc[3 * ch + 1]));
            sz = __dadd_rn(sz, __dmul_rn(Q[ch], zc[3 * ch + 2]));
        }
    }
    Q[c] = q;
    if (q != 0.0) {
        zc[3 * c] = __ddiv_rn(sx, q);
        zc[3 * c + 1] = __ddiv_rn(sy, q);
        zc[3 * c + 2] = __ddiv_rn(sz, q);
    }
}

// AP: the dipole (rank-1 components 1..3 of the node-major multipoles) set to 0
__global__ void k_zero_dipole(int nn, int nc, double* __restrict__ M) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nn) { M[(int64_t)c * nc + 1] = 0.0; M[(int64_t)c * nc + 2] = 0.0; M[(int64_t)c * nc + 3] = 0.0; }
}

// radii in units of side / 2^22 (the unit of the integer centres), rounded to FP32
__global__ void k_radf(int nn, const double* __restrict__ rad, const double* __restrict__ box,
                       float* __restrict__ radf) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nn) radf[c] = (float)(rad[c] / box[3] * 4194304.0);
}
int ad_radf(int nn, const double* rad, const double* box, float* radf, cudaStream_t s) {
    if (nn > 0) { k_radf<<<(nn + 255) / 256, 256, 0, s>>>(nn, rad, box, radf); count_launch(); }
    return 0;
}

// Radii of the nodes [lb, le) (one level), children already done: 8 lanes per
// node over its particles (leaf) or children.  The rounded square root is
// monotonic, so a leaf's largest distance is the root of its largest square:
// one root per leaf instead of one per particle (some 20 FP64 instructions
// each).
__global__ void __launch_bounds__(256)
k_radii(int lb, int le, const int* __restrict__ nb, const int* __restrict__ ne, const int* __restrict__ child0,
        const int* __restrict__ nchild, const double* __restrict__ zc, const double* __restrict__ xs,
        const double* __restrict__ ys, const double* __restrict__ zs, double* __restrict__ rad) {
    const int c = lb + blockIdx.x * 32 + (threadIdx.x >> 3), sub = threadIdx.x & 7;
    double r = 0.0;
    int nk = 0;
    if (c < le) {
        const double* z = zc + 3 * c;
        nk = nchild[c];
        if (nk == 0) {
            const double zx = z[0], zy = z[1], zz = z[2];
            for (int a = nb[c] + sub; a < ne[c]; a += 8) {
                const double dx = __dsub_rn(xs[a], zx), dy = __dsub_rn(ys[a], zy), dz = __dsub_rn(zs[a], zz);
                const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                if (d2 > r) r = d2;
            }
        } else if (sub < nk) {
            const int ch = child0[c] + sub;
            r = __dadd_rn(dist3_rn(zc + 3 * ch, z), rad[ch]);
        }
    }
#pragma unroll
    for (int o = 4; o; o >>= 1) r = fmax(r, __shfl_xor_sync(0xffffffffu, r, o));
    if (c < le && sub == 0) rad[c] = nk == 0 ? __dsqrt_rn(r) : r;
}

// ---------------------------------------------------------------------------
// directed dual-tree traversal, one breadth-first step per launch pair
// ---------------------------------------------------------------------------
// mode per pair: 0 = M2L, 1 = P2P, 2 = self split, 3 = split target, 4 = split source.
// The MAC theta |z_A - z_B| > r_A + r_B is evaluated squared (both sides are
// non-negative), theta^2 |z_A - z_B|^2 > (r_A + r_B)^2, with explicitly rounded
// FP64 operations in the oracle's order: no square root per pair.
__device__ __forceinline__ int trav_mode(int A, int B, double theta, const int* nchild, const double* zc,
                                         const double* rad) {
    const bool la = nchild[A] == 0, lb = nchild[B] == 0;
    if (A == B) return la ? 1 : 2;
    const double* a = zc + 3 * A;
    const double* b = zc + 3 * B;
    const double dx = __dsub_rn(a[0], b[0]), dy = __dsub_rn(a[1], b[1]), dz = __dsub_rn(a[2], b[2]);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    const double sr = __dadd_rn(rad[A], rad[B]);
    if (__dmul_rn(__dmul_rn(theta, theta), d2) > __dmul_rn(sr, sr)) return 0;
    if (la && lb) return 1;
    if (!la && (lb || rad[A] >= rad[B])) return 3;
    return 4;
}

// FP32 screen of the MAC, in units of side / 2^22 so that no operand leaves
// FP32's normal range: the centre offset is the exact integer difference of
// the integer centres (below 2^23, exact in FP32), the radii are FP32
// copies in the same unit.  Outside a relative band around the boundary
// (wider than the FP32 rounding plus that of the FP64 centres) the FP32
// comparison gives the FP64 rule's answer; inside it the pair is decided by
// trav_mode in FP64.  Returns 0 (accept), 1 (reject), 2 (undecided).
__device__ __forceinline__ int mac_screen(int A, int B, float theta2, float band, const int4* __restrict__ ic,
                                          const float* __restrict__ radf) {
    const int4 a = ic[A], b = ic[B];
    const float dx = (float)(a.x - b.x), dy = (float)(a.y - b.y), dz = (float)(a.z - b.z);
    const float lhs = theta2 * (dx * dx + dy * dy + dz * dz);
    const float sr = radf[A] + radf[B];
    const float rhs = sr * sr;
    if (lhs > rhs * (1.f + band)) return 0;
    if (lhs < rhs * (1.f - band)) return 1;
    return 2;
}

// One step of the traversal over the frontier of nq pairs, in tiles of
// TRAV_TILE pairs per block: k_trav_count decides every pair once (its mode is
// kept) and counts the tile's M2L, P2P and next-frontier entries, k_trav_scan
// scans the three rows of tile counts (a block each), k_trav_write recomputes
// the offsets inside its tile and writes the entries in frontier order.
// Bound: memory; a pair takes 8 bytes and its mode twice and its entry once
// (26 bytes) instead of three full-length scans between two passes (about 100).
constexpr int TRAV_TILE = 1024;
__device__ __forceinline__ unsigned long long trav_pack(int m, int A, int B, const int* __restrict__ nchild) {
    // M2L | P2P << 16 | frontier << 32 (a tile holds at most 1024, 1024 and 65536)
    if (m == 0) return 1ull;
    if (m == 1) return 1ull << 16;
    const int na = nchild[A];
    return (unsigned long long)(m == 2 ? na * na : m == 3 ? na : nchild[B]) << 32;
}
__global__ void __launch_bounds__(256)
k_trav_count(int nq, const int2* __restrict__ q, double theta, const int* __restrict__ nchild,
             const double* __restrict__ zc, const double* __restrict__ rad, unsigned char* __restrict__ mode,
             const int4* __restrict__ ic, const float* __restrict__ radf, float theta2, float band, int ntile,
             int* __restrict__ tsum) {
    __shared__ unsigned long long ws[8];
    unsigned long long t = 0;
#pragma unroll
    for (int r = 0; r < TRAV_TILE / 256; ++r) {
        const int64_t k = (int64_t)blockIdx.x * TRAV_TILE + r * 256 + threadIdx.x;
        if (k >= nq) break;
        const int A = q[k].x, B = q[k].y;
        int m;
        const int sc = A == B ? 2 : mac_screen(A, B, theta2, band, ic, radf);
        if (sc == 0) {
            m = 0;
        } else if (sc == 1) {
            const bool la = nchild[A] == 0, lb = nchild[B] == 0;
            m = (la && lb) ? 1 : (!la && (lb || rad[A] >= rad[B])) ? 3 : 4;
        } else {
            m = trav_mode(A, B, theta, nchild, zc, rad);
        }
        mode[k] = (unsigned char)m;
        t += trav_pack(m, A, B, nchild);
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) t += ws[w];
        tsum[blockIdx.x] = (int)(t & 0xffff);
        tsum[ntile + blockIdx.x] = (int)((t >> 16) & 0xffff);
        tsum[2 * ntile + blockIdx.x] = (int)(t >> 32);
    }
}

// exclusive scan of row blockIdx.x of the tile counts in place, total to tot
__global__ void __launch_bounds__(1024) k_trav_scan(int ntile, int* __restrict__ tsum, int* __restrict__ tot) {
    __shared__ int ws[32];
    int* row = tsum + (int64_t)blockIdx.x * ntile;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int carry = 0;
    for (int b = 0; b < ntile; b += 8 * 1024) {
        int v[8], t = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = b + 8 * threadIdx.x + j;
            v[j] = i < ntile ? row[i] : 0;
            t += v[j];
        }
        int inc = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        int x = ws[lane];
        const int own = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += u;
        }
        int ex = carry + __shfl_sync(0xffffffffu, x - own, w) + inc - t;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int i = b + 8 * threadIdx.x + j;
            if (i < ntile) row[i] = ex;
            ex += v[j];
        }
        carry += __shfl_sync(0xffffffffu, x, 31);
        __syncthreads();
    }
    if (threadIdx.x == 0) tot[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(256)
k_trav_write(int nq, const int2* __restrict__ q, const unsigned char* __restrict__ mode,
             const int* __restrict__ nchild, const int* __restrict__ child0, int ntile, const int* __restrict__ tsum,
             uint32_t* __restrict__ mt, int* __restrict__ ms, uint32_t* __restrict__ pt, int* __restrict__ ps,
             int2* __restrict__ qn) {
    __shared__ unsigned long long ws[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int om = tsum[blockIdx.x], op = tsum[ntile + blockIdx.x], oq = tsum[2 * ntile + blockIdx.x];
    for (int r = 0; r < TRAV_TILE / 256; ++r) {
        const int64_t k = (int64_t)blockIdx.x * TRAV_TILE + r * 256 + threadIdx.x;
        int A = 0, B = 0, m = 0;
        unsigned long long t = 0;
        if (k < nq) {
            const int2 ab = q[k];
            A = ab.x; B = ab.y;
            m = mode[k];
            t = trav_pack(m, A, B, nchild);
        }
        unsigned long long inc = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) ws[w] = inc;
        __syncthreads();
        unsigned long long pre = inc - t, tot = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            pre += j < w ? ws[j] : 0;
            tot += ws[j];
        }
        if (k < nq) {
            if (m == 0) {
                const int o = om + (int)(pre & 0xffff);
                mt[o] = (uint32_t)A; ms[o] = B;
            } else if (m == 1) {
                const int o = op + (int)((pre >> 16) & 0xffff);
                pt[o] = (uint32_t)A; ps[o] = B;
            } else {
                int o = oq + (int)(pre >> 32);
                const int na = nchild[A], ca = child0[A];
                if (m == 2) {
                    for (int i = 0; i < na; ++i)
                        for (int j = 0; j < na; ++j) qn[o++] = make_int2(ca + i, ca + j);
                } else if (m == 3) {
                    for (int i = 0; i < na; ++i) qn[o++] = make_int2(ca + i, B);
                } else {
                    const int nbc = nchild[B], cb = child0[B];
                    for (int j = 0; j < nbc; ++j) qn[o++] = make_int2(A, cb + j);
                }
            }
        }
        om += (int)(tot & 0xffff);
        op += (int)((tot >> 16) & 0xffff);
        oq += (int)(tot >> 32);
        __syncthreads();
    }
}

// CSR offsets of pairs sorted by target: off[t] = first position whose target
// is >= t (a binary search per target instead of counting atomics and a scan)
__global__ void k_csr_off(int n, int nn, const uint32_t* __restrict__ key, int* __restrict__ off) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t > nn) return;
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (int)(((unsigned)lo + (unsigned)hi) >> 1);
        if (key[mid] < (uint32_t)t) lo = mid + 1; else hi = mid;
    }
    off[t] = lo;
}

// M2L work order: targets with non-empty lists, longest lists first (lengths
// from 65535 on count as equal: a schedule only); counts the targets with a
// list and the leaves
__global__ void k_len_keys(int nn, const int* __restrict__ off, const int* __restrict__ nchild,
                           uint32_t* __restrict__ key, int* __restrict__ counts) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    int len = 0, leaf = 0;
    if (c < nn) {
        len = off[c + 1] - off[c];
        leaf = nchild[c] == 0;
        key[c] = 65535u - (uint32_t)min(len, 65535);
    }
    const int nt = __popc(__ballot_sync(0xffffffffu, len > 0)), nl = __popc(__ballot_sync(0xffffffffu, leaf));
    if ((threadIdx.x & 31) == 0) {
        if (nt) atomicAdd(counts, nt);
        if (nl) atomicAdd(counts + 1, nl);
    }
}

// leaves in particle order: key = first particle, the other nodes after all
__global__ void k_leaf_keys(int nn, int n, const int* __restrict__ nchild, const int* __restrict__ nb,
                            uint32_t* __restrict__ key) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < nn) key[c] = (uint32_t)(nchild[c] ? n : nb[c]);
}

// sorted copies of the particles; the octree gathers them from the 32-byte
// records that k_morton wrote beside the keys (one sector per particle
// instead of four)
__global__ void k_gather_sorted(int64_t n, const int* __restrict__ perm, const double* __restrict__ x,
                                const double* __restrict__ y, const double* __restrict__ z,
                                const double* __restrict__ q, double* __restrict__ xs, double* __restrict__ ys,
                                double* __restrict__ zs, double* __restrict__ qs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int o = perm[i];
    xs[i] = x[o]; ys[i] = y[o]; zs[i] = z[o]; qs[i] = q[o];
}
__global__ void k_gather_rec(int64_t n, const int* __restrict__ perm, const double2* __restrict__ rec,
                             double* __restrict__ xs, double* __restrict__ ys, double* __restrict__ zs,
                             double* __restrict__ qs) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t o = perm[i];
    const double2 a = rec[2 * o], b = rec[2 * o + 1];
    xs[i] = a.x; ys[i] = a.y; zs[i] = b.x; qs[i] = b.y;
}

// ---------------------------------------------------------------------------
// launch helpers
// ---------------------------------------------------------------------------
#define G256(n) (unsigned)(((int64_t)(n) + 255) / 256), 256, 0, s
int ad_bbox(int64_t n, const double* x, const double* y, const double* z, double* part, double* box, cudaStream_t s) {
    const int nblk = 256;
    k_bbox_partial<<<nblk, 256, 0, s>>>(n, x, y, z, part);
    k_bbox_final<<<1, 256, 0, s>>>(nblk, part, box);
    count_launch(); count_launch();
    return 0;
}
int ad_morton(int64_t n, const double* x, const double* y, const double* z, const double* q, const double* box,
              uint64_t* key, double* rec, cudaStream_t s) {
    if (n) { k_morton<<<G256(n)>>>(n, x, y, z, q, box, key, (double2*)rec); count_launch(); }
    return 0;
}
int ad_gather_rec(int64_t n, const int* perm, const double* rec, double* xs, double* ys, double* zs, double* qs,
                  cudaStream_t s) {
    if (n) { k_gather_rec<<<G256(n)>>>(n, perm, (const double2*)rec, xs, ys, zs, qs); count_launch(); }
    return 0;
}
int ad_gather(int64_t n, const int* perm, const double* x, const double* y, const double* z, const double* q,
              double* xs, double* ys, double* zs, double* qs, cudaStream_t s) {
    if (n) { k_gather_sorted<<<G256(n)>>>(n, perm, x, y, z, q, xs, ys, zs, qs); count_launch(); }
    return 0;
}
int ad_split_count(int lb, int le, int max_leaf, const int* lev, const int* nb, const int* ne, const uint64_t* key,
                   int* bounds, int* nch, cudaStream_t s) {
    k_split_count<<<(unsigned)((le - lb + 31) / 32), 256, 0, s>>>(lb, le, max_leaf, lev, nb, ne, key, bounds, nch);
    count_launch();
    return 0;
}
int ad_split_write(int lb, int le, const int* bounds, const int* nch, const int* choff, int* lev, int* ix, int* iy,
                   int* iz, int* nb, int* ne, int* child0, int* nchild, int* parent, cudaStream_t s) {
    k_split_write<<<G256(le - lb)>>>(lb, le, bounds, nch, choff, lev, ix, iy, iz, nb, ne, child0, nchild, parent);
    count_launch();
    return 0;
}
int ad_centres(int nn, const int* lev, const int* ix, const int* iy, const int* iz, const double* box, double* zc,
               cudaStream_t s) {
    k_centres<<<G256(nn)>>>(nn, lev, ix, iy, iz, box, zc);
    count_launch();
    return 0;
}
int ad_com(int lb, int le, const int* nb, const int* ne, const int* child0, const int* nchild, const double* xs,
           const double* ys, const double* zs, const double* qs, double* Q, double* zc, cudaStream_t s) {
    if (le <= lb) return 0;
    k_com<<<(le - lb + 255) / 256, 256, 0, s>>>(lb, le, nb, ne, child0, nchild, xs, ys, zs, qs, Q, zc);
    count_launch();
    return 0;
}
int ad_zero_dipole(int nn, int nc, double* M, cudaStream_t s) {
    if (nn <= 0 || nc < 4) return 0;
    k_zero_dipole<<<(nn + 255) / 256, 256, 0, s>>>(nn, nc, M);
    count_launch();
    return 0;
}

int ad_radii(int lb, int le, const int* nb, const int* ne, const int* child0, const int* nchild, const double* zc,
             const double* xs, const double* ys, const double* zs, double* rad, cudaStream_t s) {
    k_radii<<<(unsigned)((le - lb + 31) / 32), 256, 0, s>>>(lb, le, nb, ne, child0, nchild, zc, xs, ys, zs, rad);
    count_launch();
    return 0;
}
int ad_trav_tiles(int nq) { return (int)(((int64_t)nq + TRAV_TILE - 1) / TRAV_TILE); }
int ad_trav_count(int nq, const int2* q, double theta, const int* nchild, const double* zc, const double* rad,
                  unsigned char* mode, const int4* ic, const float* radf, float band, int* tsum, int* tot,
                  cudaStream_t s) {
    const int nt = ad_trav_tiles(nq);
    k_trav_count<<<nt, 256, 0, s>>>(nq, q, theta, nchild, zc, rad, mode, ic, radf, (float)(theta * theta), band, nt,
                                    tsum);
    k_trav_scan<<<3, 1024, 0, s>>>(nt, tsum, tot);
    count_launch(); count_launch();
    return 0;
}
int ad_trav_write(int nq, const int2* q, const unsigned char* mode, const int* nchild, const int* child0,
                  const int* tsum, uint32_t* mt, int* ms, uint32_t* pt, int* ps, int2* qn, cudaStream_t s) {
    const int nt = ad_trav_tiles(nq);
    k_trav_write<<<nt, 256, 0, s>>>(nq, q, mode, nchild, child0, nt, tsum, mt, ms, pt, ps, qn);
    count_launch();
    return 0;
}
int ad_csr_off(int n, int nn, const uint32_t* key, int* off, cudaStream_t s) {
    k_csr_off<<<G256(nn + 1)>>>(n, nn, key, off);
    count_launch();
    return 0;
}
int ad_len_keys(int nn, const int* off, const int* nchild, uint32_t* key, int* counts, cudaStream_t s) {
    k_len_keys<<<G256(nn)>>>(nn, off, nchild, key, counts);
    count_launch();
    return 0;
}
int ad_leaf_keys(int nn, int n, const int* nchild, const int* nb, uint32_t* key, cudaStream_t s) {
    k_leaf_keys<<<G256(nn)>>>(nn, n, nchild, nb, key);
    count_launch();
    return 0;
}
// Folded multipoles of the list M2L: row c of F holds the reduced
// representative of node c's multipole with the weights of Eq. M2L,
//   c_(a,b,c) = sum_{i <= a/2, k <= b/2} (-1)^(i+k) C(i+k, i) M_m / m!,
//   m = (a - 2i, b - 2k, c + 2(i + k)),  c = 0 or 1
// (traceless storage: with the dependent M_m written out in the stored ones),
// summed in FP64 and rounded once to T, rows of ldm, padded with zeros.  Done once per node here instead of once
// per pair: a row is nt(p) components instead of ns(p) (p = 6: 49 instead of 84),
// which the M2L kernels gather per pair.  The terms of a component are a table
// (generated, the same for every order), copied to shared memory once per
// FOLD_ROWS rows.  Bound: reading the expansions.
constexpr int FOLD_ROWS = 64;
template <typename T>
__global__ void __launch_bounds__(256)
k_fold(int64_t rows, int p, int basis, int ldm, const double* __restrict__ M, T* __restrict__ F) {
    __shared__ double sC[FMM_FOLD_MAX];
    __shared__ unsigned short sIdx[FMM_FOLD_MAX], sOff[FMM_NT_MAX + 1];
    const int nt = nt_of(p), nc = ncoef_of(p, basis);
    const unsigned short* off = basis ? d_fold_off1 : d_fold_off0;
    const unsigned short* idx = basis ? d_fold_idx1 : d_fold_idx0;
    const double* cf = basis ? d_fold_c1 : d_fold_c0;
    for (int t = threadIdx.x; t <= nt; t += 256) sOff[t] = off[t];
    for (int k = threadIdx.x; k < off[nt]; k += 256) { sIdx[k] = idx[k]; sC[k] = cf[k]; }
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * FOLD_ROWS;
    const int cnt = (int)(rows - r0 < FOLD_ROWS ? rows - r0 : FOLD_ROWS) * ldm;
    for (int i = threadIdx.x; i < cnt; i += 256) {
        const int r = i / ldm, t = i - r * ldm;
        double v = 0.0;
        if (t < nt) {
            const double* Mr = M + (r0 + r) * nc;
            for (int k = sOff[t]; k < sOff[t + 1]; ++k) v = fma(sC[k], Mr[sIdx[k]], v);
        }
        F[r0 * ldm + i] = T(v);
    }
}
int ad_fold(int prec, int64_t rows, int p, int basis, int ldm, const double* M, void* F, cudaStream_t s) {
    if (rows <= 0) return 0;
    const unsigned g = (unsigned)((rows + FOLD_ROWS - 1) / FOLD_ROWS);
    if (prec) k_fold<float><<<g, 256, 0, s>>>(rows, p, basis, ldm, M, (float*)F);
    else k_fold<double><<<g, 256, 0, s>>>(rows, p, basis, ldm, M, (double*)F);
    count_launch();
    return 0;
}
// M2M and L2L of one level (generated adshift_P<p>.cu; physical units, or the
// cells' scaled units in FP32)
#define AD_SHIFT(P)                                                                                               \
    int launch_ad_m2m_p##P(int prec, int basis, int lb, int le, const int* child0, const int* nchild,            \
                           const double* zc, const int4* ic, double* Mn, const DevTables& Tb, cudaStream_t s);    \
    int launch_ad_l2l_p##P(int prec, int basis, int lb, int le, const int* parent, const double* zc,             \
                           const int4* ic, double* Ln, cudaStream_t s);
AD_SHIFT(0) AD_SHIFT(1) AD_SHIFT(2) AD_SHIFT(3) AD_SHIFT(4) AD_SHIFT(5)
AD_SHIFT(6) AD_SHIFT(7) AD_SHIFT(8) AD_SHIFT(9) AD_SHIFT(10)
#undef AD_SHIFT
int ad_m2m(int prec, int p, int basis, int lb, int le, const int* child0, const int* nchild, const double* zc,
           const int4* ic, double* Mn, const DevTables& Tb, cudaStream_t s) {
    static decltype(&launch_ad_m2m_p0) const f[FMM_PMAX + 1] = {
        launch_ad_m2m_p0, launch_ad_m2m_p1, launch_ad_m2m_p2, launch_ad_m2m_p3, launch_ad_m2m_p4, launch_ad_m2m_p5,
        launch_ad_m2m_p6, launch_ad_m2m_p7, launch_ad_m2m_p8, launch_ad_m2m_p9, launch_ad_m2m_p10};
    if (le <= lb) return 0;
    f[p](prec ? 1 : 0, basis, lb, le, child0, nchild, zc, ic, Mn, Tb, s);
    count_launch();
    return 0;
}
int ad_l2l(int prec, int p, int basis, int lb, int le, const int* parent, const double* zc, const int4* ic,
           double* Ln, cudaStream_t s) {
    static decltype(&launch_ad_l2l_p0) const f[FMM_PMAX + 1] = {
        launch_ad_l2l_p0, launch_ad_l2l_p1, launch_ad_l2l_p2, launch_ad_l2l_p3, launch_ad_l2l_p4, launch_ad_l2l_p5,
        launch_ad_l2l_p6, launch_ad_l2l_p7, launch_ad_l2l_p8, launch_ad_l2l_p9, launch_ad_l2l_p10};
    if (le <= lb) return 0;
    f[p](prec ? 1 : 0, basis, lb, le, parent, zc, ic, Ln, s);
    count_launch();
    return 0;
}
#undef G256

}  // namespace fmm
