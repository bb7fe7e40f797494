// Host side of the uniform M2L by reflections (fmm_reflect.cuh): the folded
// multipoles of all levels, the split of the lists into warps' shares, and the
// sums of the shares' partial results.
#include <algorithm>

#include "fmm_internal.h"
#include "_gen/fmm_fold.cuh"

namespace fmm {

constexpr int RF_PAD_CELLS = 32;   // RF_PAD of fmm_reflect.cuh

#define RF_DECL(P)                                                                                                  \
    int launch_m2l_rf_p##P##_float_float(const RfLevels&, const void*, const double*, void*, void*, int, int, int,  \
                                         cudaStream_t);                                                             \
    int launch_m2l_rf_p##P##_float_double(const RfLevels&, const void*, const double*, void*, void*, int, int, int, \
                                          cudaStream_t);                                                            \
    int launch_m2l_rf_p##P##_double_double(const RfLevels&, const void*, const double*, void*, void*, int, int, int, \
                                           cudaStream_t);
RF_DECL(0) RF_DECL(1) RF_DECL(2) RF_DECL(3) RF_DECL(4) RF_DECL(5)
RF_DECL(6) RF_DECL(7) RF_DECL(8) RF_DECL(9) RF_DECL(10)
#undef RF_DECL

int64_t rf_fold_elems(int p, int lo, int hi) {
    int64_t n = 0;
    for (int l = lo; l <= hi; ++l) n += nt_of(p) * (((int64_t)1 << (3 * l)) + RF_PAD_CELLS);
    return n;
}

static int64_t rf_warps(int l) {   // warps of 32 cells of one class
    const int64_t h3 = (int64_t)1 << (3 * (l - 1));
    return 8 * std::max<int64_t>(1, h3 / 32);
}

// Shares of the 56 orbits per cell of level l of a plan whose levels 2..deep
// run here: one where the level alone gives 32 warps per SM; else so many that
// all levels together give about 24 warps per SM (three times what an SM holds
// in FP64 at p = 8: the last shares are short), at most `most`.  It does not
// depend on the levels of one call: a call per level sums as one call does.
// FP32 (f32): an orbit per share on levels 2 and 3.  Most of the far potential
// comes from them, and a thread's sum over many orbits rounds each product at
// the size of the whole sum (k_rf_sum adds the shares without that).  Rounding
// error of the far potential, depth 5, p = 4 / 6 / 8 traceless, rms: 1.91 / 2.33 /
// 2.54e-7 with the rule below on every level, 1.74 / 2.15 / 2.31e-7 so (1.80 /
// 2.21 / 2.40e-7 with offset by offset sums); the M2L 113 / 273 / 691 -> 121 / 265
// / 650 us at 1,000,003 particles.
static int rf_shares(int l, int deep, int sms, int most, bool f32) {
    if (f32 && l <= 3) return most;
    int64_t tot = 0;
    for (int k = 2; k <= deep; ++k) tot += rf_warps(k);
    if (rf_warps(l) >= 32 * (int64_t)sms) return 1;
    return (int)std::max<int64_t>(1, std::min<int64_t>(most, (24 * (int64_t)sms + tot - 1) / tot));
}

// layout of levels lo..hi; returns the number of units (warps' shares)
static int rf_levels(int nrow, int lo, int hi, int deep, const int64_t* lvl_off, int p, int sms, int most, bool f32,
                     RfLevels& lv) {
    int64_t F = 0, part = 0;
    int unit = 0;
    lv.n = 0;
    for (int l = lo; l <= hi; ++l) {
        RfLevel& v = lv.v[lv.n++];
        v.l = l;
        v.g = rf_shares(l, deep, sms, most, f32);
        unit += (int)rf_warps(l) * v.g;
        v.end = unit;
        v.F = F;
        v.L = lvl_off[l] - lvl_off[lo];
        v.part = part;
        F += nt_of(p) * (((int64_t)1 << (3 * l)) + RF_PAD_CELLS);
        if (v.g > 1) part += (int64_t)v.g * nrow << (3 * l);
    }
    return unit;
}

static int rf_sms() {
    int d = 0, sms = 0;
    cudaGetDevice(&d);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, d);
    return sms > 0 ? sms : 1;
}

int64_t rf_part_elems(int nrow, int deep, int most, bool f32) {
    int64_t n = 0;
    for (int l = 2; l <= deep; ++l) {
        const int g = rf_shares(l, deep, rf_sms(), most, f32);
        if (g > 1) n += (int64_t)g * nrow << (3 * l);
    }
    return n;
}

// Folded multipoles, component-major with RF_PAD_CELLS zero cells after each
// row: from symmetric storage (sym) the fold of k_fold, from the uniform
// plans' traceless storage (already the reduced representative) c_t = M_t / t!.
template <typename TI, typename T>
__global__ void __launch_bounds__(256)
k_rf_fold(int sym, int nc, int nt, int lo, int hi, const TI* __restrict__ M, T* __restrict__ F) {
    const int t = blockIdx.y;
    int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
    int64_t ncell = 0;
    for (int l = lo; l <= hi; ++l) {
        ncell = (int64_t)1 << (3 * l);
        if (i < ncell + RF_PAD_CELLS) break;
        i -= ncell + RF_PAD_CELLS;
        M += nc * ncell;
        F += nt * (ncell + RF_PAD_CELLS);
        if (l == hi) return;
    }
    T v = T(0);
    if (i < ncell) {
        if (sym) {
            const int k1 = d_fold_off0[t + 1];
            for (int k = d_fold_off0[t]; k < k1; ++k)
                v = fma(T(d_fold_c0[k]), T(M[(int64_t)d_fold_idx0[k] * ncell + i]), v);
        } else {
            const double inv = c_invfact[c_tl_idx[t][0]] * c_invfact[c_tl_idx[t][1]];   // nz <= 1
            v = T(M[(int64_t)t * ncell + i]) * T(inv);
        }
    }
    F[(int64_t)t * (ncell + RF_PAD_CELLS) + i] = v;
}

// one more share's partial sum onto s; FP32: its rounding error, exact, onto c
template <typename OT>
__device__ __forceinline__ void rf_add(OT a, OT& s, OT& c) {
    const OT t = s + a;
    if constexpr (sizeof(OT) == 4) {
        const OT u = t - s;
        c += (s - (t - u)) + (a - u);
    }
    s = t;
}

// Partial sums of the split levels, in a fixed order; FP32 sums carry their
// rounding errors along, so that the result is rounded once whatever the number
// of shares.  Where levels of up to 512 cells have more than RF_FEW shares, the
// first `deep` blocks take 32 components each, a warp every eighth share (a thread
// alone would wait for 56 loads in turn; loads unrolled in flight took longer
// still, for the instructions' own fetches: depth 2, p = 3, 18 and 27 us; so 6.5).
constexpr int RF_FEW = 8;
__host__ __device__ __forceinline__ bool rf_many(const RfLevel& v) { return v.l <= 3 && v.g > RF_FEW; }
template <typename OT>
__global__ void __launch_bounds__(256)
k_rf_sum(RfLevels lv, int nrow, int deep, const OT* __restrict__ part, OT* __restrict__ Lt) {
    __shared__ OT sS[8][32], sC[8][32];
    const bool many = (int)blockIdx.x < deep;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int64_t i = many ? (int64_t)blockIdx.x * 32 + lane : (int64_t)(blockIdx.x - deep) * 256 + threadIdx.x;
    int k = 0;
    for (; k < lv.n; ++k) {
        if (rf_many(lv.v[k]) != many || lv.v[k].g == 1) continue;
        const int64_t m = (int64_t)nrow << (3 * lv.v[k].l);
        if (i < m) break;
        i -= m;
    }
    if (k >= lv.n) return;   // many: the components are a multiple of 32, so never
    const RfLevel& v = lv.v[k];
    const int64_t m = (int64_t)nrow << (3 * v.l);
    const OT* p = part + v.part + i;
    OT s = OT(0), c = OT(0);
    if (!many) {
#pragma unroll 4
        for (int g = 0; g < v.g; ++g) rf_add(p[g * m], s, c);
    } else {
#pragma unroll 1
        for (int g = w; g < v.g; g += 8) rf_add(p[g * m], s, c);
        sS[w][lane] = s;
        sC[w][lane] = c;
        __syncthreads();
        if (w) return;
#pragma unroll 1
        for (int g = 1; g < 8; ++g) {
            rf_add(sS[g][lane], s, c);
            c += sC[g][lane];
        }
    }
    Lt[v.L + i] = s + c;
}

// M2L of the uniform levels lo..hi of a plan whose levels 2..deep run here.
// out: 0 FP64 arithmetic, 1 FP32 with FP64 locals, 2 FP32 with FP32 locals.
// symM, symL: symmetric storage of the multipoles and the locals.  M: the
// multipoles from level lo on (M32 instead where given: their FP32 copy), Lt:
// the locals from level lo on, lvl_off: the levels' offsets.  F: rf_fold_elems
// elements, part: rf_part_elems with the same `most` (shares at most, 1..56) and f32 = (out != 0).
// Returns the launches made.
int launch_m2l_reflect(int out, int p, int symM, int symL, int lo, int hi, int deep, const int64_t* lvl_off,
                       const double* M, const float* M32, const double* Dtab, void* F, void* Lt, void* part, int most,
                       cudaStream_t s) {
    if (lo > hi) return 0;
    const int nt = nt_of(p), ncM = symM ? ns_of(p) : nt, nrow = symL ? ns_of(p) : nt;
    RfLevels lv;
    const int units = rf_levels(nrow, lo, hi, deep, lvl_off, p, rf_sms(), most, out != 0, lv);
    int64_t cells = 0, many = 0, few = 0;   // components summed over many shares, over few
    for (int l = lo; l <= hi; ++l) cells += ((int64_t)1 << (3 * l)) + RF_PAD_CELLS;
    for (int i = 0; i < lv.n; ++i)
        if (lv.v[i].g > 1) (rf_many(lv.v[i]) ? many : few) += (int64_t)nrow << (3 * lv.v[i].l);
    const dim3 gf((unsigned)((cells + 255) / 256), (unsigned)nt);
    if (out == 0) k_rf_fold<double, double><<<gf, 256, 0, s>>>(symM, ncM, nt, lo, hi, M, (double*)F);
    else if (M32) k_rf_fold<float, float><<<gf, 256, 0, s>>>(symM, ncM, nt, lo, hi, M32, (float*)F);
    else k_rf_fold<double, float><<<gf, 256, 0, s>>>(symM, ncM, nt, lo, hi, M, (float*)F);
    typedef int (*fn)(const RfLevels&, const void*, const double*, void*, void*, int, int, int, cudaStream_t);
#define RF_ROW(P) {launch_m2l_rf_p##P##_double_double, launch_m2l_rf_p##P##_float_double, launch_m2l_rf_p##P##_float_float}
    static const fn f[FMM_PMAX + 1][3] = {RF_ROW(0), RF_ROW(1), RF_ROW(2), RF_ROW(3), RF_ROW(4), RF_ROW(5),
                                          RF_ROW(6), RF_ROW(7), RF_ROW(8), RF_ROW(9), RF_ROW(10)};
#undef RF_ROW
    int n = 1 + f[p][out](lv, F, Dtab, Lt, part, symL, nrow, (units + 3) / 4, s);
    if (many + few > 0) {
        const unsigned deep = (unsigned)(many / 32), g = deep + (unsigned)((few + 255) / 256);
        if (out == 2) k_rf_sum<float><<<g, 256, 0, s>>>(lv, nrow, (int)deep, (const float*)part, (float*)Lt);
        else k_rf_sum<double><<<g, 256, 0, s>>>(lv, nrow, (int)deep, (const double*)part, (double*)Lt);
        ++n;
    }
    return n;
}

}  // namespace fmm
