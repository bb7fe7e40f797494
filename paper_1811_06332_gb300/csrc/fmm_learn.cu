// Learned per-pair M2L order (an addition to the paper, which fixes one
// order per run): per-pair features and FP64 truncation-error labels of an
// adaptive plan's M2L list, and an FP32 trainer (forward, backward, Adam)
// for the 11 -> 64 -> 64 -> 64 -> 9 ReLU network that predicts the log10
// force error of a pair's M2L at orders 2..10.
//
// Features of a pair (source A, target B, d = z_B - z_A):
//   a = max(r_A/|d|, 1e-6), b = max(r_B/|d|, 1e-6)
//   f0 = ln(a + b) (the MAC ratio of App. C), f1 = ln a, f2 = ln b,
//   f3..f6 = ln max(|M_A^(j)| / (|M_A,0| r_A^j), 1e-6), j = 1..4,
//   f7..f8 = the same for M_B, j = 1..2,  f9 = ln min(n_A, 1024),
//   f10 = ln min(n_B, 1024),
//   f11 = ln max(g_AB / T_B, 1e-12), g_AB = |M_A,0|/|d|^2 and T_B the sum of
//         g over the M2L lists of B and of all its ancestors,
// with |M^(j)|^2 = sum_{|m|=j} j!/m! M_m^2 (Frobenius norm of the rank-j
// symmetric tensor; a ratio with a zero denominator counts as 0).
// Label of a pair at order p: log10 max(e_p, 1e-12), e_p the error of the
// force of the pair's order-p M2L + L2P (Eqs. M2L, L2P) at up to 64 target
// particles of B (all when n_B <= 64, else sorted positions
// b_B + floor(j n_B/64)) against the direct sum over A's particles, relative
// to the total force at those particles.
#include <algorithm>

#include "fmm_adaptive.h"
#include "fmm_learn.h"

namespace fmm {

// ---------------------------------------------------------------------------
// node data: shape terms of the multipole (ranks 1..4), ln count, radius
// ---------------------------------------------------------------------------
// (multipoles of FP32 plans are stored in the cell's scaled units,
// Mt_m = M_m / h^|m|: the ratio then uses r / h in place of r)
__global__ void k_node_feat(int nn, int ld, const double* __restrict__ Mn, const double* __restrict__ rad,
                            const int* __restrict__ nb, const int* __restrict__ ne, const int* __restrict__ lev,
                            int scaled, double side, float* __restrict__ nodeF) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nn) return;
    const double* M = Mn + (int64_t)c * ld;
    const double m0 = fabs(M[0]), r = scaled ? rad[c] * ldexp(1.0 / side, lev[c]) : rad[c];
    float out[8];
    double rj = 1.0;
    for (int j = 1; j <= 4; ++j) {
        rj *= r;
        double s = 0.0;
        const int b = ns_of(j - 1), e = ns_of(j);
        for (int t = b; t < e; ++t) {
            const double mult = (double)c_fact_small(j) * c_invfact[c_sym_idx[t][0]] * c_invfact[c_sym_idx[t][1]] *
                                c_invfact[c_sym_idx[t][2]];
            s += mult * M[t] * M[t];
        }
        double g = 0.0;
        if (m0 > 0.0 && r > 0.0) g = sqrt(s) / (m0 * rj);
        out[j - 1] = (float)log(g > 1e-6 ? g : 1e-6);
    }
    out[4] = logf((float)min(ne[c] - nb[c], 1024));   // counts saturate at 1024
    out[5] = (float)rad[c];
    out[6] = 0.f;           // T_c, set by the far-field estimate
    out[7] = (float)m0;     // |M_0| (the same in scaled units)
    float4* o = (float4*)(nodeF + 8 * (int64_t)c);
    o[0] = make_float4(out[0], out[1], out[2], out[3]);
    o[1] = make_float4(out[4], out[5], out[6], out[7]);
}

// far-field magnitude estimate: S_c = sum over c's M2L list of |M_A,0|/|d|^2,
// then T_c = sum of S over c and its ancestors (written to nodeF slot 6)
__global__ void k_far_sum(int nn, const int* __restrict__ off, const int* __restrict__ src,
                          const int4* __restrict__ ic, float scale, const float* __restrict__ nodeF,
                          float* __restrict__ S, float* __restrict__ K) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nn) return;
    const int4 it = ic[c];
    float acc = 0.f;
    for (int k = off[c]; k < off[c + 1]; ++k) {
        const int A = src[k];
        const int4 ia = ic[A];
        const float dx = (float)(it.x - ia.x) * scale, dy = (float)(it.y - ia.y) * scale,
                    dz = (float)(it.z - ia.z) * scale;
        acc += nodeF[8 * (int64_t)A + 7] / (dx * dx + dy * dy + dz * dz);
    }
    S[c] = acc;
    K[c] = (float)(off[c + 1] - off[c]);
}
// (also K_c = number of M2L pairs of c and its ancestors, stored as log10 max(K_c, 1))
__global__ void k_far_down(int nn, const int* __restrict__ parent, const float* __restrict__ S,
                           const float* __restrict__ K, float* __restrict__ nodeF, float* __restrict__ nodeK) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nn) return;
    float t = 0.f, kk = 0.f;
    for (int a = c; a >= 0; a = parent[a]) { t += S[a]; kk += K[a]; }
    nodeF[8 * (int64_t)c + 6] = t;
    nodeK[c] = log10f(fmaxf(kk, 1.f));
}

// M2L pair index -> its target (CSR rows expanded)
__global__ void k_pair_target(int nn, const int* __restrict__ off, int* __restrict__ ptgt) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nn) return;
    for (int k = off[c]; k < off[c + 1]; ++k) ptgt[k] = c;
}

__global__ void k_pair_features(int npair, const int* __restrict__ ptgt, const int* __restrict__ msrc,
                                const int4* __restrict__ ic, float scale, const float* __restrict__ nodeF,
                                float* __restrict__ feat) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= npair) return;
    float f[FMM_MLP_NF];
    pair_features(msrc[k], ptgt[k], ic, scale, nodeF, f);
    for (int j = 0; j < FMM_MLP_NF; ++j) feat[(int64_t)k * FMM_MLP_NF + j] = f[j];
}

// ---------------------------------------------------------------------------
// FP64 labels, one warp per pair
// ---------------------------------------------------------------------------
// Full symmetric D_k(r), |k| <= p (Eq. traceless grad), by the recurrence
//   |r|^2 D_k = -[(2k_i - 1) r_i D_{k-e_i} + sum_{j != i} 2 k_j r_j D_{k-e_j}
//                + (k_i - 1)^2 D_{k-2e_i} + sum_{j != i} k_j (k_j - 1) D_{k-2e_j}],
// i the first axis with k_i > 0; lanes split each rank.
static __device__ void dtensor_warp(int p, const double r[3], double* D, int lane) {
    const double r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2], ir2 = 1.0 / r2;
    if (lane == 0) D[0] = 1.0 / sqrt(r2);
    __syncwarp();
    for (int j = 1; j <= p; ++j) {
        const int base = ns_of(j - 1), cnt = (j + 1) * (j + 2) / 2;
        for (int t = lane; t < cnt; t += 32) {
            const int s = base + t;
            const int k[3] = {c_sym_idx[s][0], c_sym_idx[s][1], c_sym_idx[s][2]};
            const int i = k[0] > 0 ? 0 : (k[1] > 0 ? 1 : 2);
            double acc = 0.0;
            for (int a = 0; a < 3; ++a) {
                if (k[a] == 0) continue;
                int km[3] = {k[0], k[1], k[2]};
                km[a] -= 1;
                acc += (a == i ? 2.0 * k[a] - 1.0 : 2.0 * k[a]) * r[a] * D[pos_sym(km[0], km[1], km[2])];
                if (k[a] >= 2) {
                    km[a] -= 1;
                    acc += (a == i ? (double)(k[a] - 1) * (k[a] - 1) : (double)k[a] * (k[a] - 1)) *
                           D[pos_sym(km[0], km[1], km[2])];
                }
            }
            D[s] = -acc * ir2;
        }
        __syncwarp();
    }
}

constexpr int LBL_P = 10;
constexpr int LBL_NS = 286;   // ns(10)

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32)
k_pair_labels(int npair, const int* __restrict__ ptgt, const int* __restrict__ msrc, const double* __restrict__ zc,
              const int* __restrict__ nb, const int* __restrict__ ne, const double* __restrict__ xs,
              const double* __restrict__ ys, const double* __restrict__ zs, const double* __restrict__ qs,
              const double* __restrict__ Mn, int ld, const double* __restrict__ atx,
              const double* __restrict__ aty, const double* __restrict__ atz, double* __restrict__ lab) {
    __shared__ double sM[WARPS][LBL_NS], sD[WARPS][LBL_NS], sL[WARPS][LBL_NS];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int k = blockIdx.x * WARPS + w;
    if (k >= npair) return;
    const int A = msrc[k], B = ptgt[k];
    const double d[3] = {zc[3 * B] - zc[3 * A], zc[3 * B + 1] - zc[3 * A + 1], zc[3 * B + 2] - zc[3 * A + 2]};
    for (int s = lane; s < LBL_NS; s += 32)
        sM[w][s] = Mn[(int64_t)A * ld + s] * c_invfact[c_sym_idx[s][0]] * c_invfact[c_sym_idx[s][1]] *
                   c_invfact[c_sym_idx[s][2]];
    dtensor_warp(LBL_P, d, sD[w], lane);
    // targets of this lane (two at most) and their exact field
    const int bB = nb[B], nB = ne[B] - nb[B];
    const int ny = nB <= 64 ? nB : 64;
    double rb[2][3], g[2][3];
    bool act[2];
    double tot = 0.0;   // squared total force at this lane's targets
    for (int u = 0; u < 2; ++u) {
        const int j = lane + 32 * u;
        act[u] = j < ny;
        g[u][0] = g[u][1] = g[u][2] = 0.0;
        rb[u][0] = rb[u][1] = rb[u][2] = 0.0;
        if (!act[u]) continue;
        const int sp = bB + (nB <= 64 ? j : (int)((int64_t)j * nB / 64));
        tot += atx[sp] * atx[sp] + aty[sp] * aty[sp] + atz[sp] * atz[sp];
        const double y[3] = {xs[sp], ys[sp], zs[sp]};
        for (int c = 0; c < 3; ++c) rb[u][c] = y[c] - zc[3 * B + c];
        for (int a = nb[A]; a < ne[A]; ++a) {
            const double dx = xs[a] - y[0], dy = ys[a] - y[1], dz = zs[a] - y[2];
            const double r2 = dx * dx + dy * dy + dz * dz;
            const double ir = 1.0 / sqrt(r2), ir3 = ir * ir * ir;
            g[u][0] += qs[a] * dx * ir3;
            g[u][1] += qs[a] * dy * ir3;
            g[u][2] += qs[a] * dz * ir3;
        }
    }
    const double den = warp_sum(tot);
    for (int p = 2; p <= LBL_P; ++p) {
        __syncwarp();
        // Eq. M2L at order p: L_n = sum_{|m| <= p-|n|} M_m/m! D_{n+m}
        for (int n = lane; n < ns_of(p); n += 32) {
            const int nx = c_sym_idx[n][0], ny2 = c_sym_idx[n][1], nz = c_sym_idx[n][2];
            const int mcount = ns_of(p - nx - ny2 - nz);
            double v = 0.0;
            for (int m = 0; m < mcount; ++m)
                v += sM[w][m] * sD[w][pos_sym(nx + c_sym_idx[m][0], ny2 + c_sym_idx[m][1], nz + c_sym_idx[m][2])];
            sL[w][n] = v;
        }
        __syncwarp();
        // Eq. L2P gradient at order p: dPhi/dx_i = sum_{|k| <= p-1} rb^k/k! L_{k+e_i}
        double num = 0.0;
        for (int u = 0; u < 2; ++u) {
            if (!act[u]) continue;
            double px[LBL_P + 1], py[LBL_P + 1], pz[LBL_P + 1];
            px[0] = py[0] = pz[0] = 1.0;
            for (int e = 1; e < p; ++e) {
                px[e] = px[e - 1] * rb[u][0] / e;
                py[e] = py[e - 1] * rb[u][1] / e;
                pz[e] = pz[e - 1] * rb[u][2] / e;
            }
            double gx = 0.0, gy = 0.0, gz = 0.0;
            const int nk = ns_of(p - 1);
            for (int s = 0; s < nk; ++s) {
                const int kx = c_sym_idx[s][0], ky = c_sym_idx[s][1], kz = c_sym_idx[s][2];
                const double wgt = px[kx] * py[ky] * pz[kz];
                gx += wgt * sL[w][pos_sym(kx + 1, ky, kz)];
                gy += wgt * sL[w][pos_sym(kx, ky + 1, kz)];
                gz += wgt * sL[w][pos_sym(kx, ky, kz + 1)];
            }
            num += (gx - g[u][0]) * (gx - g[u][0]) + (gy - g[u][1]) * (gy - g[u][1]) +
                   (gz - g[u][2]) * (gz - g[u][2]);
        }
        num = warp_sum(num);
        if (lane == 0) {
            const double e = den > 0.0 ? sqrt(num / den) : 0.0;
            lab[(int64_t)k * FMM_MLP_NOUT + (p - 2)] = log10(e > 1e-12 ? e : 1e-12);
        }
    }
}

// ---------------------------------------------------------------------------
// FP32 trainer
// ---------------------------------------------------------------------------
// Feature means and standard deviations (FP64 sums): every block sums the
// rows blockIdx.x 32 + r, += 32 gridDim.x (thread r 12 + f: row r, feature f,
// so a block reads 384 consecutive floats), k_mlp_moments adds the blocks' sums
// in block order.
__global__ void __launch_bounds__(32 * FMM_MLP_NF)
k_mlp_moments_part(int64_t n, const float* __restrict__ feat, double* __restrict__ part) {
    __shared__ double s1[32][FMM_MLP_NF], s2[32][FMM_MLP_NF];
    const int r = threadIdx.x / FMM_MLP_NF, f = threadIdx.x % FMM_MLP_NF;
    double a = 0.0, b = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * 32 + r; i < n; i += (int64_t)gridDim.x * 32) {
        const double v = feat[i * FMM_MLP_NF + f];
        a += v;
        b += v * v;
    }
    s1[r][f] = a;
    s2[r][f] = b;
    __syncthreads();
    if (r == 0) {
        for (int k = 1; k < 32; ++k) { a += s1[k][f]; b += s2[k][f]; }
        part[(blockIdx.x * FMM_MLP_NF + f) * 2] = a;
        part[(blockIdx.x * FMM_MLP_NF + f) * 2 + 1] = b;
    }
}
__global__ void k_mlp_moments(int64_t n, int nblk, const double* __restrict__ part, float* __restrict__ mu,
                              float* __restrict__ sd) {
    const int f = threadIdx.x;
    if (f >= FMM_MLP_NF) return;
    double s1 = 0.0, s2 = 0.0;
    for (int k = 0; k < nblk; ++k) { s1 += part[(k * FMM_MLP_NF + f) * 2]; s2 += part[(k * FMM_MLP_NF + f) * 2 + 1]; }
    const double m = s1 / (double)n;
    const double var = s2 / (double)n - m * m;
    const double s = var > 0.0 ? sqrt(var) : 0.0;
    mu[f] = (float)m;
    sd[f] = s > 1e-6 ? (float)s : 1.0f;
}

// One training step is two launches: k_mlp_step (forward, backward and each
// block's share of the parameter gradient) and k_mlp_update (gradient summed
// over the blocks, Adam).
//
// Bound: a step is 6 flops per parameter and sample (60 MFLOP for a batch of
// 1024: 2 us of one SM's worth on every SM) and follows the one before, so
// its time is the latency of the chain of layers.  Groups of 8 samples per
// block spread a batch of 1024 over 128 blocks; weights and activations sit in
// shared memory, a thread computes two units of one sample (the 8 lanes of a
// quarter-warp share the unit: weights are broadcasts, activation rows padded
// to 68 floats have no bank conflicts), and the gradient of the 64 x 64 layers
// is 4 x 4 per thread in registers over all groups of the block.  Sums run
// in a fixed order.  Measured, batches of 1024 of 65,536 samples, two passes:
// one thread per sample and one thread per parameter over the batch took
// 335 us a step, these two
// launches, the second overlapping the first's start, 17.6 us.
constexpr int MLP_SPB = 8;       // samples per group
constexpr int MLP_HP = 68;       // activation row pitch
constexpr int MLP_MAXBLK = 304;  // blocks of a step (two per SM)
constexpr int MLP_PARP = (FMM_MLP_NPAR + 31) / 32 * 32;   // pitch of the blocks' gradients
struct MlpSmem {
    float P[(FMM_MLP_NPAR + 3) / 4 * 4];
    float H[3][MLP_SPB][MLP_HP], G[3][MLP_SPB][MLP_HP];
    float Z[MLP_SPB][FMM_MLP_NF], Y[MLP_SPB][FMM_MLP_NOUT];
    float red[4];
};

// one 64-unit ReLU layer: units u0 and u0 + 32 of sample s
__device__ __forceinline__ void mlp_layer(const float* W, const float* b, const float* h, int u0, float* out) {
    float a0 = b[u0], a1 = b[u0 + 32];
#pragma unroll
    for (int j = 0; j < FMM_MLP_H; j += 4) {
        const float4 x = *(const float4*)(h + j), w0 = *(const float4*)(W + u0 * FMM_MLP_H + j),
                     w1 = *(const float4*)(W + (u0 + 32) * FMM_MLP_H + j);
        a0 = fmaf(w0.x, x.x, a0); a1 = fmaf(w1.x, x.x, a1);
        a0 = fmaf(w0.y, x.y, a0); a1 = fmaf(w1.y, x.y, a1);
        a0 = fmaf(w0.z, x.z, a0); a1 = fmaf(w1.z, x.z, a1);
        a0 = fmaf(w0.w, x.w, a0); a1 = fmaf(w1.w, x.w, a1);
    }
    out[u0] = fmaxf(a0, 0.f);
    out[u0 + 32] = fmaxf(a1, 0.f);
}
// gradient at the layer's input, masked by the input's ReLU: (W^T g)_j [h_j > 0]
__device__ __forceinline__ void mlp_back(const float* W, const float* g, const float* h, int j0, float* out) {
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int u = 0; u < FMM_MLP_H; u += 4) {
        const float4 x = *(const float4*)(g + u);
        const float* w = W + u * FMM_MLP_H + j0;
        a0 = fmaf(w[0], x.x, a0);               a1 = fmaf(w[32], x.x, a1);
        a0 = fmaf(w[FMM_MLP_H], x.y, a0);       a1 = fmaf(w[FMM_MLP_H + 32], x.y, a1);
        a0 = fmaf(w[2 * FMM_MLP_H], x.z, a0);   a1 = fmaf(w[2 * FMM_MLP_H + 32], x.z, a1);
        a0 = fmaf(w[3 * FMM_MLP_H], x.w, a0);   a1 = fmaf(w[3 * FMM_MLP_H + 32], x.w, a1);
    }
    out[j0] = h[j0] > 0.f ? a0 : 0.f;
    out[j0 + 32] = h[j0 + 32] > 0.f ? a1 : 0.f;
}
// 4 x 4 block of dW += g x^T
__device__ __forceinline__ void mlp_outer(const float* g, const float* x, float (&d)[16]) {
    const float4 gv = *(const float4*)g, xv = *(const float4*)x;
    const float ga[4] = {gv.x, gv.y, gv.z, gv.w}, xa[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) d[4 * i + j] = fmaf(ga[i], xa[j], d[4 * i + j]);
}

// Forward and backward of the batch rows order[0..nb); loss: mean over the
// batch and the 9 outputs of (y - t)^2.  Block b takes the groups b, b + gridDim.x,
// ..., and writes its gradient (blob order) to part[b] and its loss to lossp[b].
// prm is what the step before writes while this kernel may already run: it is no
// __restrict__ pointer, so that its loads are ordinary ones, which the wait orders
// (a read-only load takes its data as unchanged for the whole kernel, and may be
// moved ahead of the wait); likewise part and lossp in k_mlp_update.
__global__ void __launch_bounds__(256)
k_mlp_step(int nb, int64_t n, const int* __restrict__ order, const float* __restrict__ feat,
           const float* __restrict__ lab, const float* prm, const float* __restrict__ mu,
           const float* __restrict__ sd, float* part, float* lossp) {
    extern __shared__ __align__(16) unsigned char raw[];
    MlpSmem& S = *reinterpret_cast<MlpSmem*>(raw);
    const int tid = threadIdx.x, s = tid & 7, u0 = tid >> 3;
    // the group's normalised features; an index outside the data contributes nothing (below)
    auto load_z = [&](int base) {
        if (tid < MLP_SPB * FMM_MLP_NF) {
            const int r = tid / FMM_MLP_NF, f = tid % FMM_MLP_NF;
            float z = 0.f;
            if (base + r < nb) {
                int64_t i = order ? order[base + r] : base + r;
                if (i < 0 || i >= n) i = 0;
                z = (feat[i * FMM_MLP_NF + f] - mu[f]) / sd[f];
            }
            S.Z[r][f] = z;
        }
    };
    // what does not depend on the step before runs beside it: the first group's
    // features; everything after waits for the parameters
    load_z(blockIdx.x * MLP_SPB);
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();   // after the wait: the update that starts now finds the last one done
    // parameters by 16-byte loads, all in flight at once (the scratch is padded)
    {
        constexpr int NV = (FMM_MLP_NPAR + 3) / 4, PER = (NV + 255) / 256;
        float4 v[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (tid + 256 * k < NV) v[k] = ((const float4*)prm)[tid + 256 * k];
#pragma unroll
        for (int k = 0; k < PER; ++k)
            if (tid + 256 * k < NV) ((float4*)S.P)[tid + 256 * k] = v[k];
    }
    const MlpView P(S.P);
    float d2[16], d3[16], d1[3], d4[3], db = 0.f, sq = 0.f;
#pragma unroll
    for (int k = 0; k < 16; ++k) d2[k] = d3[k] = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) d1[k] = d4[k] = 0.f;
    const float gscale = 2.0f / ((float)nb * FMM_MLP_NOUT);
    const int ngrp = (nb + MLP_SPB - 1) / MLP_SPB;
    for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x) {
        const int base = grp * MLP_SPB;
        if (grp != (int)blockIdx.x) {
            __syncthreads();
            load_z(base);
        }
        __syncthreads();
        {
            float a0 = P.b1[u0], a1 = P.b1[u0 + 32];
#pragma unroll
            for (int f = 0; f < FMM_MLP_NF; ++f) {
                a0 = fmaf(P.W1[u0 * FMM_MLP_NF + f], S.Z[s][f], a0);
                a1 = fmaf(P.W1[(u0 + 32) * FMM_MLP_NF + f], S.Z[s][f], a1);
            }
            S.H[0][s][u0] = fmaxf(a0, 0.f);
            S.H[0][s][u0 + 32] = fmaxf(a1, 0.f);
        }
        __syncthreads();
        mlp_layer(P.W2, P.b2, S.H[0][s], u0, S.H[1][s]);
        __syncthreads();
        mlp_layer(P.W3, P.b3, S.H[1][s], u0, S.H[2][s]);
        __syncthreads();
        if (u0 < FMM_MLP_NOUT) {
            float a = P.b4[u0];
#pragma unroll
            for (int j = 0; j < FMM_MLP_H; j += 4) {
                const float4 x = *(const float4*)&S.H[2][s][j], w = *(const float4*)(P.W4 + u0 * FMM_MLP_H + j);
                a = fmaf(w.x, x.x, a); a = fmaf(w.y, x.y, a); a = fmaf(w.z, x.z, a); a = fmaf(w.w, x.w, a);
            }
            float r = 0.f;
            if (base + s < nb) {
                const int64_t i = order ? order[base + s] : base + s;
                if (i >= 0 && i < n) r = a - lab[i * FMM_MLP_NOUT + u0];
            }
            sq = fmaf(r, r, sq);
            S.Y[s][u0] = gscale * r;   // dL/dy
        }
        __syncthreads();
        {
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int k = 0; k < FMM_MLP_NOUT; ++k) {
                a0 = fmaf(P.W4[k * FMM_MLP_H + u0], S.Y[s][k], a0);
                a1 = fmaf(P.W4[k * FMM_MLP_H + u0 + 32], S.Y[s][k], a1);
            }
            S.G[2][s][u0] = S.H[2][s][u0] > 0.f ? a0 : 0.f;
            S.G[2][s][u0 + 32] = S.H[2][s][u0 + 32] > 0.f ? a1 : 0.f;
        }
        __syncthreads();
        mlp_back(P.W3, S.G[2][s], S.H[1][s], u0, S.G[1][s]);
        __syncthreads();
        mlp_back(P.W2, S.G[1][s], S.H[0][s], u0, S.G[0][s]);
        __syncthreads();
        // dW_l[u][j] = sum_s G_l[s][u] X_l[s][j], db_l[u] = sum_s G_l[s][u]
#pragma unroll 2
        for (int r = 0; r < MLP_SPB; ++r) {
            mlp_outer(&S.G[1][r][4 * (tid >> 4)], &S.H[0][r][4 * (tid & 15)], d2);
            mlp_outer(&S.G[2][r][4 * (tid >> 4)], &S.H[1][r][4 * (tid & 15)], d3);
            const float g1 = S.G[0][r][tid >> 2];
#pragma unroll
            for (int k = 0; k < 3; ++k) d1[k] = fmaf(g1, S.Z[r][3 * (tid & 3) + k], d1[k]);
            const float h3 = S.H[2][r][tid & 63];
#pragma unroll
            for (int k = 0; k < 3; ++k)
                if ((tid >> 6) + 4 * k < FMM_MLP_NOUT) d4[k] = fmaf(S.Y[r][(tid >> 6) + 4 * k], h3, d4[k]);
            if (tid < 192) db += S.G[tid >> 6][r][tid & 63];
            else if (tid < 192 + FMM_MLP_NOUT) db += S.Y[r][tid - 192];
        }
    }
    float* o = part + (int64_t)blockIdx.x * MLP_PARP;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int at = (4 * (tid >> 4) + i) * FMM_MLP_H + 4 * (tid & 15);
        *(float4*)(o + MLP_W2 + at) = make_float4(d2[4 * i], d2[4 * i + 1], d2[4 * i + 2], d2[4 * i + 3]);
        *(float4*)(o + MLP_W3 + at) = make_float4(d3[4 * i], d3[4 * i + 1], d3[4 * i + 2], d3[4 * i + 3]);
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        o[MLP_W1 + (tid >> 2) * FMM_MLP_NF + 3 * (tid & 3) + k] = d1[k];
        if ((tid >> 6) + 4 * k < FMM_MLP_NOUT) o[MLP_W4 + ((tid >> 6) + 4 * k) * FMM_MLP_H + (tid & 63)] = d4[k];
    }
    if (tid < 192) o[(tid < 64 ? MLP_B1 : tid < 128 ? MLP_B2 : MLP_B3) + (tid & 63)] = db;
    else if (tid < 192 + FMM_MLP_NOUT) o[MLP_B4 + tid - 192] = db;
    // the 72 threads that hold squares: warps 0..2
    if (tid < 96) {
#pragma unroll
        for (int q = 16; q; q >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, q);
        if ((tid & 31) == 0) S.red[tid >> 5] = sq;
    }
    __syncthreads();
    if (tid == 0) lossp[blockIdx.x] = (S.red[0] + S.red[1] + S.red[2]) / ((float)nb * FMM_MLP_NOUT);
}
static_assert(MLP_W2 % 4 == 0 && MLP_W3 % 4 == 0 && MLP_W4 % 4 == 0 && MLP_PARP % 4 == 0, "16-byte rows");
static_assert(FMM_MLP_NF == 12 && FMM_MLP_NOUT == 9 && FMM_MLP_H == 64, "thread layout of k_mlp_step");

// Gradient summed over the blocks of k_mlp_step (8 interleaved partial sums per
// parameter, added in order), the loss added to *loss; then, with m, Adam:
// m = b1 m + (1-b1) g, v = b2 v + (1-b2) g^2,
// theta -= lr (m/(1-b1^t)) / (sqrt(v/(1-b2^t)) + eps); without m, g to grad.
__global__ void __launch_bounds__(256)
k_mlp_update(int nblk, const float* part, const float* lossp, float* loss, float* grad, float* prm, float* m, float* v,
             float lr, float b1, float b2, float eps, float c1, float c2) {
    __shared__ float sg[8][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, t = blockIdx.x * 32 + lane;
    float a = 0.f, m0 = 0.f, v0 = 0.f, p0 = 0.f;
    // the state is the last update's, done before this step's kernel let this one start
    const bool adam = m && w == 0 && t < FMM_MLP_NPAR;
    if (adam) { m0 = m[t]; v0 = v[t]; p0 = prm[t]; }
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
#pragma unroll 16
    for (int b = w; b < nblk; b += 8) a += part[(int64_t)b * MLP_PARP + t];   // t < MLP_PARP
    sg[w][lane] = a;
    __syncthreads();
    if (blockIdx.x == 0 && w == 1) {   // the loss, 32 interleaved sums in order
        float l = 0.f;
        for (int b = lane; b < nblk; b += 32) l += lossp[b];
        for (int o = 16; o; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
        if (lane == 0) *loss += l;
    }
    if (w != 0 || t >= FMM_MLP_NPAR) return;
    float g = sg[0][lane];
#pragma unroll
    for (int k = 1; k < 8; ++k) g += sg[k][lane];
    if (!m) { grad[t] = g; return; }
    const float mm = b1 * m0 + (1.f - b1) * g;
    const float vv = b2 * v0 + (1.f - b2) * g * g;
    m[t] = mm;
    v[t] = vv;
    prm[t] = p0 - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
int ad_node_features(AdState* a, cudaStream_t s) {
    if (a->nn <= 0) return 0;
    k_node_feat<<<(a->nn + 255) / 256, 256, 0, s>>>(a->nn, a->nc, a->M, a->rad, a->nb, a->ne, a->lev,
                                                    a->pos32 ? 1 : 0, a->side, a->nodeF);
    count_launch();
    return 0;
}

int ad_pair_targets_launch(int nn, int npair, const int* off, int* ptgt, cudaStream_t s) {
    if (npair <= 0 || nn <= 0) return 0;
    k_pair_target<<<(nn + 255) / 256, 256, 0, s>>>(nn, off, ptgt);
    count_launch();
    return 0;
}

__global__ void k_iota(int n, int* __restrict__ a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) a[i] = i;
}
int ad_iota(int n, int* a, cudaStream_t s) {
    if (n <= 0) return 0;
    k_iota<<<(n + 255) / 256, 256, 0, s>>>(n, a);
    count_launch();
    return 0;
}

__global__ void k_order_keys(int n, const signed char* __restrict__ porder, uint32_t* __restrict__ key) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) key[k] = (uint32_t)(unsigned char)porder[k];
}
int ad_order_keys(int n, const signed char* porder, uint32_t* key, cudaStream_t s) {
    if (n <= 0) return 0;
    k_order_keys<<<(n + 255) / 256, 256, 0, s>>>(n, porder, key);
    count_launch();
    return 0;
}

// pairs sorted by order (stable, so targets stay ascending inside an order):
// bsrc = their sources, bcnt[q * nn + t] = pairs of target t at order q,
// from the segment boundaries of the key (q, t)
__global__ void k_bucket_csr(int n, int nn, const uint32_t* __restrict__ key, const int* __restrict__ val,
                             const int* __restrict__ ptgt, const int* __restrict__ msrc, int* __restrict__ bsrc,
                             int* __restrict__ bcnt) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int k = val[i];
    bsrc[i] = msrc[k];
    const int64_t kk = (int64_t)key[i] * nn + ptgt[k];
    const bool first = i == 0 || ((int64_t)key[i - 1] * nn + ptgt[val[i - 1]]) != kk;
    const bool last = i == n - 1 || ((int64_t)key[i + 1] * nn + ptgt[val[i + 1]]) != kk;
    if (first) atomicAdd(&bcnt[kk], -i);
    if (last) atomicAdd(&bcnt[kk], i + 1);
}
int ad_bucket_csr(int n, int nn, const uint32_t* key, const int* val, const int* ptgt, const int* msrc, int* bsrc,
                  int* bcnt, cudaStream_t s) {
    if (n <= 0) return 0;
    k_bucket_csr<<<(n + 255) / 256, 256, 0, s>>>(n, nn, key, val, ptgt, msrc, bsrc, bcnt);
    count_launch();
    return 0;
}

int ad_far_estimate(AdState* a, cudaStream_t s) {
    if (a->nn <= 0) return 0;
    k_far_sum<<<(a->nn + 255) / 256, 256, 0, s>>>(a->nn, a->moff, a->msrc, a->ic, a->scale32, a->nodeF, a->fsum,
                                                  a->fsum + a->nn);
    k_far_down<<<(a->nn + 255) / 256, 256, 0, s>>>(a->nn, a->parent, a->fsum, a->fsum + a->nn, a->nodeF, a->nodeK);
    count_launch();
    count_launch();
    return 0;
}

int ad_pair_features(AdState* a, float* feat, cudaStream_t s) {
    if (a->nm2l <= 0) return 0;
    k_pair_features<<<(a->nm2l + 255) / 256, 256, 0, s>>>(a->nm2l, a->ptgt, a->msrc, a->ic, a->scale32, a->nodeF,
                                                          feat);
    count_launch();
    return 0;
}

int ad_pair_labels(AdState* a, double* lab, const double* atx, const double* aty, const double* atz, cudaStream_t s) {
    if (a->nm2l <= 0) return 0;
    constexpr int W = 4;
    k_pair_labels<W><<<(a->nm2l + W - 1) / W, W * 32, 0, s>>>(a->nm2l, a->ptgt, a->msrc, a->zc, a->nb, a->ne, a->xs,
                                                             a->ys, a->zs, a->qs, a->M, a->nc, atx, aty, atz, lab);
    count_launch();
    return 0;
}

// Device scratch of the trainer in one allocation: blob, Adam's m and v, the
// gradient, losses, the blocks' gradients and losses, the moments' partial sums.
struct MlpScratch {
    unsigned char* base = nullptr;
    float *blob, *m, *v, *grad, *loss, *part, *lossp;
    double* mom;
    bool alloc(int epochs, int nblk) {
        size_t at = 0;
        auto take = [&](size_t bytes) { const size_t o = at; at += (bytes + 255) / 256 * 256; return o; };
        const size_t o_blob = take(FMM_MLP_NBLOB * 4), o_m = take(FMM_MLP_NPAR * 4), o_v = take(FMM_MLP_NPAR * 4),
                     o_grad = take(FMM_MLP_NPAR * 4), o_loss = take((size_t)(epochs > 0 ? epochs : 1) * 4),
                     o_part = take((size_t)nblk * MLP_PARP * 4), o_lossp = take((size_t)nblk * 4),
                     o_mom = take((size_t)MLP_MAXBLK * FMM_MLP_NF * 2 * 8);
        if (cudaMalloc(&base, at) != cudaSuccess) { base = nullptr; return false; }
        blob = (float*)(base + o_blob); m = (float*)(base + o_m); v = (float*)(base + o_v);
        grad = (float*)(base + o_grad); loss = (float*)(base + o_loss); part = (float*)(base + o_part);
        lossp = (float*)(base + o_lossp); mom = (double*)(base + o_mom);
        return true;
    }
    ~MlpScratch() { cudaFree(base); }
};

// blocks of a step over nb samples
static int mlp_blocks(int64_t nb) {
    return (int)std::max<int64_t>(1, std::min<int64_t>((nb + MLP_SPB - 1) / MLP_SPB, MLP_MAXBLK));
}

// A launch that may begin before the one ahead of it in the stream has ended;
// the kernel waits for it where it says so.  Each of a step's kernels waits for
// the whole of its predecessor before it reads or writes anything that one of
// them writes, so any two steps are ordered.  The first step (first) begins
// after everything before it: it reads the moments ahead of its wait.
template <typename... KA, typename... A>
static void launch_chained(bool first, void (*k)(KA...), unsigned grid, unsigned block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = first ? 0 : 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(block);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, KA(args)...);
    count_launch();
}

// One step over nb samples (rows order[0..nb) or 0..nb): forward, backward and
// the blocks' gradients in S.part, their losses in S.lossp.
static int mlp_batch(const MlpScratch& S, bool first, int nb, int64_t ntot, const int* order, const float* feat,
                     const float* lab, cudaStream_t s) {
    const int nblk = mlp_blocks(nb);
    launch_chained(first, k_mlp_step, nblk, 256, sizeof(MlpSmem), s, nb, ntot, order, feat, lab, S.blob + FMM_MLP_OFF_PAR,
                   S.blob + FMM_MLP_OFF_MU, S.blob + FMM_MLP_OFF_SD, S.part, S.lossp);
    return nblk;
}

static bool mlp_step_ready() {
    return cudaFuncSetAttribute(k_mlp_step, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MlpSmem)) ==
           cudaSuccess;
}

int mlp_grad_host(const float* blob, int64_t n, const float* feat, const float* lab, float* loss_out, float* grad_out,
                  cudaStream_t s) {
    MlpScratch S;
    if (!mlp_step_ready()) return -2;
    if (!S.alloc(1, mlp_blocks(n))) return -3;
    cudaMemcpyAsync(S.blob, blob, FMM_MLP_NBLOB * 4, cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(S.loss, 0, 4, s);
    const int nblk = mlp_batch(S, true, (int)n, n, nullptr, feat, lab, s);
    launch_chained(false, k_mlp_update, MLP_PARP / 32, 256, 0, s, nblk, S.part, S.lossp, S.loss, S.grad, nullptr, nullptr,
                   nullptr, 0.f, 0.f, 0.f, 0.f, 1.f, 1.f);
    cudaMemcpyAsync(grad_out, S.grad, FMM_MLP_NPAR * 4, cudaMemcpyDeviceToHost, s);
    cudaMemcpyAsync(loss_out, S.loss, 4, cudaMemcpyDeviceToHost, s);
    return cudaStreamSynchronize(s) == cudaSuccess ? 0 : -2;
}

int mlp_train_host(float* blob, int64_t n, const float* feat, const float* lab, const int* order, int epochs,
                   int batch, float lr, int fit_moments, float* loss_out, cudaStream_t s) {
    const int B = batch;
    const int nbatch = (int)((n + B - 1) / B);
    MlpScratch S;
    if (!mlp_step_ready()) return -2;
    if (!S.alloc(epochs, mlp_blocks(std::min<int64_t>(B, n)))) return -3;
    cudaMemcpyAsync(S.blob, blob, FMM_MLP_NBLOB * 4, cudaMemcpyHostToDevice, s);
    cudaMemsetAsync(S.m, 0, FMM_MLP_NPAR * 4, s);
    cudaMemsetAsync(S.v, 0, FMM_MLP_NPAR * 4, s);
    cudaMemsetAsync(S.loss, 0, (size_t)(epochs > 0 ? epochs : 1) * 4, s);
    if (fit_moments) {
        // 128 rows per block up to two blocks per SM
        const int nblk = (int)std::max<int64_t>(1, std::min<int64_t>((n + 127) / 128, MLP_MAXBLK));
        k_mlp_moments_part<<<nblk, 32 * FMM_MLP_NF, 0, s>>>(n, feat, S.mom);
        k_mlp_moments<<<1, 32, 0, s>>>(n, nblk, S.mom, S.blob + FMM_MLP_OFF_MU, S.blob + FMM_MLP_OFF_SD);
        count_launch();
        count_launch();
    }
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    int64_t t = 0;
    for (int e = 0; e < epochs; ++e) {
        for (int bi = 0; bi < nbatch; ++bi) {
            const int64_t r0 = (int64_t)bi * B;
            const int nb = (int)((n - r0) < B ? (n - r0) : B);
            ++t;
            const int nblk = mlp_batch(S, t == 1, nb, n, order + r0, feat, lab, s);
            const float c1 = (float)(1.0 - pow((double)b1, (double)t));
            const float c2 = (float)(1.0 - pow((double)b2, (double)t));
            launch_chained(false, k_mlp_update, MLP_PARP / 32, 256, 0, s, nblk, S.part, S.lossp, S.loss + e, nullptr,
                           S.blob + FMM_MLP_OFF_PAR, S.m, S.v, lr, b1, b2, eps, c1, c2);
        }
    }
    cudaMemcpyAsync(blob, S.blob, FMM_MLP_NBLOB * 4, cudaMemcpyDeviceToHost, s);
    if (loss_out && epochs > 0) cudaMemcpyAsync(loss_out, S.loss, (size_t)epochs * 4, cudaMemcpyDeviceToHost, s);
    const int rc = cudaStreamSynchronize(s) == cudaSuccess ? 0 : -2;
    if (loss_out)
        for (int e = 0; e < epochs; ++e) loss_out[e] /= (float)nbatch;   // mean batch loss of the epoch
    return rc;
}

}  // namespace fmm
