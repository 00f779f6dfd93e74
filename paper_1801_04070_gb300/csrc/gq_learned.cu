// gq_learned.cu -- learned order selection (an extension; the paper chooses
// orders from its error bounds, Sec. 4.1, and notes those bounds
// overestimate the error by about two orders of magnitude, Sec. 5.1).
//
// A small MLP (32 -> 64 -> 32 -> 32 -> 2, ReLU) maps per-centre geometry
// features to the predicted log10 relative QBX truncation error at p_qbx =
// q_ref and log10 relative FMM error at p_fmm = p_ref.  Training (FP32,
// mean-squared error, Adam) and inference (BF16 weights and activations,
// FP32 sums) are CUDA kernels of this file.  Deployment turns the
// predictions into one QBX order per centre and one FMM order for the tree
// using measured per-order decay rates; the bound-driven orders remain the
// fallback and the cap.
#include <cuda_bf16.h>
#include <math.h>

#include <string.h>

#include <algorithm>
#include <random>
#include <vector>

#include "gq_eval.cuh"
#include "gq_internal.cuh"

namespace {

constexpr int kT = 256;
constexpr int kNF = 32;                       // features per centre
constexpr int kDims[5] = {32, 64, 32, 32, 2};
constexpr int kLayers = 4;
// parameter offsets: W_l [out][in] then b_l [out]
__host__ __device__ constexpr int woff(int l) {
    return l == 0 ? 0 : woff(l - 1) + (l == 1 ? 32 * 64 + 64 : l == 2 ? 64 * 32 + 32 : l == 3 ? 32 * 32 + 32 : 32 * 2 + 2);
}
constexpr int kNParams = woff(kLayers);
__host__ __device__ constexpr int cdim(int l) { return l == 1 ? 64 : l == 4 ? 2 : 32; }   // kDims, for device code

// ------------------------------------------------------------------ features
// curvature at base nodes from the turning of the normal between the
// neighbouring nodes of the same panel (one-sided at the panel ends)
__global__ void k_base_curvature(int nbase, int nb, const double *__restrict__ xy, const double *__restrict__ n,
                                 float *__restrict__ kappa) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nbase) return;
    int j = i % nb;
    int a = j == 0 ? i : i - 1, b = j == nb - 1 ? i : i + 1;
    double cr = n[2 * a] * n[2 * b + 1] - n[2 * a + 1] * n[2 * b];
    double dt = n[2 * a] * n[2 * b] + n[2 * a + 1] * n[2 * b + 1];
    double ds = hypot(xy[2 * b] - xy[2 * a], xy[2 * b + 1] - xy[2 * a + 1]);
    kappa[i] = ds > 0 ? (float)(atan2(cr, dt) / ds) : 0.f;
}

// The nearest panels of one centre (not its own) among the sources of its box's
// direct lists: pd[k], pp[k] the 8 smallest distances (over r, ascending) and
// their panels.  Every source's distance in FP64, by one thread.
__device__ __noinline__ void nearest_panels_exact(const EvalView &E, const int *src_perm, int b, int nu, int panel, double2 c,
                                                  double r, float (&pd)[8], int (&pp)[8]) {
    for (int k = 0; k < 8; ++k) { pd[k] = 3.0e38f; pp[k] = -1; }
    const int lists[3] = {0, 2, 4};
    for (int L = 0; L < 3; ++L)
        for (int e = E.loff[lists[L]][b]; e < E.loff[lists[L]][b + 1]; ++e) {
            int d = E.lidx[lists[L]][e];
            for (int s = E.src_beg[d]; s < E.src_end[d]; ++s) {
                int p = src_perm[s] / nu;
                if (p == panel) continue;
                float dist = (float)(hypot(E.s_xy[s].x - c.x, E.s_xy[s].y - c.y) / r);
                int at = -1;
                for (int k = 0; k < 8; ++k) if (pp[k] == p) at = k;
                if (at >= 0) {
                    if (dist >= pd[at]) continue;
                    // move the improved entry towards the front
                    while (at > 0 && pd[at - 1] > dist) { pd[at] = pd[at - 1]; pp[at] = pp[at - 1]; --at; }
                    pd[at] = dist; pp[at] = p;
                } else if (dist < pd[7]) {
                    int k = 7;
                    while (k > 0 && pd[k - 1] > dist) { pd[k] = pd[k - 1]; pp[k] = pp[k - 1]; --k; }
                    pd[k] = dist; pp[k] = p;
                }
            }
        }
}

// Features of the centres of one box per block, a warp per centre: among the
// sources of the box's direct lists, the 8 nearest distinct panels (distance to
// their nearest source, over r, ascending) and their lengths (over the centre's
// own panel length); then the curvature times r at the base nodes k - 8 .. k + 7
// of its own panel (k its own node, clamped to the panel), signed so that positive
// means the curve bends towards the centre.
//
// An FP64 distance takes about 40 FP64 instructions, and one thread a centre
// measuring its 270 sources so took 6 ms for 131,072 centres.  Here the box's
// sources get the slots of their panels once; a warp's lanes take FP32
// distances of differences formed in FP64 (within 2^-21 of themselves of the exact
// ones), which give each panel's minimum (boxes have up to 3,000 sources, and the
// few that have were the old kernel's last threads); where the ninth panel is clear of the
// eighth, only the sources that can be the nearest of one of the 8 are measured in
// FP64, gathered so that one pass of the warp measures all of them.  Boxes with
// more sources or panels than fit, and centres without that gap, take
// nearest_panels_exact.  6.1 -> 1.8 ms, the same features.
constexpr int kFtSrc = 4096;    // sources of a box at most
constexpr int kFtSlots = 256;   // panel slots, kFtSlots / 32 a lane
constexpr int kFtCand = 64;     // gathered candidates of a centre
constexpr unsigned kFtNone = 0x7f7fffffu;   // FLT_MAX

__global__ void __launch_bounds__(kNearThreads) k_centre_features(EvalView E, const int *__restrict__ boxes, int nb, int nu,
                                                                  const int *__restrict__ ctr_perm,
                                                                  const int *__restrict__ src_perm,
                                                                  const double *__restrict__ panel_len,
                                                                  const float *__restrict__ kappa, float *__restrict__ feat) {
    constexpr int W = kNearThreads / 32, NS = kFtSlots / 32;
    __shared__ NearRanges R;
    __shared__ int wsum[W];
    __shared__ unsigned char sslot[kFtSrc];
    __shared__ int tab[kFtSlots];             // panel of a slot, -1 free
    __shared__ int over;                      // more than fits
    __shared__ unsigned smin[W][kFtSlots];
    __shared__ unsigned long long sex[W][kFtSlots];   // exact distance, then the source that has it first
    __shared__ unsigned short cand[W][kFtCand];
    const int b = boxes[blockIdx.x], lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ne = (E.loff[0][b + 1] - E.loff[0][b]) + (E.loff[2][b + 1] - E.loff[2][b]) + (E.loff[4][b + 1] - E.loff[4][b]);
    for (int i = threadIdx.x; i < kFtSlots; i += kNearThreads) tab[i] = -1;
    if (threadIdx.x == 0) over = ne > kNearRanges;
    __syncthreads();
    load_ranges(E, b, 0, min(ne, kNearRanges), R, wsum);
    const int T = R.pre[R.n];
    if (T > kFtSrc && threadIdx.x == 0) over = 1;
    __syncthreads();
    if (!over)
        for (int r = w; r < R.n; r += W)
            for (int v = R.pre[r] + lane; v < R.pre[r + 1]; v += 32) {
                const int s = R.beg[r] + (v - R.pre[r]), p = src_perm[s] / nu;
                int h = p & (kFtSlots - 1), tries = 0;
                for (; tries < kFtSlots; ++tries, h = (h + 1) & (kFtSlots - 1)) {
                    const int was = atomicCAS(&tab[h], -1, p);
                    if (was == -1 || was == p) break;
                }
                if (tries == kFtSlots) over = 1;
                sslot[v] = (unsigned char)h;
            }
    __syncthreads();
    if (over) {   // a thread per centre
        for (int c = E.ctr_beg[b] + threadIdx.x; c < E.ctr_end[b]; c += kNearThreads) {
            const int cid = ctr_perm[c], node = cid >> 1, side = cid & 1, panel = node / nb;
            const double r = E.sc_r[c], own = panel_len[panel];
            float pd[8];
            int pp[8];
            nearest_panels_exact(E, src_perm, b, nu, panel, E.sc_xy[c], r, pd, pp);
            float *f = feat + (size_t)cid * kNF;
            for (int k = 0; k < 8; ++k) {
                f[k] = pp[k] >= 0 ? fminf(pd[k], 64.f) : 64.f;
                f[8 + k] = pp[k] >= 0 ? (float)(panel_len[pp[k]] / own) : 0.f;
            }
            for (int k = 0; k < 16; ++k) {
                const int kk = min(max(node - panel * nb + k - 8, 0), nb - 1);
                f[16 + k] = (side ? -1.f : 1.f) * kappa[panel * nb + kk] * (float)r;
            }
        }
        return;
    }
    for (int c = E.ctr_beg[b] + w; c < E.ctr_end[b]; c += W) {
        const int cid = ctr_perm[c], node = cid >> 1, side = cid & 1, panel = node / nb;
        const double2 cz = E.sc_xy[c];
        const double r = E.sc_r[c];
        const float ir = (float)(1.0 / r);
        const double own = panel_len[panel];
        float d8 = 64.f, len8 = 0.f;          // lane k < 8: the k-th nearest panel's features
        bool ok = ir < 1e15f && ir > 1e-15f;   // squares within FP32's range
        if (ok) {
#pragma unroll
            for (int k = 0; k < NS; ++k) {
                smin[w][lane + 32 * k] = kFtNone;
                sex[w][lane + 32 * k] = (unsigned long long)kFtNone << 32;
            }
            __syncwarp();
            // FP32 distance of source v (r: the lane's range, moving with v)
            auto dist32 = [&](int v, int &rg) {
                while (R.pre[rg + 1] <= v) ++rg;
                const double2 y = E.s_xy[R.beg[rg] + (v - R.pre[rg])];
                const float dx = (float)(y.x - cz.x), dy = (float)(y.y - cz.y);
                return sqrtf(dx * dx + dy * dy) * ir;
            };
            for (int v = lane, rg = 0; v < T; v += 32) {
                const int sl = sslot[v];
                if (tab[sl] != panel) atomicMin(&smin[w][sl], __float_as_uint(dist32(v, rg)));
            }
            __syncwarp();
            // the eighth and ninth smallest panel minima
            unsigned x8[NS], t8 = kFtNone, t9 = kFtNone;
#pragma unroll
            for (int k = 0; k < NS; ++k) x8[k] = smin[w][lane + 32 * k];
            // the warp's smallest value, which is taken out
            auto take_min = [&]() {
                unsigned lm = x8[0];
#pragma unroll
                for (int k = 1; k < NS; ++k) lm = min(lm, x8[k]);
                const unsigned m = __reduce_min_sync(0xffffffffu, lm);
                if (m < kFtNone) {
                    const int src = __ffs(__ballot_sync(0xffffffffu, lm == m)) - 1;
                    int mine = 0;
#pragma unroll
                    for (int k = NS - 1; k >= 0; --k)
                        if (x8[k] == m) mine = k;
#pragma unroll
                    for (int k = 0; k < NS; ++k)
                        if (lane == src && k == mine) x8[k] = kFtNone;
                }
                return m;
            };
            for (int k = 0; k < 9; ++k) {
                const unsigned m = take_min();
                if (k == 7) t8 = m;
                if (k == 8) t9 = m;
            }
            const float f8 = __uint_as_float(t8), f9 = __uint_as_float(t9);
            if (t9 < kFtNone && f9 - f8 <= 0x1p-20f * f9) ok = false;
            // candidates
            int n = 0;
            for (int v0 = 0, rg = 0; v0 < T; v0 += 32) {
                const int v = v0 + lane;
                bool in = false;
                if (v < T) {
                    const unsigned ms = smin[w][sslot[v]];
                    if (ms < kFtNone && ms <= t8) {
                        const float a = dist32(v, rg);
                        in = a - __uint_as_float(ms) <= 0x1p-20f * a;
                    }
                }
                const unsigned who = __ballot_sync(0xffffffffu, in);
                const int at = n + __popc(who & ((1u << lane) - 1));
                if (in && at < kFtCand) cand[w][at] = (unsigned short)v;
                n += __popc(who);
            }
            if (n > kFtCand) ok = false;
            __syncwarp();
            if (ok) {
                for (int i = lane; i < n; i += 32) {
                    const int v = cand[w][i];
                    int rg = 0;
                    while (R.pre[rg + 1] <= v) ++rg;
                    const double2 y = E.s_xy[R.beg[rg] + (v - R.pre[rg])];
                    const float dist = (float)(hypot(y.x - cz.x, y.y - cz.y) / r);
                    atomicMin(&sex[w][sslot[v]], (unsigned long long)__float_as_uint(dist) << 32 | (unsigned)v);
                }
                __syncwarp();
                // ascending; of equal distances the panel that has it at the earlier source
                unsigned long long y8[NS];
#pragma unroll
                for (int k = 0; k < NS; ++k) y8[k] = sex[w][lane + 32 * k];
                for (int k = 0; k < 8; ++k) {
                    unsigned long long lm = y8[0];
#pragma unroll
                    for (int i = 1; i < NS; ++i) lm = min(lm, y8[i]);
                    const unsigned m = __reduce_min_sync(0xffffffffu, (unsigned)(lm >> 32));
                    if (m >= kFtNone) break;
                    const unsigned v = __reduce_min_sync(0xffffffffu, (unsigned)(lm >> 32) == m ? (unsigned)lm : 0xffffffffu);
                    const unsigned long long key = (unsigned long long)m << 32 | v;
                    const int src = __ffs(__ballot_sync(0xffffffffu, lm == key)) - 1;
                    int mine = 0;
#pragma unroll
                    for (int i = 0; i < NS; ++i)
                        if (y8[i] == key) {
                            mine = i;
                            if (lane == src) y8[i] = (unsigned long long)kFtNone << 32;
                        }
                    const int slot = __shfl_sync(0xffffffffu, lane + 32 * mine, src);
                    if (lane == k) {
                        d8 = fminf(__uint_as_float(m), 64.f);
                        len8 = (float)(panel_len[tab[slot]] / own);
                    }
                }
            }
            __syncwarp();
        }
        if (!ok) {
            float pd[8];
            int pp[8];
            if (lane == 0) nearest_panels_exact(E, src_perm, b, nu, panel, cz, r, pd, pp);
            for (int k = 0; k < 8; ++k) {
                const float dk = __shfl_sync(0xffffffffu, pd[k], 0);
                const int pk = __shfl_sync(0xffffffffu, pp[k], 0);
                if (lane == k) {
                    d8 = pk >= 0 ? fminf(dk, 64.f) : 64.f;
                    len8 = pk >= 0 ? (float)(panel_len[pk] / own) : 0.f;
                }
            }
        }
        const float l = __shfl_sync(0xffffffffu, len8, lane & 7);
        float x = lane < 8 ? d8 : l;
        if (lane >= 16) {
            int kk = node - panel * nb + lane - 24;   // window centred on the centre's own node, clamped to its panel
            kk = kk < 0 ? 0 : (kk > nb - 1 ? nb - 1 : kk);
            // interior centre (side 0) sits on the concave side when kappa > 0
            x = (side ? -1.f : 1.f) * kappa[panel * nb + kk] * (float)r;
        }
        feat[(size_t)cid * kNF + lane] = x;
    }
}

// ------------------------------------------------------------------ MLP kernels
// A training step is two launches: k_mlp_samples (gather, forward, error,
// deltas; samples are independent) and k_mlp_params (gradient and Adam;
// parameters are independent).  One launch per layer and pass (13 a step, each
// thread reading its operands from L2) took 0.35 ms a step of 1,024 samples;
// these two about 0.015 ms.  Every sum keeps its order (over inputs, outputs or
// samples, ascending, from the same start), so the trained weights are
// unchanged bit for bit.
constexpr int kSB = 8;            // samples per block of k_mlp_samples
constexpr int kPT = 128;          // weights per block of k_mlp_params
constexpr int kChunk = 64;        // samples staged at a time by k_mlp_params

// activations and deltas of a batch, per layer [B][width]
struct MlpBatch {
    float *X;                     // inputs as used (normalised when training)
    float *A[kLayers];            // layer outputs
    float *D[kLayers];            // d loss / d (layer output before ReLU)
    double *sse;                  // per block of k_mlp_samples: sum of squared errors (may be null)
};

template <int L>
__device__ __forceinline__ void mlp_forward(const float *sw, const float *in, float *out, int nb, int s0, float *gout) {
    constexpr int NI = cdim(L), NO = cdim(L + 1), LD = NI + 1;
    for (int t = threadIdx.x; t < kSB * NO; t += blockDim.x) {
        const int s = t / NO, o = t % NO;
        const float *a = in + s * NI, *w = sw + o * LD;
        float z = sw[NO * LD + o];
#pragma unroll 16
        for (int i = 0; i < NI; ++i) z = fmaf(w[i], a[i], z);
        if (L < kLayers - 1) z = fmaxf(z, 0.f);
        out[t] = z;
        if (s < nb) gout[(size_t)(s0 + s) * NO + o] = z;
    }
    __syncthreads();
}

// delta_prev = (W^T delta) relu', relu' = 1 where the layer's output is positive
template <int L>
__device__ __forceinline__ void mlp_backward(const float *sw, const float *delta, const float *aprev, float *dprev, int nb,
                                             int s0, float *gout) {
    constexpr int NI = cdim(L), NO = cdim(L + 1), LD = NI + 1;
    for (int t = threadIdx.x; t < kSB * NI; t += blockDim.x) {
        const int s = t / NI, i = t % NI;
        float g = 0.f;
#pragma unroll 16
        for (int o = 0; o < NO; ++o) g = fmaf(delta[s * NO + o], sw[o * LD + i], g);
        g = aprev[t] > 0.f ? g : 0.f;
        dprev[t] = g;
        if (s < nb) gout[(size_t)(s0 + s) * NI + i] = g;
    }
    __syncthreads();
}

// offset of layer l's weights in shared memory (rows padded by one word)
__host__ __device__ constexpr int swoff(int l) {
    return l == 0 ? 0 : swoff(l - 1) + cdim(l) * (cdim(l - 1) + 1) + cdim(l);
}

// Rows perm[s] (or row s) of X and Y, standardised when mu and sd are given.
__global__ void __launch_bounds__(256) k_mlp_samples(int B, const int *__restrict__ perm, const float *__restrict__ X,
                                                     const float *__restrict__ Y, const float *__restrict__ xmu,
                                                     const float *__restrict__ xsd, const float *__restrict__ ymu,
                                                     const float *__restrict__ ysd, const float *__restrict__ w, MlpBatch M) {
    __shared__ float sw[swoff(kLayers)];
    __shared__ float x[kSB * 32], a0[kSB * 64], a1[kSB * 32], a2[kSB * 32], a3[kSB * 2], d3[kSB * 2], da[kSB * 64], db[kSB * 64];
    __shared__ float se[kSB * 2];
    const int s0 = blockIdx.x * kSB, nb = min(kSB, B - s0);
#pragma unroll
    for (int l = 0; l < kLayers; ++l) {
        const int ni = cdim(l), no = cdim(l + 1);
        for (int t = threadIdx.x; t < no * ni; t += blockDim.x) sw[swoff(l) + t / ni * (ni + 1) + t % ni] = w[woff(l) + t];
        for (int t = threadIdx.x; t < no; t += blockDim.x) sw[swoff(l) + no * (ni + 1) + t] = w[woff(l) + no * ni + t];
    }
    for (int t = threadIdx.x; t < kSB * kNF; t += blockDim.x) {
        const int s = t / kNF, c = t % kNF;
        float v = 0.f;
        if (s < nb) {
            v = X[(size_t)(perm ? perm[s0 + s] : s0 + s) * kNF + c];
            if (xmu) v = (v - xmu[c]) / xsd[c];
            M.X[(size_t)(s0 + s) * kNF + c] = v;
        }
        x[t] = v;
    }
    __syncthreads();
    mlp_forward<0>(sw + swoff(0), x, a0, nb, s0, M.A[0]);
    mlp_forward<1>(sw + swoff(1), a0, a1, nb, s0, M.A[1]);
    mlp_forward<2>(sw + swoff(2), a1, a2, nb, s0, M.A[2]);
    mlp_forward<3>(sw + swoff(3), a2, a3, nb, s0, M.A[3]);
    // delta = 2 (Yhat - Y) / (2 B)
    if (threadIdx.x < kSB * 2) {
        const int t = threadIdx.x, s = t / 2, c = t % 2;
        float d = 0.f;
        if (s < nb) {
            float y = Y[(size_t)(perm ? perm[s0 + s] : s0 + s) * 2 + c];
            if (ymu) y = (y - ymu[c]) / ysd[c];
            d = a3[t] - y;
            M.D[3][(size_t)(s0 + s) * 2 + c] = 2.f * d / (float)(B * 2);
        }
        d3[t] = 2.f * d / (float)(B * 2);
        se[t] = d * d;
    }
    __syncthreads();
    if (M.sse && threadIdx.x == 0) {
        double e = 0.0;
        for (int t = 0; t < kSB * 2; ++t) e += se[t];
        M.sse[blockIdx.x] = e;
    }
    mlp_backward<3>(sw + swoff(3), d3, a2, da, nb, s0, M.D[2]);
    mlp_backward<2>(sw + swoff(2), da, a1, db, nb, s0, M.D[1]);
    mlp_backward<1>(sw + swoff(1), db, a0, da, nb, s0, M.D[0]);
}

struct AdamStep {
    float *w, *m, *v;             // null w: gradient only
    float lr, b1, b2, c1, c2;
};

// Gradient of kPT weights of layer L (whole output rows) and of their rows'
// biases, summed over the samples in order; the samples' activations and deltas
// come through shared memory, a chunk ahead of the sums.
template <int L>
__device__ __forceinline__ void mlp_params_layer(int blk, int B, const MlpBatch &M, float *__restrict__ grad,
                                                 const AdamStep &ad, float (*sA)[kChunk * 64], float (*sD)[kChunk * 4]) {
    constexpr int NI = cdim(L), NO = cdim(L + 1), R = kPT / NI < NO ? kPT / NI : NO;
    const float *Ain = L == 0 ? M.X : M.A[L > 0 ? L - 1 : 0], *D = M.D[L];
    const int o0 = blk * R, tid = threadIdx.x;
    auto stage = [&](int s0, int buf) {
        const int n = min(kChunk, B - s0);
        for (int t = tid; t < n * NI / 4; t += blockDim.x) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(&sA[buf][t * 4]);
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(Ain + (size_t)s0 * NI + t * 4));
        }
        for (int t = tid; t < n * R; t += blockDim.x) {
            const unsigned dst = (unsigned)__cvta_generic_to_shared(&sD[buf][t]);
            asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(D + (size_t)(s0 + t / R) * NO + o0 + t % R));
        }
        asm volatile("cp.async.commit_group;");
    };
    // thread: a weight (r, i), or a bias of row r
    const bool isw = tid < R * NI, isb = tid >= kPT && tid < kPT + R;
    const int r = isw ? tid / NI : tid - kPT, i = tid % NI;
    float g = 0.f;
    stage(0, 0);
    for (int s0 = 0, buf = 0; s0 < B; s0 += kChunk, buf ^= 1) {
        if (s0 + kChunk < B) {
            stage(s0 + kChunk, buf ^ 1);
            asm volatile("cp.async.wait_group 1;");
        } else {
            asm volatile("cp.async.wait_group 0;");
        }
        __syncthreads();
        const int n = min(kChunk, B - s0);
        if (isw) {
#pragma unroll 16
            for (int s = 0; s < n; ++s) g = fmaf(sD[buf][s * R + r], sA[buf][s * NI + i], g);
        } else if (isb) {
#pragma unroll 16
            for (int s = 0; s < n; ++s) g += sD[buf][s * R + r];
        }
        __syncthreads();
    }
    if (!isw && !isb) return;
    const int p = woff(L) + (isw ? (o0 + r) * NI + i : NO * NI + o0 + r);
    grad[p] = g;
    if (ad.w) {
        const float mi = ad.b1 * ad.m[p] + (1.f - ad.b1) * g, vi = ad.b2 * ad.v[p] + (1.f - ad.b2) * g * g;
        ad.m[p] = mi;
        ad.v[p] = vi;
        ad.w[p] -= ad.lr * (mi / ad.c1) / (sqrtf(vi / ad.c2) + 1e-8f);
    }
}

__host__ __device__ constexpr int mlp_param_blocks(int l) { return (cdim(l) * cdim(l + 1) + kPT - 1) / kPT; }

__global__ void __launch_bounds__(kPT + 32) k_mlp_params(int B, MlpBatch M, float *__restrict__ grad, AdamStep ad) {
    __shared__ __align__(16) float sA[2][kChunk * 64];
    __shared__ float sD[2][kChunk * 4];
    constexpr int b1 = mlp_param_blocks(0), b2 = b1 + mlp_param_blocks(1), b3 = b2 + mlp_param_blocks(2);
    const int b = blockIdx.x;
    if (b < b1) mlp_params_layer<0>(b, B, M, grad, ad, sA, sD);
    else if (b < b2) mlp_params_layer<1>(b - b1, B, M, grad, ad, sA, sD);
    else if (b < b3) mlp_params_layer<2>(b - b2, B, M, grad, ad, sA, sD);
    else mlp_params_layer<3>(b - b3, B, M, grad, ad, sA, sD);
}

// Column sums and sums of squares of X [n][d] (d = 32 or 2) in FP64: per block
// part[block][2 d], then k_col_stats makes mean and deviation (1 where it is
// below 1e-6) of the blocks' parts, in order.
constexpr int kStatBlocks = 64;
__global__ void __launch_bounds__(256) k_col_sums(int n, int d, const float *__restrict__ X, double *__restrict__ part) {
    __shared__ double s1[256], s2[256];
    const int c = threadIdx.x % d, rows = blockDim.x / d;
    double a = 0.0, b = 0.0;
    for (int i = blockIdx.x * rows + threadIdx.x / d; i < n; i += gridDim.x * rows) {
        const double x = X[(size_t)i * d + c];
        a += x;
        b += x * x;
    }
    s1[threadIdx.x] = a;
    s2[threadIdx.x] = b;
    __syncthreads();
    if (threadIdx.x < d) {
        for (int r = 1; r < rows; ++r) {
            a += s1[r * d + c];
            b += s2[r * d + c];
        }
        part[(size_t)blockIdx.x * 2 * d + c] = a;
        part[(size_t)blockIdx.x * 2 * d + d + c] = b;
    }
}

__global__ void k_col_stats(int n, int d, const double *__restrict__ part, float *__restrict__ mu, float *__restrict__ sd) {
    const int c = threadIdx.x;
    if (c >= d) return;
    double s = 0.0, q = 0.0;
    for (int b = 0; b < kStatBlocks; ++b) {
        s += part[(size_t)b * 2 * d + c];
        q += part[(size_t)b * 2 * d + d + c];
    }
    const double m = s / n;
    double v = sqrt(fmax(q / n - m * m, 0.0));
    if (v < 1e-6) v = 1.0;
    mu[c] = (float)m;
    sd[c] = (float)v;
}

// BF16 inference on the tensor cores (mma.sync m16n8k16, BF16 inputs, FP32
// accumulators): a warp takes 16 samples through all four layers.  Inputs
// are normalised and rounded to BF16; each layer's accumulators start at its
// BF16 bias, and after ReLU the accumulator fragments of output columns
// 16k ... 16k+15 are, packed to BF16 pairs, exactly the A fragment of the
// next layer's k-block k (row g = lane / 4 and g + 8, columns 2 (lane % 4)
// and + 1, + 8), so activations never leave registers.  The last layer
// (2 outputs) fills the first two columns of one 8-wide tile; its weight
// rows 2 ... 7 read as zero.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<uint32_t *>(&v);
}

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// one dense layer for a warp's 16 rows: NIN inputs as NIN/16 A fragments,
// NOUT outputs as NOUT/8 accumulator tiles; W [nout_real][NIN] BF16 in
// shared memory, rows >= nout_real read as zero
template <int NIN, int NOUT>
__device__ __forceinline__ void mma_layer(const uint32_t (&A)[NIN / 16][4], const __nv_bfloat16 *W,
                                          const __nv_bfloat16 *bias, int nout_real, float (&C)[NOUT / 8][4]) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int j = 0; j < NOUT / 8; ++j) {
        const int c0 = 8 * j + 2 * t;
        const float bl = c0 < nout_real ? __bfloat162float(bias[c0]) : 0.f;
        const float bh = c0 + 1 < nout_real ? __bfloat162float(bias[c0 + 1]) : 0.f;
        C[j][0] = bl; C[j][1] = bh; C[j][2] = bl; C[j][3] = bh;
        const int n = 8 * j + g;
#pragma unroll
        for (int kb = 0; kb < NIN / 16; ++kb) {
            uint32_t b0 = 0, b1 = 0;
            if (n < nout_real) {
                const __nv_bfloat16 *wr = W + n * NIN + 16 * kb + 2 * t;
                b0 = *reinterpret_cast<const uint32_t *>(wr);
                b1 = *reinterpret_cast<const uint32_t *>(wr + 8);
            }
            mma_bf16_16816(C[j], A[kb], b0, b1);
        }
    }
}

// accumulators of a hidden layer -> ReLU -> BF16 A fragments of the next layer
template <int NOUT>
__device__ __forceinline__ void relu_to_frags(const float (&C)[NOUT / 8][4], uint32_t (&A)[NOUT / 16][4]) {
#pragma unroll
    for (int kb = 0; kb < NOUT / 16; ++kb) {
        A[kb][0] = pack_bf16x2(fmaxf(C[2 * kb][0], 0.f), fmaxf(C[2 * kb][1], 0.f));
        A[kb][1] = pack_bf16x2(fmaxf(C[2 * kb][2], 0.f), fmaxf(C[2 * kb][3], 0.f));
        A[kb][2] = pack_bf16x2(fmaxf(C[2 * kb + 1][0], 0.f), fmaxf(C[2 * kb + 1][1], 0.f));
        A[kb][3] = pack_bf16x2(fmaxf(C[2 * kb + 1][2], 0.f), fmaxf(C[2 * kb + 1][3], 0.f));
    }
}

static_assert(kDims[0] == 32 && kDims[1] == 64 && kDims[2] == 32 && kDims[3] == 32 && kDims[4] == 2,
              "the tensor-core inference is written for 32-64-32-32-2");

__global__ void __launch_bounds__(128) k_mlp_infer_mma(int n, const float *__restrict__ X,
                                                       const __nv_bfloat16 *__restrict__ Wb,
                                                       const float *__restrict__ xmu, const float *__restrict__ xsd,
                                                       const float *__restrict__ ymu, const float *__restrict__ ysd,
                                                       float *__restrict__ Y) {
    __shared__ __align__(16) __nv_bfloat16 sw[kNParams + 8];
    for (int i = threadIdx.x; i < kNParams; i += blockDim.x) sw[i] = Wb[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int s0 = 16 * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); s0 < n; s0 += 16 * warps) {
        // input fragments: rows s0 + g, s0 + g + 8; features 16 kb + 2t (+1), + 8
        uint32_t A0[2][4];
#pragma unroll
        for (int kb = 0; kb < 2; ++kb)
#pragma unroll
            for (int h = 0; h < 2; ++h)        // column half: + 0 or + 8
#pragma unroll
                for (int r = 0; r < 2; ++r) {  // row g or g + 8
                    const int s = s0 + g + 8 * r, f = 16 * kb + 8 * h + 2 * t;
                    float lo = 0.f, hi = 0.f;
                    if (s < n) {
                        lo = (X[(size_t)s * kNF + f] - xmu[f]) / xsd[f];
                        hi = (X[(size_t)s * kNF + f + 1] - xmu[f + 1]) / xsd[f + 1];
                    }
                    A0[kb][2 * h + r] = pack_bf16x2(lo, hi);
                }
        float C1[8][4];
        mma_layer<32, 64>(A0, sw + woff(0), sw + woff(0) + 32 * 64, 64, C1);
        uint32_t A1[4][4];
        relu_to_frags<64>(C1, A1);
        float C2[4][4];
        mma_layer<64, 32>(A1, sw + woff(1), sw + woff(1) + 64 * 32, 32, C2);
        uint32_t A2[2][4];
        relu_to_frags<32>(C2, A2);
        float C3[4][4];
        mma_layer<32, 32>(A2, sw + woff(2), sw + woff(2) + 32 * 32, 32, C3);
        uint32_t A3[2][4];
        relu_to_frags<32>(C3, A3);
        float C4[1][4];
        mma_layer<32, 8>(A3, sw + woff(3), sw + woff(3) + 32 * 2, 2, C4);
        if (t == 0) {   // columns 0 and 1 of rows g and g + 8
            const int sa = s0 + g, sb = s0 + g + 8;
            if (sa < n) {
                Y[(size_t)sa * 2] = C4[0][0] * ysd[0] + ymu[0];
                Y[(size_t)sa * 2 + 1] = C4[0][1] * ysd[1] + ymu[1];
            }
            if (sb < n) {
                Y[(size_t)sb * 2] = C4[0][2] * ysd[0] + ymu[0];
                Y[(size_t)sb * 2 + 1] = C4[0][3] * ysd[1] + ymu[1];
            }
        }
    }
}

__global__ void k_to_bf16(int n, const float *__restrict__ in, __nv_bfloat16 *__restrict__ out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = __float2bfloat16(in[i]);
}

// per-centre QBX order from the predicted truncation error at q_ref; the FMM
// prediction is reduced to its maximum (the tree uses one FMM order)
__global__ void k_learned_q(int nc, const int *__restrict__ ctr_perm, const float *__restrict__ pred, double log_tol,
                            double margin, int q_ref, double qbx_slope, int q_cap, int *__restrict__ q_sorted,
                            unsigned int *__restrict__ fmm_max_bits, int *__restrict__ qmax) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= nc) return;
    int cid = ctr_perm[j];
    double yq = pred[(size_t)cid * 2], yf = pred[(size_t)cid * 2 + 1];
    int q = q_ref + (int)ceil((yq + margin - log_tol) / qbx_slope);
    q = q < 1 ? 1 : (q > q_cap ? q_cap : q);
    q_sorted[j] = q;
    atomicMax(qmax, q);
    // order-preserving map of a float to unsigned int for atomicMax
    float f = (float)yf;
    unsigned int u = __float_as_uint(f);
    u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
    atomicMax(fmm_max_bits, u);
}

}  // namespace

// ====================================================================== host side
struct gq_mlp {
    gq_ctx *ctx = nullptr;
    dbuf<float> w, m, v, g;
    dbuf<__nv_bfloat16> wb;
    dbuf<float> xmu, xsd, ymu, ysd;   // normalisation (identity until trained)
    int adam_t = 0;
    // work buffers for a batch
    int cap = 0;
    dbuf<float> Xb, A[kLayers], D[kLayers];
};

namespace {

void ensure_batch(gq_mlp *M, int B) {
    if (B <= M->cap) return;
    M->Xb.alloc((size_t)B * kNF);
    for (int l = 0; l < kLayers; ++l) {
        M->A[l].alloc((size_t)B * kDims[l + 1]);
        M->D[l].alloc((size_t)B * kDims[l + 1]);
    }
    M->cap = B;
}

// One batch: forward and backward on rows perm[0 .. B) (or the first B rows) of
// X and Y, standardised with the network's statistics when norm; the gradient
// goes to M->g, and with ad.w the Adam step is taken.  sse (may be null): one
// sum of squared errors per kSB samples.
void mlp_batch(gq_mlp *M, int B, const int *perm, const float *X, const float *Y, bool norm, double *sse, const AdamStep &ad) {
    MlpBatch b;
    b.X = M->Xb;
    for (int l = 0; l < kLayers; ++l) {
        b.A[l] = M->A[l];
        b.D[l] = M->D[l];
    }
    b.sse = sse;
    const float *null = nullptr;
    GQ_LAUNCH(M->ctx, k_mlp_samples, gq_blocks(B, kSB), 256, 0, B, perm, X, Y, norm ? (const float *)M->xmu : null,
              norm ? (const float *)M->xsd : null, norm ? (const float *)M->ymu : null, norm ? (const float *)M->ysd : null,
              (const float *)M->w, b);
    constexpr int blocks = mlp_param_blocks(0) + mlp_param_blocks(1) + mlp_param_blocks(2) + mlp_param_blocks(3);
    GQ_LAUNCH(M->ctx, k_mlp_params, blocks, kPT + 32, 0, B, b, M->g.p, ad);
}

double sum_on_host(gq_ctx *ctx, const double *dev, size_t n) {
    std::vector<double> h(n);
    GQ_CUDA(cudaMemcpyAsync(h.data(), dev, sizeof(double) * n, cudaMemcpyDeviceToHost, ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
    double s = 0;
    for (double x : h) s += x;
    return s;
}

const float *to_device(gq_ctx *ctx, const float *p, size_t n, dbuf<float> &tmp, bool is_dev) {
    if (is_dev) return p;
    tmp.alloc(n);
    GQ_CUDA(cudaMemcpyAsync(tmp.p, p, sizeof(float) * n, cudaMemcpyDefault, ctx->stream));
    return tmp.p;
}

}  // namespace

int gq_mlp_param_count() { return kNParams; }

gq_mlp *gq_mlp_new(gq_ctx *ctx, uint64_t seed) {
    gq_mlp *M = new gq_mlp;
    M->ctx = ctx;
    std::vector<float> w(kNParams, 0.f);
    std::mt19937_64 rng(seed);
    for (int l = 0; l < kLayers; ++l) {
        int nin = kDims[l], nout = kDims[l + 1];
        std::normal_distribution<float> nd(0.f, sqrtf(2.f / nin));   // He initialisation
        for (int i = 0; i < nin * nout; ++i) w[woff(l) + i] = nd(rng);
    }
    M->w.alloc(kNParams);
    M->m.alloc(kNParams);
    M->v.alloc(kNParams);
    M->g.alloc(kNParams);
    M->wb.alloc(kNParams);
    GQ_CUDA(cudaMemcpyAsync(M->w.p, w.data(), sizeof(float) * kNParams, cudaMemcpyHostToDevice, ctx->stream));
    GQ_CUDA(cudaMemsetAsync(M->m.p, 0, sizeof(float) * kNParams, ctx->stream));
    GQ_CUDA(cudaMemsetAsync(M->v.p, 0, sizeof(float) * kNParams, ctx->stream));
    std::vector<float> zero(kNF, 0.f), one(kNF, 1.f);
    M->xmu.alloc(kNF); M->xsd.alloc(kNF); M->ymu.alloc(2); M->ysd.alloc(2);
    GQ_CUDA(cudaMemcpyAsync(M->xmu.p, zero.data(), sizeof(float) * kNF, cudaMemcpyHostToDevice, ctx->stream));
    GQ_CUDA(cudaMemcpyAsync(M->xsd.p, one.data(), sizeof(float) * kNF, cudaMemcpyHostToDevice, ctx->stream));
    GQ_CUDA(cudaMemcpyAsync(M->ymu.p, zero.data(), sizeof(float) * 2, cudaMemcpyHostToDevice, ctx->stream));
    GQ_CUDA(cudaMemcpyAsync(M->ysd.p, one.data(), sizeof(float) * 2, cudaMemcpyHostToDevice, ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
    return M;
}

void gq_mlp_free(gq_mlp *M) { delete M; }
gq_ctx *gq_mlp_ctx(const gq_mlp *M) { return M->ctx; }

void gq_mlp_weights_impl(gq_mlp *M, float *get, const float *set) {
    if (set) GQ_CUDA(cudaMemcpyAsync(M->w.p, set, sizeof(float) * kNParams, cudaMemcpyDefault, M->ctx->stream));
    if (get) GQ_CUDA(cudaMemcpyAsync(get, M->w.p, sizeof(float) * kNParams, cudaMemcpyDefault, M->ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(M->ctx->stream));
}

// loss = mean squared error of the raw network on (X, Y); grad = d loss / d parameters
void gq_mlp_loss_grad_impl(gq_mlp *M, const float *X, const float *Y, int n, bool dev, float *loss, float *grad) {
    ensure_batch(M, n);
    dbuf<float> tx, ty;
    const float *Xd = to_device(M->ctx, X, (size_t)n * kNF, tx, dev), *Yd = to_device(M->ctx, Y, (size_t)n * 2, ty, dev);
    dbuf<double> sse;
    sse.alloc(gq_blocks(n, kSB));
    mlp_batch(M, n, nullptr, Xd, Yd, false, sse.p, AdamStep{});
    const double e = sum_on_host(M->ctx, sse.p, gq_blocks(n, kSB));
    if (loss) *loss = (float)(e / (2.0 * n));
    if (grad) GQ_CUDA(cudaMemcpy(grad, M->g.p, sizeof(float) * kNParams, cudaMemcpyDeviceToHost));
}

// Adam on normalised features and labels (statistics of this training set)
double gq_mlp_train_impl(gq_mlp *M, const float *X, const float *Y, int n, bool dev, int epochs, int B, float lr,
                         uint64_t seed) {
    gq_ctx *ctx = M->ctx;
    cudaStream_t st = ctx->stream;
    B = B < n ? B : n;
    ensure_batch(M, B);
    dbuf<float> tx, ty;
    const float *Xd = to_device(ctx, X, (size_t)n * kNF, tx, dev), *Yd = to_device(ctx, Y, (size_t)n * 2, ty, dev);
    // normalisation statistics of this training set (FP64 sums)
    dbuf<double> part;
    part.alloc((size_t)kStatBlocks * 2 * kNF);
    for (int k = 0; k < 2; ++k) {
        const int d = k ? 2 : kNF;
        GQ_LAUNCH(ctx, k_col_sums, kStatBlocks, 256, 0, n, d, k ? Yd : Xd, part.p);
        GQ_LAUNCH(ctx, k_col_stats, 1, 32, 0, n, d, (const double *)part, k ? M->ymu.p : M->xmu.p, k ? M->ysd.p : M->xsd.p);
    }
    dbuf<int> permall;
    permall.alloc(n);
    std::vector<int> perm(n);
    for (int i = 0; i < n; ++i) perm[i] = i;
    std::mt19937_64 rng(seed);
    const float b1 = 0.9f, b2 = 0.999f;
    const int per = gq_blocks(B, kSB);
    dbuf<double> sse;   // squared errors of the last epoch's batches
    sse.alloc((size_t)(n / B) * per);
    GQ_CUDA(cudaMemsetAsync(sse.p, 0, sizeof(double) * (n / B) * per, st));
    for (int ep = 0; ep < epochs; ++ep) {
        std::shuffle(perm.begin(), perm.end(), rng);
        GQ_CUDA(cudaMemcpyAsync(permall.p, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
        const bool last_epoch = ep == epochs - 1;
        for (int s0 = 0, k = 0; s0 + B <= n; s0 += B, ++k) {
            ++M->adam_t;
            const float c1 = 1.f - powf(b1, (float)M->adam_t), c2 = 1.f - powf(b2, (float)M->adam_t);
            mlp_batch(M, B, (const int *)permall + s0, Xd, Yd, true, last_epoch ? sse.p + (size_t)k * per : nullptr,
                      AdamStep{M->w, M->m, M->v, lr, b1, b2, c1, c2});
        }
    }
    const double last = sum_on_host(ctx, sse.p, (size_t)(n / B) * per) / (2.0 * (n / B) * B);
    GQ_CUDA(cudaStreamSynchronize(st));
    return last;   // mean squared error of the last epoch, in normalised units
}

void gq_mlp_predict_impl(gq_mlp *M, const float *X, int n, bool xdev, float *Y, bool ydev) {
    gq_ctx *ctx = M->ctx;
    dbuf<float> tx, ty;
    const float *Xd = to_device(ctx, X, (size_t)n * kNF, tx, xdev);
    float *Yd = Y;
    if (!ydev) {
        ty.alloc((size_t)n * 2);
        Yd = ty.p;
    }
    GQ_LAUNCH(ctx, k_to_bf16, gq_blocks(kNParams, kT), kT, 0, kNParams, (const float *)M->w.p, M->wb.p);
    if (n > 0) {
        const int blocks = std::min(gq_blocks(n, 64), 152 * 8);
        GQ_LAUNCH(ctx, k_mlp_infer_mma, blocks, 128, 0, n, Xd, (const __nv_bfloat16 *)M->wb.p,
                  (const float *)M->xmu.p, (const float *)M->xsd.p, (const float *)M->ymu.p, (const float *)M->ysd.p, Yd);
    }
    if (!ydev) GQ_CUDA(cudaMemcpyAsync(Y, Yd, sizeof(float) * n * 2, cudaMemcpyDeviceToHost, ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
}

void gq_centre_features_impl(gq_geom *g, float *feat_dev) {
    gq_ctx *ctx = g->ctx;
    dbuf<float> kappa;
    kappa.alloc(g->nbase);
    GQ_LAUNCH(ctx, k_base_curvature, gq_blocks(g->nbase, kT), kT, 0, g->nbase, g->nb, (const double *)g->base_xy,
              (const double *)g->base_n, kappa.p);
    if (g->n_ctr_boxes) {
        EvalView E{};
        E.src_beg = g->src_beg;
        E.src_end = g->src_end;
        E.ctr_beg = g->ctr_beg;
        E.ctr_end = g->ctr_end;
        E.s_xy = g->s_xy;
        E.sc_xy = g->sc_xy;
        E.sc_r = g->sc_r;
        for (int i = 0; i < 6; ++i) {
            E.loff[i] = g->list_off[i];
            E.lidx[i] = g->list_idx[i];
        }
        GQ_LAUNCH(ctx, k_centre_features, g->n_ctr_boxes, kNearThreads, 0, E, (const int *)g->ctr_boxes, g->nb, g->nu,
                  (const int *)g->ctr_perm, (const int *)g->src_perm, (const double *)g->panel_len, (const float *)kappa.p,
                  feat_dev);
    }
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
}

// Learned orders: per-centre q = q_ref + ceil((yq + margin - log10(eps/2)) / qbx_slope),
// p_fmm = p_ref + ceil((max yf + margin_fmm - log10(eps/2)) / fmm_slope), capped by the
// bound-driven order (its fallback).
void gq_learned_orders_impl(gq_geom *g, gq_mlp *M, double eps, double margin, double margin_fmm, int q_ref,
                            int p_ref, int q_bound, int p_bound, int *p_out, int *q_out) {
    gq_ctx *ctx = g->ctx;
    dbuf<float> feat, pred;
    feat.alloc((size_t)g->nc * kNF);
    pred.alloc((size_t)g->nc * 2);
    gq_centre_features_impl(g, feat.p);
    gq_mlp_predict_impl(M, feat.p, g->nc, true, pred.p, true);
    dbuf<unsigned int> fbits;
    dbuf<int> qmax;
    fbits.alloc(1);
    qmax.alloc(1);
    GQ_CUDA(cudaMemsetAsync(fbits.p, 0, sizeof(unsigned int), ctx->stream));
    GQ_CUDA(cudaMemsetAsync(qmax.p, 0, sizeof(int), ctx->stream));
    const bool per_centre = q_ref > 0;
    g->q_ctr.alloc(g->nc);
    double log_tol = log10(eps / 2.0);
    const double qbx_slope = 1.26, fmm_slope = 0.5;   // decades per order, measured on starfish curves
    if (g->nc)
        GQ_LAUNCH(ctx, k_learned_q, gq_blocks(g->nc, kT), kT, 0, g->nc, (const int *)g->ctr_perm, (const float *)pred.p,
                  log_tol, margin, per_centre ? q_ref : 1, qbx_slope, q_bound, g->q_ctr.p, fbits.p, qmax.p);
    unsigned int ub = 0;
    int qm = 0;
    GQ_CUDA(cudaMemcpyAsync(&ub, fbits.p, sizeof(ub), cudaMemcpyDeviceToHost, ctx->stream));
    GQ_CUDA(cudaMemcpyAsync(&qm, qmax.p, sizeof(qm), cudaMemcpyDeviceToHost, ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
    ub = (ub & 0x80000000u) ? (ub & 0x7fffffffu) : ~ub;
    float yf;
    memcpy(&yf, &ub, sizeof(yf));
    int p = p_ref + (int)ceil((yf + margin_fmm - log_tol) / fmm_slope);
    p = p < 1 ? 1 : (p > p_bound ? p_bound : p);
    g->prm.p_fmm = p;
    if (per_centre) {
        g->prm.p_qbx = qm < 1 ? 1 : qm;
        g->has_qc = true;
    }
    g->have_eval = false;
    *p_out = p;
    *q_out = g->prm.p_qbx;
}

__global__ void k_scatter_orders(int nc, const int *__restrict__ ctr_pos, const int *__restrict__ q_by_id,
                                 int *__restrict__ q_sorted, int *__restrict__ qmax) {
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    int q = q_by_id[c];
    q_sorted[ctr_pos[c]] = q;
    atomicMax(qmax, q);
}

void gq_set_centre_orders_impl(gq_geom *g, const int *q_dev) {
    gq_ctx *ctx = g->ctx;
    g->q_ctr.alloc(g->nc);
    dbuf<int> qmax;
    qmax.alloc(1);
    GQ_CUDA(cudaMemsetAsync(qmax.p, 0, sizeof(int), ctx->stream));
    if (g->nc)
        GQ_LAUNCH(ctx, k_scatter_orders, gq_blocks(g->nc, 256), 256, 0, g->nc, (const int *)g->ctr_pos, q_dev,
                  g->q_ctr.p, qmax.p);
    int qm = 0;
    GQ_CUDA(cudaMemcpyAsync(&qm, qmax.p, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
    GQ_CUDA(cudaStreamSynchronize(ctx->stream));
    g->prm.p_qbx = qm < 1 ? 1 : qm;
    g->has_qc = true;
    g->have_eval = false;
}

