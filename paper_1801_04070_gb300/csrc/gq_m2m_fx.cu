// gq_m2m_fx.cu -- Stage 2: M2M in 64-bit fixed point (gq_fix.cuh).
//
// With A_k = A'_k S 2^ceil(k/2) (S a power of two over the four children) the
// quadrant matrices T_q[m][k] of k_m2m_t become T'_q[m][k] = T_q[m][k]
// 2^(ceil(k/2) - ceil(m/2)), |T'| <= 1 and sum_k |T'_q[m][k]| <= 0.8, so a parent's
// A'_m is a sum of known range: one complex multiply-add of twelve 32 x 32 + 64 bit
// multiply-adds (48 cycles of a warp) in place of four dependent-pair FP64 ones (260),
// rounded at 2^-57 of the largest scaled coefficient.  A level of a small tree is
// one short kernel after another, which the FP64 chains of 4 (m + 1) products made
// 15 us long each.  One curve: P2M + M2M 0.19 -> 0.15 ms, its evaluation
// 0.41 -> 0.36; 1.05 M nodes, p = 19: evaluation 8.70 -> 8.44.
#include <math.h>

#include <map>
#include <mutex>
#include <vector>

#include "gq_eval.cuh"

namespace {

constexpr int kP1 = GQ_MAX_PFMM + 1;
constexpr int kM2MThreads = 128;

__device__ __forceinline__ int child_of(int4 c4, int q) { return q == 0 ? c4.x : q == 1 ? c4.y : q == 2 ? c4.z : c4.w; }

// One level: entries [lstart, lend) of `boxes` (its non-leaf boxes with sources
// below).  A block takes 128 / (P + 1) boxes, thread (box, order m); T at
// (q kP1 + k) 32 + m, so that a warp's loads are contiguous.
__global__ void __launch_bounds__(kM2MThreads) k_m2m_fx(EvalView E, const int *__restrict__ boxes, int lstart, int lend,
                                                        const int4 *__restrict__ T, double2 *__restrict__ M) {
    __shared__ int4 sA[4 * kM2MThreads];
    __shared__ int sE[kM2MThreads];
    const int P1 = E.P + 1, bpb = kM2MThreads / P1;
    const int i0 = lstart + blockIdx.x * bpb;
    if (threadIdx.x < bpb) sE[threadIdx.x] = -100000;
    __syncthreads();
    // the children's multipoles, at most four a thread, and each box's largest scaled exponent
    double2 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = threadIdx.x + r * kM2MThreads;
        v[r] = make_double2(0.0, 0.0);
        if (i >= bpb * 4 * P1) continue;
        const int bb = i / (4 * P1), rest = i - bb * 4 * P1, q = rest / P1, k = rest - q * P1;
        if (i0 + bb >= lend) continue;
        const int c = child_of(E.bchild[boxes[i0 + bb]], q);
        if (c >= 0) v[r] = M[(size_t)c * P1 + k];
        const int e = max(fx_expo1(v[r].x), fx_expo1(v[r].y));
        if (e) atomicMax(&sE[bb], e - (k + 1) / 2 + (e == 0x7ff ? 4096 : 0));   // infinite or NaN: above any scale
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = threadIdx.x + r * kM2MThreads;
        if (i >= bpb * 4 * P1) continue;
        const int bb = i / (4 * P1), k = (i - bb * 4 * P1) % P1;
        const int e = sE[bb] + (k + 1) / 2;
        const gfx x = fx_bal(fx_from_double(v[r].x, e) >> 5), y = fx_bal(fx_from_double(v[r].y, e) >> 5);   // [57]
        sA[i] = make_int4(x.h, x.l, y.h, y.l);
    }
    __syncthreads();
    const int bl = threadIdx.x / P1, m = threadIdx.x - bl * P1, ib = i0 + bl;
    if (bl >= bpb || ib >= lend) return;
    const int b = boxes[ib], Eb = sE[bl];
    long long sr = 0, si = 0;   // [60]
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int4 *A = sA + (bl * 4 + q) * P1, *Tq = T + q * kP1 * 32 + m;
        // the positive and negative products of the real part apart; rounded once a child
        long long hp = 0, hn = 0, hi = 0, mp = 1ll << 25, mn = 0, mi = 1ll << 25;
        for (int k = 0; k <= m; ++k) {
            const int4 t = __ldg(Tq + k * 32), a = A[k];
            hp = fx_mw(a.x, t.x, hp);
            mp = fx_mw(a.x, t.y, fx_mw(a.y, t.x, mp));
            hn = fx_mw(a.z, t.z, hn);
            mn = fx_mw(a.z, t.w, fx_mw(a.w, t.z, mn));
            hi = fx_mw(a.x, t.z, fx_mw(a.z, t.x, hi));
            mi = fx_mw(a.x, t.w, fx_mw(a.y, t.z, fx_mw(a.z, t.y, fx_mw(a.w, t.x, mi))));
        }
        // upper sums [54], middle ones 32 bits below
        sr += fx_shl(hp - hn, 6) + ((mp - mn) >> 26);
        si += fx_shl(hi, 6) + (mi >> 26);
    }
    double2 out;
    if (Eb > 2048) {
        out.x = out.y = __longlong_as_double(0x7ff8000000000000ll);
    } else if (Eb < -2000) {   // no multipole at all
        out.x = out.y = 0.0;
    } else {
        double x = (double)sr, y = (double)si;
        const int e = Eb + (m + 1) / 2 + 1 - 60;
        const double sx = fx_scale(x, e), sy = fx_scale(y, e);
        out = make_double2(x * sx, m ? y * sy : 0.0);
    }
    M[(size_t)b * P1 + m] = out;
}

// T'_q[m][k] [61], once per device (61 KB)
const int4 *table(int dev) {
    static std::mutex mu;
    static std::map<int, const int4 *> per_dev;
    std::lock_guard<std::mutex> lk(mu);
    auto it = per_dev.find(dev);
    if (it != per_dev.end()) return it->second;
    std::vector<int4> h(4 * kP1 * 32, make_int4(0, 0, 0, 0));
    for (int q = 0; q < 4; ++q) {
        // powers of eta = (+-1 +- i)/2
        long double pr[kP1 + 1], pi[kP1 + 1];
        const long double ex = q & 1 ? 0.5L : -0.5L, ey = q & 2 ? 0.5L : -0.5L;
        pr[0] = 1.0L;
        pi[0] = 0.0L;
        for (int j = 1; j <= kP1; ++j) {
            pr[j] = pr[j - 1] * ex - pi[j - 1] * ey;
            pi[j] = pr[j - 1] * ey + pi[j - 1] * ex;
        }
        for (int m = 0; m < kP1; ++m) {
            long double C = 1.0L;   // C(m-1, k-1)
            for (int k = 0; k <= m; ++k) {
                long double re, im;
                if (k == 0) {
                    re = m ? -pr[m] / m : 1.0L;
                    im = m ? -pi[m] / m : 0.0L;
                } else {
                    if (k >= 2) C = C * (m - k + 1) / (k - 1);
                    re = ldexpl(C * pr[m - k], -k);
                    im = ldexpl(C * pi[m - k], -k);
                }
                const int sh = (k + 1) / 2 - (m + 1) / 2 + 61;
                const gfx x = fx_bal(llroundl(ldexpl(re, sh))), y = fx_bal(llroundl(ldexpl(im, sh)));
                h[(q * kP1 + k) * 32 + m] = make_int4(x.h, x.l, y.h, y.l);
            }
        }
    }
    int cur = 0;
    GQ_CUDA(cudaGetDevice(&cur));
    GQ_CUDA(cudaSetDevice(dev));
    int4 *d = nullptr;
    GQ_CUDA(cudaMalloc(&d, sizeof(int4) * h.size()));
    GQ_CUDA(cudaMemcpy(d, h.data(), sizeof(int4) * h.size(), cudaMemcpyHostToDevice));
    GQ_CUDA(cudaSetDevice(cur));
    return per_dev.emplace(dev, d).first->second;
}

}  // namespace

void gq_m2m_fx_prepare(int dev) { table(dev); }

void gq_m2m_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, double2 *M) {
    const int4 *T = table(ctx->device);
    const int bpb = kM2MThreads / (E.P + 1);
    for (int l = g->nlev - 2; l >= 0; --l) {
        const int s = g->m2m_level_start_h[l], e = g->m2m_level_start_h[l + 1];
        if (e > s)
            GQ_LAUNCH(ctx, k_m2m_fx, gq_blocks(e - s, bpb), kM2MThreads, 0, E, (const int *)g->m2m_boxes, s, e, T, M);
    }
}
