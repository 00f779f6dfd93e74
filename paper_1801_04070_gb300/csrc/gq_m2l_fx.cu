// gq_m2l_fx.cu -- Stage 4: List 2 translations (M2L) of orders above the
// tensor-core kernel's range in 64-bit fixed point (gq_fix.cuh).
//
//   L_m += (-1)^m delta^-m G_m,  G_m = sum_k C(m+k-1, k-1) A_k delta^-k - A_0/m
//
// (m = 0: sum_k A_k delta^-k + A_0 log|y|).  |delta| >= 4 and |A_k| <= S 2^(k/2), so
// with A_k = S 2^ceil(k/2) A'_k the terms are a_k = A'_k (4/delta)^k, |a_k| < 1.5,
// and G_m = S 2^e_m sum_k c_mk a_k with constants c_mk = C(m+k-1, k-1)
// 2^(ceil(k/2) - 2k - e_m) whose sum over k is at most 1/2.  An order's rounding
// then enters the potential at 2^-56 S times (2.69/(4 - sqrt 2))^m = 1.04^m (2.69:
// the furthest point of an expansion disk), below FP64's own 2^-53 of S.
//
// A warp takes a target box, lane m an output order; two list entries at a time.
// Lane k forms a_k for both (one complex product each) into shared memory; every
// lane then sums its row: per k and entry six 32 x 32 + 64 bit multiply-adds into
// an upper and a middle sum (24 cycles) in place of two FP64 multiply-adds and
// four shuffles (150).  Measured (1.74 M list entries): p = 19 5.49 -> 1.7 ms, p = 30 (0.83 M
// entries) 3.64 -> 1.0 ms.  Error of the potentials against long double (12 curves,
// p = 30, root mean square): S 5.7e-16 -> 5.6e-16, D 5.7e-16 -> 5.3e-16.
#include <math.h>

#include <map>
#include <mutex>
#include <vector>

#include "gq_eval.cuh"

namespace {

constexpr int kP1 = GQ_MAX_PFMM + 1;

constexpr int kM2LWarps = 4;

__global__ void __launch_bounds__(kM2LWarps * 32) k_m2l_fx(EvalView E, int nwork, const int *__restrict__ work,
                                                           const double2 *__restrict__ M, const longlong2 *__restrict__ Mf,
                                                           const int *__restrict__ Ef, const int2 *__restrict__ ctab,
                                                           const int4 *__restrict__ dfix, const double2 *__restrict__ stab,
                                                           const double *__restrict__ logtab, double2 *__restrict__ L) {
    __shared__ int2 sc[kP1 * 32];
    __shared__ int4 sa[kM2LWarps][32][2];
    const int P = E.P, P1 = P + 1;
    for (int i = threadIdx.x; i < P1 * 32; i += blockDim.x) sc[i] = ctab[i];
    __syncthreads();
    const int m = threadIdx.x & 31, w = threadIdx.x >> 5;
    const bool act = m <= P;
    for (int i = blockIdx.x * kM2LWarps + w; i < nwork; i += gridDim.x * kM2LWarps) {
        const int b = work[i];
        const int beg = E.loff[1][b], end = E.loff[1][b + 1];
        if (beg == end) continue;
        const int bx = E.bix[b], by = E.biy[b];
        const double logrho = log(box_rho(E.R, E.blev[b]));
        double2 acc = make_double2(0.0, 0.0);
        for (int j = beg; j < end; j += 2) {
            int off[2], dd[2];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                const int d = dd[p] = E.lidx[1][min(j + p, end - 1)];
                off[p] = (by - E.biy[d] + 5) * 11 + (bx - E.bix[d] + 5);
                int4 a4 = make_int4(0, 0, 0, 0);
                if (act && j + p < end) {
                    const longlong2 A = Mf[(size_t)d * P1 + m];
                    const int4 D = dfix[off[p] * 32 + m];
                    long long re, im;
                    fx_cmul30(fx_split30(A.x), fx_split30(A.y), gfx{D.x, D.y}, gfx{D.z, D.w}, gfx{-D.z, -D.w}, re, im);
                    const gfx x = fx_bal(re), y = fx_bal(im);
                    a4 = make_int4(x.h, x.l, y.h, y.l);
                }
                sa[w][m][p] = a4;
            }
            __syncwarp();
            long long hr[2] = {0, 0}, hi[2] = {0, 0}, mr[2] = {1ll << 31, 1ll << 31}, mi[2] = {1ll << 31, 1ll << 31};
#pragma unroll 2
            for (int k = 0; k < P1; ++k) {
                const int2 c = sc[k * 32 + m];
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    const int4 a = sa[w][k][p];
                    hr[p] = fx_mw(a.x, c.x, hr[p]);
                    mr[p] = fx_mw(a.x, c.y, fx_mw(a.y, c.x, mr[p]));
                    hi[p] = fx_mw(a.z, c.x, hi[p]);
                    mi[p] = fx_mw(a.z, c.y, fx_mw(a.w, c.x, mi[p]));
                }
            }
            __syncwarp();
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                if (j + p >= end) break;
                double2 t = make_double2((double)(hr[p] + (int)(mr[p] >> 32)), (double)(hi[p] + (int)(mi[p] >> 32)));
                const int e = Ef[dd[p]] + 1 - 56;
                const double sx = fx_scale(t.x, e), sy = fx_scale(t.y, e);
                t.x *= sx;
                t.y *= sy;
                const double2 f = stab[off[p] * 32 + m];
                // the entry's own terms first: one rounding of the running sum an entry
                const double lg = m == 0 ? M[(size_t)dd[p] * P1].x * (logrho + logtab[off[p]]) : 0.0;
                acc.x += fma(f.x, t.x, fma(-f.y, t.y, lg));
                acc.y += fma(f.x, t.y, f.y * t.x);
            }
        }
        if (act) {
            double2 *dst = L + (size_t)b * P1 + m;
            *dst = cadd(*dst, acc);
        }
    }
}

struct M2LFxTables {
    const int2 *c = nullptr;        // [kP1][32] c_mk [62]: entry k * 32 + m
    const int4 *d = nullptr;        // [121][32] (4/delta)^k [62]
    const double2 *s = nullptr;     // [121][32] (-1)^m delta^-m 2^e_m
    const double *logd = nullptr;   // [121] log|delta|
};

template <class T>
const T *upload(const std::vector<T> &h) {
    void *p = nullptr;
    GQ_CUDA(cudaMalloc(&p, sizeof(T) * h.size()));
    GQ_CUDA(cudaMemcpy(p, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice));
    return (const T *)p;
}

int2 words(long double v) {   // v 2^62 as balanced words; an odd low word has a negative
    const gfx g = fx_bal((long long)(v * 0x1p62L) | 1);
    return make_int2(g.h, g.l);
}

// Built once per device (about 150 KB), kept for the life of the process.
const M2LFxTables &tables(int dev) {
    static std::mutex mu;
    static std::map<int, M2LFxTables> per_dev;
    std::lock_guard<std::mutex> lk(mu);
    auto it = per_dev.find(dev);
    if (it != per_dev.end()) return it->second;
    std::vector<long double> C(64 * 64, 0.0L);
    for (int n = 0; n < 64; ++n) {
        C[n * 64] = 1.0L;
        for (int k = 1; k <= n; ++k) C[n * 64 + k] = C[(n - 1) * 64 + k - 1] + (k < n ? C[(n - 1) * 64 + k] : 0.0L);
    }
    std::vector<int2> c(kP1 * 32, make_int2(0, 0));
    int em[32] = {0};
    for (int m = 0; m < kP1; ++m) {
        long double row[kP1], sum = 0.0L;
        for (int k = 0; k < kP1; ++k) {
            row[k] = k == 0 ? (m ? -1.0L / m : 0.0L)
                            : ldexpl(m ? C[(m + k - 1) * 64 + k - 1] : 1.0L, (k + 1) / 2 - 2 * k);
            sum += fabsl(row[k]);
        }
        while (ldexpl(sum, -em[m]) > 0.5L) ++em[m];
        for (int k = 0; k < kP1; ++k) c[k * 32 + m] = words(ldexpl(row[k], -em[m]));
    }
    std::vector<int4> d(121 * 32, make_int4(0, 0, 0, 0));
    std::vector<double2> s(121 * 32, make_double2(0.0, 0.0));
    std::vector<double> lg(121, 0.0);
    for (int dy = -5; dy <= 5; ++dy)
        for (int dx = -5; dx <= 5; ++dx) {
            const int off = (dy + 5) * 11 + dx + 5;
            const long double re = 2.0L * dx, im = 2.0L * dy, n2 = re * re + im * im;
            if (n2 < 16.0L) continue;   // no List 2 offset
            lg[off] = (double)(0.5L * logl(n2));
            long double pr = 1.0L, pi = 0.0L;   // (4/delta)^k
            for (int k = 0; k < kP1; ++k) {
                const int2 x = words(pr), y = words(pi);
                d[off * 32 + k] = make_int4(x.x, x.y, y.x, y.y);
                const long double f = ldexpl(k & 1 ? -1.0L : 1.0L, em[k] - 2 * k);
                s[off * 32 + k] = make_double2((double)(f * pr), (double)(f * pi));
                const long double nr = 4.0L * (pr * re + pi * im) / n2;
                pi = 4.0L * (pi * re - pr * im) / n2;
                pr = nr;
            }
        }
    int cur = 0;
    GQ_CUDA(cudaGetDevice(&cur));
    GQ_CUDA(cudaSetDevice(dev));
    M2LFxTables T;
    T.c = upload(c);
    T.d = upload(d);
    T.s = upload(s);
    T.logd = upload(lg);
    GQ_CUDA(cudaSetDevice(cur));
    return per_dev.emplace(dev, T).first->second;
}

}  // namespace

void gq_m2l_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double2 *L) {
    const M2LFxTables &T = tables(ctx->device);
    const int blocks = gq_blocks(g->n_far_boxes, kM2LWarps);
    GQ_LAUNCH(ctx, k_m2l_fx, blocks < 152 * 32 ? blocks : 152 * 32, kM2LWarps * 32, 0, E, g->n_far_boxes,
              (const int *)g->far_boxes, M, (const longlong2 *)g->Mfx, (const int *)g->Efx, T.c, T.d, T.s, T.logd, L);
}

void gq_m2l_fx_prepare(int dev) { tables(dev); }
