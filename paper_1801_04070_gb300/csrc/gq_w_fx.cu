// gq_w_fx.cu -- Stage 5b: List 3 far multipoles at the point targets (M2P) and to
// the QBX centres (M2QBXL) in 64-bit fixed point (gq_fix.cuh).
//
// A far box d of half-width rho is at least 3 rho from the target or centre
// (|v| = rho/|z| <= 1/3), and its multipoles are held as A_k = A'_k S 2^ceil(k/2),
// |A'_k| < 1.5 (gq_mfix), so every factor has a known range:
//   points   Phi = A_0 log|z| + 2 S v H_1,  H_k = A'_k + (k even ? 2v : v) H_{k+1},
//            |H| < 4: one complex product an order (60 cycles of a warp against
//            four FP64 multiply-adds, 260);
//   centres  G_m = sum_k C(m+k-1, k-1) A_k v^k - A_0/m as in gq_m2l_fx.cu, with
//            a_k = A'_k (2^e v)^k, e the largest power with |2^e v| <= 1, and one
//            constant table per e; then Q_m += (-r/y)^m G_m.  A pair's rounding is
//            2^-56 S (|r/y| / (1 - sqrt 2/2^e))^m, and |r/y| <= 1 - 3|v| keeps that
//            factor below 1.  One FP64 multiply-add pair a (k, m) becomes six
//            32 x 32 + 64 bit ones (24 cycles against 130).
// Measured: M2P at 0.86 M targets, p = 15: 1.33 -> 0.42 ms; M2QBXL at 0.29 M
// centres, p = 30, q = 7: 4.37 -> 1.23 ms.
#include <math.h>

#include <map>
#include <mutex>
#include <vector>

#include "gq_eval.cuh"

namespace {

constexpr int kP1 = GQ_MAX_PFMM + 1;
constexpr int kWFxE = 6;           // tables for e = 1 .. 6 (a larger e uses the last)

// Multipoles in fixed point at their box's exponent E: A_k = A'_k 2^(E - 1022 + ceil(k/2)),
// |Re A'_k|, |Im A'_k| < 1 with 58 bits behind the point; a warp per box, lane k an order.
__global__ void k_mfix(int nbox, int P1, const double2 *__restrict__ M, longlong2 *__restrict__ Mf,
                       int *__restrict__ Ef) {
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, k = threadIdx.x & 31;
    if (b >= nbox) return;
    const bool act = k < P1;
    const double2 A = act ? M[(size_t)b * P1 + k] : make_double2(0.0, 0.0);
    const int e = max(fx_expo1(A.x), fx_expo1(A.y));
    const int kc = (k + 1) / 2;
    const int E = __reduce_max_sync(0xffffffffu, e ? e - kc : -1000);
    const bool bad = __any_sync(0xffffffffu, e == 0x7ff);
    if (act) {
        Mf[(size_t)b * P1 + k] = make_longlong2(fx_from_double(A.x, E + kc) >> 4, fx_from_double(A.y, E + kc) >> 4);
    }
    if (k == 0) Ef[b] = bad ? kFxNaNExp : E;
}

// log|z| of |z|^2 = n2 (its bits): relative to 1 while that fits the fixed point (64),
// else to rho = 2^(erho - 1023) and plus log rho, which rounds at 2^-53 log rho also
// where |z| is near 1.
__device__ __forceinline__ double fx_log_abs(uint64_t nb, int erho, const long long *hl, const int *tj) {
    const int er = abs(fx_expo(nb) - 1023) <= 160 ? 1023 : 2 * erho - 1023;
    return fma((double)fx_log_half(nb, er, hl, tj), 0x1p-57, (er - 1023) * 0.34657359027997264);
}

__global__ void __launch_bounds__(128) k_w_points_fx(EvalView E, int npt, const int *__restrict__ pt_owner,
                                                     const double2 *__restrict__ M, const longlong2 *__restrict__ Mf,
                                                     const int *__restrict__ Ef, double *__restrict__ pot) {
    __shared__ long long hl[kFxLogJ];
    __shared__ int tj[kFxLogJ];
    for (int i = threadIdx.x; i < kFxLogJ; i += blockDim.x) {
        hl[i] = E.fxlog->hl[i];
        tj[i] = E.fxlog->t[i];
    }
    __syncthreads();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= npt) return;
    const int b = pt_owner[t];
    const int beg = E.loff[3][b], end = E.loff[3][b + 1];
    if (beg == end) return;
    const int P = E.P, P1 = P + 1;
    const double2 tz = E.sp_xy[t];
    double acc = 0.0;
    for (int i = beg; i < end; ++i) {
        const int d = E.lidx[3][i], l = E.blev[d];
        const double2 zd = box_centre(E.R, l, E.bix[d], E.biy[d]);
        const double zx = tz.x - zd.x, zy = tz.y - zd.y;
        const uint64_t nb = fx_bits(fma(zx, zx, zy * zy)), rb = fx_bits(box_rho(E.R, l));
        gfx x, y, ny;
        fx_ratio(zx, zy, nb, fx_bal((long long)(fx_mant(rb) << 9)), fx_expo(rb), x, y, ny);
        // 2v
        const gfx x2 = fx_bal((((long long)x.h << 32) + x.l) * 2 + 1), y2 = fx_bal((((long long)y.h << 32) + y.l) * 2 + 1);
        const gfx ny2{-y2.h, -y2.l};
        const longlong2 *A = Mf + (size_t)d * P1;
        long long hr = A[P].x, hi = A[P].y, re, im;
        int k = P - 1;
        if (k >= 1 && (k & 1)) {   // down to an even order
            fx_cmul30(fx_split30(hr), fx_split30(hi), x, y, ny, re, im);
            hr = re + A[k].x;
            hi = im + A[k].y;
            --k;
        }
        for (; k >= 2; k -= 2) {
            const longlong2 A2 = A[k], A1 = A[k - 1];
            fx_cmul30(fx_split30(hr), fx_split30(hi), x2, y2, ny2, re, im);
            hr = re + A2.x;
            hi = im + A2.y;
            fx_cmul30(fx_split30(hr), fx_split30(hi), x, y, ny, re, im);
            hr = re + A1.x;
            hi = im + A1.y;
        }
        fx_cmul30(fx_split30(hr), fx_split30(hi), x2, y2, ny2, re, im);
        double h = (double)re;
        const double s = fx_scale(h, Ef[d] + 1 - 58);
        acc += fma(h, s, M[(size_t)d * P1].x * fx_log_abs(nb, fx_expo(rb), hl, tj));
    }
    pot[t] += acc;
}

// c_mk of table e (1 .. kWFxE) at ((e - 1) kP1 + k) (kWFxMaxQ + 1) + m; the powers of two
// of its rows: G_m = 2^em S sum
struct WFxTables {
    const int2 *c = nullptr;
    const int *em = nullptr;       // [kWFxE][kWFxMaxQ + 1]
};

// Thread per centre (centres of a box share their far boxes and so, mostly, e).
template <int QQ>
__global__ void __launch_bounds__(128) k_w_centres_fx(EvalView E, int nc, const int *__restrict__ owner,
                                                      const double2 *__restrict__ M, const longlong2 *__restrict__ Mf,
                                                      const int *__restrict__ Ef, WFxTables W, double2 *__restrict__ Qout) {
    __shared__ long long hl[kFxLogJ];
    __shared__ int tj[kFxLogJ];
    for (int i = threadIdx.x; i < kFxLogJ; i += blockDim.x) {
        hl[i] = E.fxlog->hl[i];
        tj[i] = E.fxlog->t[i];
    }
    __syncthreads();
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const int b = owner[c];
    const int beg = E.loff[3][b], end = E.loff[3][b + 1];
    if (beg == end) return;
    const int P = E.P, P1 = P + 1;
    const double2 cz = E.sc_xy[c];
    const uint64_t rcb = fx_bits(E.sc_r[c]);
    double2 acc[QQ + 1];
#pragma unroll
    for (int m = 0; m <= QQ; ++m) acc[m] = make_double2(0.0, 0.0);
    for (int i = beg; i < end; ++i) {
        const int d = E.lidx[3][i], l = E.blev[d];
        const double2 zd = box_centre(E.R, l, E.bix[d], E.biy[d]);
        const double yx = cz.x - zd.x, yy = cz.y - zd.y;
        const uint64_t nb = fx_bits(fma(yx, yx, yy * yy)), rb = fx_bits(box_rho(E.R, l));
        const int erho = fx_expo(rb);
        // |v|^2 <= 2^(2 erho - en), en the exponent of |y|^2: 2^e |v| <= 1
        const int e = max(1, min(kWFxE, (fx_expo(nb) - 1023 - 2 * (erho - 1023)) >> 1));
        gfx x, y, ny;
        fx_ratio(yx, yy, nb, fx_bal((long long)(fx_mant(rb) << 9)), erho + e, x, y, ny);   // 2^e v
        long long hr[QQ + 1], hi[QQ + 1], mr[QQ + 1], mi[QQ + 1];
#pragma unroll
        for (int m = 0; m <= QQ; ++m) {
            hr[m] = hi[m] = 0;
            mr[m] = mi[m] = 1ll << 31;
        }
        const longlong2 *A = Mf + (size_t)d * P1;
        const int2 *ct = W.c + (size_t)(e - 1) * kP1 * (kWFxMaxQ + 1);
        long long pr = 1ll << 60, pi = 0;   // (2^e v)^k [60]
        for (int k = 0; k < P1; ++k, ct += kWFxMaxQ + 1) {
            const longlong2 a4 = A[k];
            gfx ar, ai;
            if (k == 0) {
                ar = fx_bal(a4.x);
                ai = fx_bal(a4.y);
            } else {
                long long re, im;
                fx_cmul30(fx_split30(pr), fx_split30(pi), x, y, ny, re, im);
                pr = re;
                pi = im;
                const gfx px = fx_bal(pr * 4 | 1), py = fx_bal(pi * 4 | 1);
                fx_cmul30(fx_split30(a4.x), fx_split30(a4.y), px, py, gfx{-py.h, -py.l}, re, im);
                ar = fx_bal(re);
                ai = fx_bal(im);
            }
#pragma unroll
            for (int m = 0; m <= QQ; ++m) {
                const int2 cc = __ldg(ct + m);
                hr[m] = fx_mw(ar.h, cc.x, hr[m]);
                mr[m] = fx_mw(ar.h, cc.y, fx_mw(ar.l, cc.x, mr[m]));
                hi[m] = fx_mw(ai.h, cc.x, hi[m]);
                mi[m] = fx_mw(ai.h, cc.y, fx_mw(ai.l, cc.x, mi[m]));
            }
        }
        // G_m / (S 2^em) [62] = the upper sum [56] and the middle one 32 bits below it
        const int es = Ef[d] + 1;
        const int *em = W.em + (e - 1) * (kWFxMaxQ + 1);
        gfx ux, uy, nuy;   // -r/y
        fx_ratio(-yx, -yy, nb, fx_bal((long long)(fx_mant(rcb) << 9)), fx_expo(rcb), ux, uy, nuy);
        pr = 1ll << 60;
        pi = 0;
#pragma unroll
        for (int m = 0; m <= QQ; ++m) {
            const long long gr = fx_shl(hr[m], 6) + (mr[m] >> 26), gi = fx_shl(hi[m], 6) + (mi[m] >> 26);
            const int e = es + em[m] - (m ? 60 : 62);   // the scale's exponent
            if (m == 0) {
                double x = (double)gr, y = (double)gi;
                const double sx = fx_scale(x, e), sy = fx_scale(y, e);
                acc[0].x += fma(x, sx, M[(size_t)d * P1].x * fx_log_abs(nb, erho, hl, tj));
                acc[0].y = fma(y, sy, acc[0].y);
            } else {
                long long re, im;
                fx_cmul30(fx_split30(pr), fx_split30(pi), ux, uy, nuy, re, im);   // (-r/y)^m
                pr = re;
                pi = im;
                const gfx gx = fx_bal(gr | 1), gy = fx_bal(gi | 1);
                fx_cmul30(fx_split30(pr), fx_split30(pi), gx, gy, gfx{-gy.h, -gy.l}, re, im);
                double x = (double)re, y = (double)im;
                const double sx = fx_scale(x, e), sy = fx_scale(y, e);
                acc[m].x = fma(x, sx, acc[m].x);
                acc[m].y = fma(y, sy, acc[m].y);
            }
        }
    }
    double2 *dst = Qout + (size_t)c * (QQ + 1);
#pragma unroll
    for (int m = 0; m <= QQ; ++m) dst[m] = cadd(dst[m], acc[m]);
}

// Built once per device, kept for the life of the process (about 16 KB).
const WFxTables &tables(int dev) {
    static std::mutex mu;
    static std::map<int, WFxTables> per_dev;
    std::lock_guard<std::mutex> lk(mu);
    auto it = per_dev.find(dev);
    if (it != per_dev.end()) return it->second;
    constexpr int Q1 = kWFxMaxQ + 1;
    std::vector<int2> c((size_t)kWFxE * kP1 * Q1);
    std::vector<int> em(kWFxE * Q1, 0);
    for (int e = 1; e <= kWFxE; ++e)
        for (int m = 0; m < Q1; ++m) {
            long double row[kP1], sum = 0.0L, C = 1.0L;   // C(m+k-1, k-1)
            for (int k = 0; k < kP1; ++k) {
                if (k >= 2) C = C * (m + k - 1) / (k - 1);
                row[k] = k == 0 ? (m ? -1.0L / m : 0.0L) : ldexpl(C, (k + 1) / 2 - e * k);
                sum += fabsl(row[k]);
            }
            int &x = em[(e - 1) * Q1 + m];
            while (ldexpl(sum, -x) > 0.5L) ++x;
            for (int k = 0; k < kP1; ++k) {
                const gfx g = fx_bal((long long)(ldexpl(row[k], 62 - x)) | 1);
                c[((size_t)(e - 1) * kP1 + k) * Q1 + m] = make_int2(g.h, g.l);
            }
        }
    int cur = 0;
    GQ_CUDA(cudaGetDevice(&cur));
    GQ_CUDA(cudaSetDevice(dev));
    WFxTables T;
    void *p = nullptr;
    GQ_CUDA(cudaMalloc(&p, sizeof(int2) * c.size()));
    GQ_CUDA(cudaMemcpy(p, c.data(), sizeof(int2) * c.size(), cudaMemcpyHostToDevice));
    T.c = (const int2 *)p;
    GQ_CUDA(cudaMalloc(&p, sizeof(int) * em.size()));
    GQ_CUDA(cudaMemcpy(p, em.data(), sizeof(int) * em.size(), cudaMemcpyHostToDevice));
    T.em = (const int *)p;
    GQ_CUDA(cudaSetDevice(cur));
    return per_dev.emplace(dev, T).first->second;
}

}  // namespace

void gq_w_fx_prepare(int dev) { tables(dev); }

void gq_mfix(gq_geom *g, gq_ctx *ctx, int P1, const double2 *M) {
    g->Mfx.alloc((size_t)g->nbox * P1);
    g->Efx.alloc(g->nbox);
    GQ_LAUNCH(ctx, k_mfix, gq_blocks((long long)g->nbox * 32, 256), 256, 0, g->nbox, P1, M, g->Mfx.p, g->Efx.p);
}

void gq_w_points_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double *pot) {
    GQ_LAUNCH(ctx, k_w_points_fx, gq_blocks(g->npt, 128), 128, 0, E, g->npt, (const int *)g->pt_owner, M,
              (const longlong2 *)g->Mfx, (const int *)g->Efx, pot);
}

void gq_w_centres_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double2 *Q) {
    const WFxTables W = tables(ctx->device);
    switch (E.Q) {
#define GQ_CASE(v)                                                                                                     \
    case v:                                                                                                            \
        GQ_LAUNCH(ctx, k_w_centres_fx<v>, gq_blocks(g->nc, 128), 128, 0, E, g->nc, (const int *)g->ctr_owner, M,    \
                  (const longlong2 *)g->Mfx, (const int *)g->Efx, W, Q);                                               \
        break;
        GQ_CASE(1) GQ_CASE(2) GQ_CASE(3) GQ_CASE(4) GQ_CASE(5) GQ_CASE(6) GQ_CASE(7) GQ_CASE(8) GQ_CASE(9) GQ_CASE(10)
#undef GQ_CASE
        default: throw gq_error{GQ_ERR_INVALID, "p_qbx out of range"};
    }
}
