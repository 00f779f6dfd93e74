// gq_near_fx.cu -- Stages 3, 5a, 6a: the direct sums to the QBX centres with the
// powers, logarithms and sums in 64-bit fixed point (gq_fix.cuh).
//
// S: Q_0 = sum q log|w|, Q_m = -(1/m) sum q (r/w)^m; D: Q_m = sum (d/w) (r/w)^m,
// w = y - c.  In FP64 this sum issues 62 FP64 instructions a pair at q = 8 and
// holds the FP64 pipe 88 % busy; here 7 are left (four a pair for w and |w|^2, the
// rest for the sums' conversions), and 1/|w|^2, r/w, log|w|, the power recurrence and
// the sums run on the integer pipes.  At q = 8 a pair costs 505 instructions of a lane
// (idle lanes of the last round included), 211 of them on the pipe of the 32 x 32 bit
// multiply-adds, which bounds the kernel: 69 % busy with 38 % of the warps resident.
// 1.05 M quadrature nodes, 142.5 M pairs, S, q = 8: 17.06 ms -> 3.4 ms;
// D on 0.14 M nodes: 2.59 -> 0.53 ms; q = 5 on one curve: 0.35 -> 0.14 ms.
//
// Formats (bits behind the binary point in brackets): u = r/w [62], t_m = q u^m
// [60] with the strengths scaled to at most 1/2, products rounded at 2^-60.
// |u| <= 1 when no source is inside the centre's disk; the loop records the
// smallest |w|^2, and a centre that meets |u| > 1 + 1/64 is summed again with the
// smallest |w| as its radius; the sums are then scaled by (r/|w|)^m.  Where that would
// raise the rounding above the terms (the sources inside are weak), they are left
// out of a third sum and their powers summed in FP64.
// Sums: 12 terms a lane (tiles of 384 sources), |t_m| < 0.65, stay below 2^63;
// the warp's sum is taken at 2^-60 (2^-55 if the lanes' sums are that large).  Error against long double sums on the nodes
// of a starfish grid (272 sources, q = 8, root mean square, in units of the
// strength scale), FP64 form -> this: Q_0 2^-46.3 -> 2^-50.9, Q_1 2^-48.7 ->
// 2^-53.0, Q_4 2^-50.9 -> 2^-52.1, Q_8 2^-50.5 -> 2^-51.5.
//
// The scale is that of the tile's own strengths.  Strengths that have none (infinite,
// NaN, exponents near the ends of the range) and centres whose terms are weak beside
// it (kFxWeak) go through near_centre_fp64 whole, with the arithmetic's own infinities
// and NaN.
#include <math.h>

#include <type_traits>

#include "gq_eval.cuh"
#include "gq_math.cuh"

namespace {

constexpr int kFxTile = 384;
constexpr int kFxWarps = kNearThreads / 32;

// a source's strength: S (h, l) [62]; D (re.h, re.l, im.h, im.l) [60], split at bit 30
template <int KERNEL> struct FxStr { typedef int2 T; };
template <> struct FxStr<GQ_D> { typedef int4 T; };

// Where a centre's terms are weak beside the largest strength of the tile (panels of
// very different length in one box), the common scale leaves them fewer bits than
// FP64's: at n sources the sum's rounding, about sqrt(n) 2^-60 of that strength, has to
// stay below 2^-53 of the sum of the terms' magnitudes, or the centre goes through
// near_centre_fp64.  The bound on that sum in units of 2^-22 of the scale is
// kFxWeak sqrt(n), half of it for S.  Errors against long double, q = 5 .. 16, one panel
// and another 2^k times longer (host build of gq_fix.cuh, root mean square): S equal to
// FP64's at 2^11, 10 times at 2^14; D at 2^8 and 2^11; the bounds cut at 2^10 and 2^7.
// Panels of one length are 28 to 160 (D 14 to 50) times above them; a tile of far
// sources alone can fall below (S with D's bound: one leaf of 8,192 sources 1.41 -> 1.70
// ms).  Cost, 64 circles with panels graded over 2^20, q = 8, D: n_max 32 2.51 ->
// 2.68 ms (all in FP64: 9.6), n_max 256 and 16 nodes a panel, where nearly all centres
// mix 2^9 and more, 5.0 -> 18.2 (17.1).
constexpr float kFxWeak = 107021.0f;   // 2^21 at 384 sources

__device__ __forceinline__ int fx_second(int2) { return 0; }
__device__ __forceinline__ int fx_second(int4 v) { return v.z; }

// -1/m
__constant__ double c_ninv[GQ_MAX_PQBX + 1] = {0.0,      -1.0,      -1.0 / 2,  -1.0 / 3,  -1.0 / 4,  -1.0 / 5,
                                               -1.0 / 6, -1.0 / 7,  -1.0 / 8,  -1.0 / 9,  -1.0 / 10, -1.0 / 11,
                                               -1.0 / 12, -1.0 / 13, -1.0 / 14, -1.0 / 15, -1.0 / 16};

// 2^(e - 1023), subnormal and infinite ends included
__device__ __forceinline__ double pow2_clamped(int e) {
    return e >= 2047 ? __longlong_as_double(0x7ff0000000000000ll)
                     : e > 0 ? __longlong_as_double((long long)e << 52)
                             : e > -52 ? __longlong_as_double(1ll << (51 + e)) : 0.0;
}

// The lane and slot that hold entry i after a warp_reduce_scatter over n values.
struct RsPlace {
    int lane, slot;
};
constexpr RsPlace rs_place(int n, int i) {
    int lane = 0;
    for (int o = 16; o > 0; o >>= 1) {
        const int h = (n + 1) / 2;
        if (i >= h) {
            lane |= o;
            i -= h;
        }
        n = h;
    }
    return RsPlace{lane, i};
}

// In FP64: the sources [v0, v1) of the loaded ranges (every warp lane takes part; with
// infinities and NaN), or the powers (no logarithms) of those whose |w|^2 has an upper
// word below nlim, added to dst (first: written).  NC orders a sweep, at most nine, so
// that their sums fit the registers and a small order's kernel spills none at the call
// (q = 4, 1.05 M nodes, evaluation 6.375 -> 6.35 ms).
constexpr unsigned kAllSources = 0xffffffffu;
template <int KERNEL, int NC>
__device__ __noinline__ void near_centre_fp64(const EvalView &E, const NearRanges &R, int v0, int v1, double2 cz, double rc,
                                              int QQ, int qc, unsigned nlim, double2 *dst, bool first) {
    const int lane = threadIdx.x & 31;
    for (int m0 = 0; m0 <= QQ; m0 += NC) {
        double2 acc[NC];
#pragma unroll
        for (int i = 0; i < NC; ++i) acc[i] = make_double2(0.0, 0.0);
        if (m0 <= qc)
            for (int v = v0 + lane, r = 0; v < v1; v += 32) {
                while (R.pre[r + 1] <= v) ++r;
                const int s = R.beg[r] + (v - R.pre[r]);
                const double2 y = E.s_xy[s];
                const double wx = y.x - cz.x, wy = y.y - cz.y, n2 = fma(wx, wx, wy * wy);
                if ((unsigned)(fx_bits(n2) >> 32) >= nlim) continue;
                const double2 st = E.str[s];
                const double inv = gq_rcp(n2);
                const double2 winv = make_double2(wx * inv, -wy * inv);
                const double2 u = make_double2(rc * winv.x, rc * winv.y);
                double2 t = KERNEL == GQ_D ? cmul(st, winv) : make_double2(st.x * u.x, st.x * u.y);   // order 0 (D) or 1
                if (m0) {   // NC = 9: t times u^8 (D: u^9)
                    double2 p = u;
                    for (int i = 0; i < 3; ++i) p = cmul(p, p);
                    t = cmul(t, p);
                    if (KERNEL == GQ_D) t = cmul(t, u);
                } else if (KERNEL != GQ_D && nlim == kAllSources) {
                    // a coincident source has log term 0
                    acc[0].x = fma(st.x, n2 == 0.0 ? 0.0 : gq_log_half(n2, E.logt), acc[0].x);
                }
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    if (KERNEL != GQ_D && i == 0 && m0 == 0) continue;
                    acc[i] = cadd(acc[i], t);
                    t = cmul(t, u);
                }
            }
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const int m = m0 + i;
            if (m > QQ) break;
            for (int o = 16; o > 0; o >>= 1)
                acc[i] = cadd(acc[i], make_double2(__shfl_xor_sync(0xffffffffu, acc[i].x, o),
                                                   __shfl_xor_sync(0xffffffffu, acc[i].y, o)));
            if (lane == 0) {
                double2 x = m <= qc ? acc[i] : make_double2(0.0, 0.0);
                if (KERNEL != GQ_D && m >= 1) x = cscale(x, c_ninv[m]);
                dst[m] = first ? x : cadd(dst[m], x);
            }
        }
    }
}

// Stage the sources [v0, v1) of the loaded ranges: positions, and strengths as
// q 2^(1022 - qe) <= 1/2 (D: each component, so that |d| <= 0.36) with qe from the
// tile's largest exponent; for S the sums of the strengths' words per warp.
// Returns qe, 0 where the strengths have no scale; ends with a barrier.  any: not all
// strengths are zero.
template <int KERNEL>
__device__ __forceinline__ int fx_stage(const EvalView &E, const NearRanges &R, int v0, int v1, double2 *sy,
                                        typename FxStr<KERNEL>::T *sq, long long *ssum, int *smax, bool &any) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int mx = 0;
    for (int r = w; r < R.n; r += kFxWarps) {   // a warp takes one range at a time
        const int p0 = R.pre[r], p1 = R.pre[r + 1];
        for (int v = max(p0, v0) + lane; v < min(p1, v1); v += 32) {
            const double2 st = E.str[R.beg[r] + (v - p0)];
            mx = max(mx, fx_expo1(st.x));
            if (KERNEL == GQ_D) mx = max(mx, fx_expo1(st.y));
        }
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) smax[w] = mx;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kFxWarps; ++k) mx = max(mx, smax[k]);
    any = mx > 0;
    if (!any) mx = 1023;
    const int qe = mx + (KERNEL == GQ_D ? 2 : 1);
    long long sh = 0, sl = 0;
    for (int r = w; r < R.n; r += kFxWarps) {
        const int p0 = R.pre[r], p1 = R.pre[r + 1];
        for (int v = max(p0, v0) + lane; v < min(p1, v1); v += 32) {
            const int s = R.beg[r] + (v - p0);
            sy[v - v0] = E.s_xy[s];
            const double2 st = E.str[s];
            if constexpr (KERNEL == GQ_D) {
                const gfx30 a = fx_split30(fx_from_double(st.x, qe + 2));
                const gfx30 c = fx_split30(fx_from_double(st.y, qe + 2));
                sq[v - v0] = make_int4(a.h, a.l, c.h, c.l);
            } else {
                const gfx a = fx_bal(fx_from_double(st.x, qe));
                sq[v - v0] = make_int2(a.h, a.l);
                sh += a.h;
                sl += a.l;
            }
        }
    }
    if (KERNEL != GQ_D) {
        for (int o = 16; o > 0; o >>= 1) {
            sh += __shfl_xor_sync(0xffffffffu, sh, o);
            sl += __shfl_xor_sync(0xffffffffu, sl, o);
        }
        if (lane == 0) {
            ssum[2 * w] = sh;
            ssum[2 * w + 1] = sl;
        }
    }
    __syncthreads();
    return mx >= 128 && mx <= 1984 ? qe : 0;
}

// sum of the tile's strengths (2^62 of them) from the warps' words
__device__ __forceinline__ double fx_strength_sum(const long long *ssum) {
    long long qh = 0, ql = 0;
#pragma unroll
    for (int k = 0; k < kFxWarps; ++k) {
        qh += ssum[2 * k];
        ql += ssum[2 * k + 1];
    }
    return fma((double)qh, 4294967296.0, (double)ql);
}

// Blocks an SM is compiled for: the sums take 4 (QQ + 1) registers, and the chains
// of dependent multiply-adds want warps to hide them (q = 8, 1.05 M quadrature
// nodes: 3 blocks 4.04 ms, 4 3.60, 5 3.39, 7 3.31).
constexpr int fx_min_blocks(int q) { return q <= 8 ? 7 : q <= 12 ? 5 : 4; }
template <int QQ, int KERNEL>
__global__ void __launch_bounds__(kNearThreads, fx_min_blocks(QQ)) k_near_centres_fx(EvalView E, const int *__restrict__ work,
                                                                   double2 *__restrict__ Qout) {
    constexpr int NV = 2 * (QQ + 1);
    typedef typename FxStr<KERNEL>::T str_t;
    __shared__ NearRanges R;
    __shared__ int wsum[kFxWarps];
    __shared__ double2 sy[kFxTile];
    __shared__ str_t sq[kFxTile];
    __shared__ long long shl_[KERNEL == GQ_D ? 1 : kFxLogJ];
    __shared__ int stj[KERNEL == GQ_D ? 1 : kFxLogJ];
    __shared__ long long ssum[KERNEL == GQ_D ? 1 : 2 * kFxWarps];
    __shared__ int smax[kFxWarps];
    if (KERNEL != GQ_D)
        for (int i = threadIdx.x; i < kFxLogJ; i += kNearThreads) {
            shl_[i] = E.fxlog->hl[i];
            stj[i] = E.fxlog->t[i];
        }
    const int b = work[blockIdx.x];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ne = (E.loff[0][b + 1] - E.loff[0][b]) + (E.loff[2][b + 1] - E.loff[2][b]) + (E.loff[4][b + 1] - E.loff[4][b]);
    const int cb = E.ctr_beg[b], ce = E.ctr_end[b];
    // exponent of the box's rho^2: the logarithms are taken relative to it
    const double rho = box_rho(E.R, E.blev[b]);
    const int eref = 2 * fx_expo(fx_bits(rho)) - 1023;
    bool first = true;
    for (int e0 = 0; e0 < ne || first; e0 += kNearRanges) {
        __syncthreads();
        load_ranges(E, b, e0, ne, R, wsum);
        const int T = R.pre[R.n];
        for (int v0 = 0; v0 < T || first; v0 += kFxTile) {
            const int v1 = min(T, v0 + kFxTile), n = v1 - v0;
            if (v0) __syncthreads();
            bool any;
            const int qe = fx_stage<KERNEL>(E, R, v0, v1, sy, sq, ssum, smax, any);
            const bool scaled = qe > 0;
            const float amin = any ? (KERNEL == GQ_D ? kFxWeak : 0.5f * kFxWeak) * sqrtf((float)n) : 0.0f;
            for (int c = cb + w; c < ce; c += kFxWarps) {
                const double2 cz = E.sc_xy[c];
                const double rc = E.sc_r[c];
                const int qc = E.qc ? E.qc[c] : QQ;
                double2 *dst = Qout + (size_t)c * (QQ + 1);
                double re = rc;      // u = re/w
                bool slow = !scaled;
                unsigned nlim = 0;   // terms of sources with an upper word of |w|^2 below it are formed in FP64
                long long acc[NV];   // S: 0 the log sum, 1 unused, then Re, Im of each order; D: Re, Im of each order
                unsigned nmin = 0xffffffffu, nmax = 0;   // upper words of |w|^2
                unsigned am = 0;     // the lane's sum of |Re t| + |Im t|, t the term of order 1 (D: 0), upper words
                auto sweep = [&](auto without) {
                    const uint64_t rb = fx_bits(re);
                    const gfx Rm = fx_bal((long long)(fx_mant(rb) << 9));
                    const int er = fx_expo(rb);
                    nmin = 0xffffffffu;
                    nmax = am = 0;
#pragma unroll
                    for (int i = 0; i < NV; ++i) acc[i] = 0;
                    for (int v = lane; v < n; v += 32) {
                        const double2 y = sy[v];
                        const double wx = y.x - cz.x, wy = y.y - cz.y;
                        const double n2 = fma(wx, wx, wy * wy);
                        const uint64_t nb = fx_bits(n2);
                        str_t sv = sq[v];
                        if constexpr (KERNEL != GQ_D)
                            acc[0] += fx_mul(gfx{sv.x, sv.y}, fx_bal(fx_log_half(nb, eref, shl_, stj)));
                        const bool in = without.value && (unsigned)(nb >> 32) < nlim;
                        if (in) {
                            am += KERNEL == GQ_D ? (abs(sv.x) + abs(fx_second(sv))) >> 2 : abs(sv.x) >> 2;
                            sv = str_t{};
                        }
                        if (!in || KERNEL != GQ_D) nmin = min(nmin, (unsigned)(nb >> 32));
                        nmax = max(nmax, (unsigned)(nb >> 32));
                        gfx ux, uy, nuy;
                        fx_ratio(wx, wy, nb, Rm, er, ux, uy, nuy);
                        long long tr, ti;
                        if constexpr (KERNEL == GQ_D) {
                            fx_cmul30(gfx30{sv.x, sv.y}, gfx30{sv.z, sv.w}, ux, uy, nuy, tr, ti);
                            acc[0] += tr;
                            acc[1] += ti;
                        } else {
                            const gfx a{sv.x, sv.y};
                            tr = fx_mul(a, ux);
                            ti = fx_mul(a, uy);
                            acc[2] += tr;
                            acc[3] += ti;
                        }
                        am += abs((int)(tr >> 32)) + abs((int)(ti >> 32));
#pragma unroll
                        for (int m = KERNEL == GQ_D ? 1 : 2; m <= QQ; ++m) {
                            if (m % 4 == 0 && m > qc) break;
                            long long xr, xi;
                            fx_cmul30(fx_split30(tr), fx_split30(ti), ux, uy, nuy, xr, xi);
                            tr = xr;
                            ti = xi;
                            acc[2 * m] += tr;
                            acc[2 * m + 1] += ti;
                        }
                    }
                    nmin = __reduce_min_sync(0xffffffffu, nmin);
                    nmax = __reduce_max_sync(0xffffffffu, nmax);
                };
                if (!slow) {
                    bool inside;   // a source inside the disk, |u|^2 > 1 + 1/32
                    for (;;) {
                        sweep(std::false_type{});
                        const double wmin2 = __hiloint2double((int)nmin, 0);
                        inside = n > 0 && rc * rc > wmin2 * (1.0 + 1.0 / 32);
                        if (!inside || re != rc || (nmin >> 20) < 128) break;
                        re = sqrt(wmin2);
                    }
                    float a = (float)__reduce_add_sync(0xffffffffu, am >> 6);
                    if (inside) {
                        // The sums are scaled by (rc/re)^m and their rounding with them: either the
                        // last order (of the sources at re) or the first has to stand above it.
                        bool held = false;
                        if (re != rc) {
                            unsigned aq = 0;
#pragma unroll
                            for (int m = 1; m <= QQ; ++m)
                                if (m == qc) aq = abs((int)(acc[2 * m] >> 32)) + abs((int)(acc[2 * m + 1] >> 32));
                            held = (float)__reduce_add_sync(0xffffffffu, aq >> 6) >= amin ||
                                   a >= amin * powf((float)(rc / re), (float)(qc - 1));
                        }
                        if (!held) {   // once more without the powers of the sources inside
                            re = rc;
                            nlim = (unsigned)(fx_bits(rc * rc * (32.0 / 33)) >> 32) + 1;
                            sweep(std::true_type{});
                            a = (float)__reduce_add_sync(0xffffffffu, am >> 6);
                        }
                    }
                    // |w|^2 a normal number far from the range's ends, the logarithms below 14, the
                    // terms not weak beside the tile's scale (kFxWeak)
                    const int emin = (int)(nmin >> 20), emax = (int)(nmax >> 20), er = fx_expo(fx_bits(re));
                    slow = n > 0 && (emin < 128 || emax > 1920 || er < 128 || er > 1920 || (re == rc && !(a >= amin)) ||
                                     (KERNEL != GQ_D && (emax - eref > 40 || eref - emin > 40)));
                }
                if (slow) {
                    near_centre_fp64<KERNEL, QQ < 9 ? QQ + 1 : 9>(E, R, v0, v1, cz, rc, QQ, qc, kAllSources, dst, first);
                    continue;
                }
                // exact sum of the log terms as two words; the others at 2^-60 or as close to
                // it as the warp's sum allows
                if (KERNEL != GQ_D) {
                    acc[1] = acc[0] & ((1 << 27) - 1);
                    acc[0] >>= 27;
                }
                unsigned top = 0;
#pragma unroll
                for (int i = KERNEL == GQ_D ? 0 : 2; i < NV; ++i) {
                    const int h = (int)(acc[i] >> 32);
                    top |= (unsigned)(h ^ (h >> 31));
                }
                // each |acc| < 2^(64 - clz); 32 of them have to stay below 2^63
                const int sh = max(0, 6 - __clz((int)__reduce_or_sync(0xffffffffu, top)));
                const long long half = (1ll << sh) >> 1;
#pragma unroll
                for (int i = KERNEL == GQ_D ? 0 : 2; i < NV; ++i) acc[i] = (acc[i] + half) >> sh;
                int base, cnt;
                warp_reduce_scatter(acc, 0ll, lane, [](long long a, long long x) { return a + x; },
                                    [](long long x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); }, base, cnt);
                long long lo = 0;
                if (KERNEL != GQ_D) {
                    constexpr RsPlace p1 = rs_place(NV, 1);
                    lo = __shfl_sync(0xffffffffu, acc[p1.slot], p1.lane);
                }
                const double sc = pow2_clamped(qe + 1 - 55), sct = pow2_clamped(qe + 1 - 60 + sh);
                double *d = reinterpret_cast<double *>(dst);
#pragma unroll
                for (int j = 0; j < (NV + 31) / 32; ++j)
                    if (j < cnt) {
                        const int i = base + j, m = i >> 1;
                        double x;
                        if (KERNEL != GQ_D && m == 0) {
                            x = 0.0;
                            if (i == 0) {
                                // the log terms have 2^55, the strengths 2^62
                                const double sumq = fx_strength_sum(ssum);
                                x = fma((double)acc[0], 134217728.0, (double)lo) * sc +
                                    sumq * (sc * 0x1p-7) * ((eref - 1023) * 0.34657359027997264);
                            }
                        } else {
                            x = m <= qc ? (double)acc[j] * sct : 0.0;
                            if (KERNEL != GQ_D) x *= c_ninv[m];
                            if (re != rc)
                                for (int k = 0; k < m; ++k) x *= rc / re;
                            if (KERNEL == GQ_D) x /= re;
                        }
                        d[i] = first ? x : d[i] + x;
                    }
                if (nlim) {
                    __syncwarp();   // lane 0 adds to what the lanes have written
                    near_centre_fp64<KERNEL, QQ < 9 ? QQ + 1 : 9>(E, R, v0, v1, cz, rc, QQ, qc, nlim, dst, false);
                }
            }
            first = false;
        }
    }
}

// Potential at the point targets for S, sum q log|t - y| (coincident sources
// skipped): a block per target box, a warp per target, lanes stride over the
// staged sources; |w|^2 in FP64, logarithm, products and sums in fixed point.  The
// FP64 pipe bounds it (79 % busy with 7.5 instructions a pair, at ten targets and 70
// sources a box, which fill three rounds of a warp to three quarters): four are
// |w|^2, so the conversions of a target's sum wait in the lanes until 32 targets are
// converted by one instruction, and the strengths' sum is formed once a tile (11.6
// instructions and 83 % before).  Resident blocks over several boxes, no staging, a
// warp a box or several targets a warp were slower.  0.86 M point targets: 1.37 (FP64)
// -> 1.11 -> 0.73 ms.  For D the point targets stay with the FP64 k_near_points.
__global__ void __launch_bounds__(kNearThreads) k_near_points_fx(EvalView E, const int *__restrict__ work,
                                                                 double *__restrict__ pot) {
    __shared__ NearRanges R;
    __shared__ int wsum[kFxWarps];
    __shared__ double2 sy[kFxTile];
    __shared__ int2 sq[kFxTile];
    __shared__ long long shl_[kFxLogJ];
    __shared__ int stj[kFxLogJ];
    __shared__ long long ssum[2 * kFxWarps];
    __shared__ int smax[kFxWarps];
    for (int i = threadIdx.x; i < kFxLogJ; i += kNearThreads) {
        shl_[i] = E.fxlog->hl[i];
        stj[i] = E.fxlog->t[i];
    }
    const int b = work[blockIdx.x];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int ne = (E.loff[0][b + 1] - E.loff[0][b]) + (E.loff[2][b + 1] - E.loff[2][b]) + (E.loff[4][b + 1] - E.loff[4][b]);
    const int tb = E.pt_beg[b], te = E.pt_end[b];
    const int eref = 2 * fx_expo(fx_bits(box_rho(E.R, E.blev[b]))) - 1023;   // logarithms relative to rho^2
    bool first = true;
    for (int e0 = 0; e0 < ne || first; e0 += kNearRanges) {
        __syncthreads();
        load_ranges(E, b, e0, ne, R, wsum);
        const int T = R.pre[R.n];
        for (int v0 = 0; v0 < T || first; v0 += kFxTile) {
            const int v1 = min(T, v0 + kFxTile), n = v1 - v0;
            if (v0) __syncthreads();
            bool any;
            const int qe = fx_stage<GQ_S>(E, R, v0, v1, sy, sq, ssum, smax, any);
            const double sc = pow2_clamped(qe + 1 - 55);
            const double q0 = qe > 0 ? fx_strength_sum(ssum) * (sc * 0x1p-7) * ((eref - 1023) * 0.34657359027997264) : 0.0;
            // the sums of up to 32 targets wait in the lanes and are converted together
            long long khi = 0;
            int klo = 0, kt = -1, held = 0;
            auto flush = [&]() {
                if (kt >= 0) {
                    const double x = fma((double)khi, 16777216.0, (double)klo) * sc + q0;
                    pot[kt] = first ? x : pot[kt] + x;
                    kt = -1;
                }
                held = 0;
            };
            for (int t = tb + w; t < te; t += kFxWarps) {
                const double2 tz = E.sp_xy[t];
                long long acc = 0;
                unsigned nmin = 0xffffffffu, nmax = 0;
                if (qe > 0)
                    for (int v = lane; v < n; v += 32) {
                        const double2 y = sy[v];
                        const double wx = y.x - tz.x, wy = y.y - tz.y;
                        const uint64_t nb = fx_bits(fma(wx, wx, wy * wy));
                        nmin = min(nmin, (unsigned)(nb >> 32));
                        nmax = max(nmax, (unsigned)(nb >> 32));
                        const int2 sv = sq[v];
                        acc += fx_mul(gfx{sv.x, sv.y}, fx_bal(fx_log_half(nb, eref, shl_, stj)));
                    }
                nmin = __reduce_min_sync(0xffffffffu, nmin);
                nmax = __reduce_max_sync(0xffffffffu, nmax);
                const int emin = (int)(nmin >> 20), emax = (int)(nmax >> 20);
                if (qe > 0 && (n == 0 || (emin >= 128 && emax <= 1920 && emax - eref <= 40 && eref - emin <= 40))) {
                    // 12 terms below 2^58.8 a lane: the sum over lanes in two words
                    int lo = (int)(acc & ((1 << 24) - 1));
                    long long hi = acc >> 24;
                    for (int o = 16; o > 0; o >>= 1) hi += __shfl_xor_sync(0xffffffffu, hi, o);
                    lo = __reduce_add_sync(0xffffffffu, lo);
                    if (lane == held) {
                        khi = hi;
                        klo = lo;
                        kt = t;
                    }
                    if (++held == 32) flush();
                } else {   // in FP64, infinities and coincident sources included
                    double x = 0.0;
                    int r = 0;
                    for (int v = v0 + lane; v < v1; v += 32) {
                        while (R.pre[r + 1] <= v) ++r;
                        const int s = R.beg[r] + (v - R.pre[r]);
                        const double2 y = E.s_xy[s];
                        const double wx = y.x - tz.x, wy = y.y - tz.y, n2 = wx * wx + wy * wy;
                        x = fma(E.str[s].x, n2 == 0.0 ? 0.0 : gq_log_half(n2, E.logt), x);
                    }
                    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                    if (lane == 0) pot[t] = first ? x : pot[t] + x;
                }
            }
            flush();
            first = false;
        }
    }
}

template <int QQ>
void launch_near_centres_fx(gq_ctx *ctx, const EvalView &E, int nwork, const int *work, double2 *Q) {
    auto kd = k_near_centres_fx<QQ, GQ_D>;
    auto ks = k_near_centres_fx<QQ, GQ_S>;
    GQ_LAUNCH(ctx, (E.kernel == GQ_D ? kd : ks), nwork, kNearThreads, 0, E, work, Q);
}

}  // namespace

void gq_near_centres_fx(gq_ctx *ctx, const EvalView &E, int nwork, const int *work, double2 *Q) {
    switch (E.Q) {
#define GQ_CASE(v) case v: launch_near_centres_fx<v>(ctx, E, nwork, work, Q); break;
        GQ_CASE(1) GQ_CASE(2) GQ_CASE(3) GQ_CASE(4) GQ_CASE(5) GQ_CASE(6) GQ_CASE(7) GQ_CASE(8)
        GQ_CASE(9) GQ_CASE(10) GQ_CASE(11) GQ_CASE(12) GQ_CASE(13) GQ_CASE(14) GQ_CASE(15) GQ_CASE(16)
#undef GQ_CASE
        default: throw gq_error{GQ_ERR_INVALID, "p_qbx out of range"};
    }
}

void gq_near_points_fx(gq_ctx *ctx, const EvalView &E, int nwork, const int *work, double *pot) {
    GQ_LAUNCH(ctx, k_near_points_fx, nwork, kNearThreads, 0, E, work, pot);
}
