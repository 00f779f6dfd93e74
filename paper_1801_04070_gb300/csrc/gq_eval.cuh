// gq_eval.cuh -- what the evaluation kernels share: the view of a built tree,
// box geometry, the direct sums' source ranges and the warp reduce-scatter.
#pragma once

#include "gq_fix.cuh"
#include "gq_internal.cuh"

struct EvalView {
    RootInfo R;
    int P, Q, kernel;
    const int *blev, *bix, *biy, *bparent;
    const int4 *bchild;
    const int *src_beg, *src_end;
    const int *ctr_beg, *ctr_end, *pt_beg, *pt_end;
    const int *sub_src, *sub_tgt;
    const double2 *s_xy;
    const double2 *str;
    const double2 *sc_xy;
    const double *sc_r;
    const double2 *sp_xy;
    const int *loff[6];
    const int *lidx[6];
    const double *binom;   // [kBinN][kBinN]
    const int *qc;         // per-centre QBX order (sorted centres) or nullptr: all use Q
    const double *logt;    // GqLogTable
    const unsigned int *qexp;   // largest biased exponent of the S strengths (k_strengths)
    const FxLogTable *fxlog;    // table of the fixed-point logarithm
    int nwork_ctr;              // boxes owning centres (batched items)
};

static __device__ __forceinline__ double box_rho(const RootInfo &R, int l) { return ldexp(R.H, -l); }
static __device__ __forceinline__ double2 box_centre(const RootInfo &R, int l, int ix, int iy) {
    double h = ldexp(R.H, -l);
    return make_double2(R.lo_x + (double)(2 * ix + 1) * h, R.lo_y + (double)(2 * iy + 1) * h);
}

// ------------------------------------------------------------------ Stages 3, 5a, 6a: direct near field
// One block per target box; the box's List 1, 3 close and 4 close source
// ranges are flattened into shared memory; each warp takes one target and its
// lanes stride over the flattened sources.
constexpr int kNearThreads = 128;
constexpr int kNearRanges = 256;

struct NearRanges {
    int beg[kNearRanges];
    int pre[kNearRanges + 1];
    int n;
};

static __device__ __forceinline__ int block_excl_scan_128(int v, int *wsum) {
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    int off = 0;
    for (int i = 0; i < w; ++i) off += wsum[i];
    __syncthreads();
    return off + x - v;
}

// load entries [e0, e0 + kNearRanges) of the concatenated lists U, WC, XC of box b
static __device__ __forceinline__ void load_ranges(const EvalView &E, int b, int e0, int ne, NearRanges &R, int *wsum) {
    int n0 = E.loff[0][b + 1] - E.loff[0][b], n2 = E.loff[2][b + 1] - E.loff[2][b];
    int cnt = min(kNearRanges, ne - e0);
    int lens[2] = {0, 0};
    for (int r = 0; r < 2; ++r) {
        int i = threadIdx.x * 2 + r;
        if (i < cnt) {
            int e = e0 + i, d;
            if (e < n0) d = E.lidx[0][E.loff[0][b] + e];
            else if (e < n0 + n2) d = E.lidx[2][E.loff[2][b] + e - n0];
            else d = E.lidx[4][E.loff[4][b] + e - n0 - n2];
            R.beg[i] = E.src_beg[d];
            lens[r] = E.src_end[d] - E.src_beg[d];
        }
    }
    int pre = block_excl_scan_128(lens[0] + lens[1], wsum);
    if (threadIdx.x * 2 < kNearRanges) R.pre[threadIdx.x * 2] = pre;
    if (threadIdx.x * 2 + 1 < kNearRanges) R.pre[threadIdx.x * 2 + 1] = pre + lens[0];
    if (threadIdx.x == kNearThreads - 1) R.pre[kNearRanges] = pre + lens[0] + lens[1];
    if (threadIdx.x == 0) R.n = cnt;
    __syncthreads();
}

// Warp reduce-scatter of NV values per lane: at each of the five butterfly
// steps a lane keeps one half of its values, sends the other half to its
// partner and adds what it receives, so a warp spends about NV adds instead of
// 5 NV.  Afterwards lane L holds the warp sums of the original entries
// base .. base + cnt - 1 in v[0 .. cnt) (cnt may be 0; for NV <= 32 it is 0 or 1).
template <int N, int O, class V, class Add, class Shfl>
__device__ __forceinline__ void rs_step(V *v, int lane, V zero, Add add, Shfl shfl, int &base, int &cnt) {
    constexpr int H = (N + 1) / 2;
    const bool up = (lane & O) != 0;
#pragma unroll
    for (int i = 0; i < H; ++i) {
        V x = v[i], y = (i + H < N) ? v[i + H < N ? i + H : 0] : zero;
        V send = up ? x : y, keep = up ? y : x;
        v[i] = add(keep, shfl(send, O));
    }
    if (up) {
        base += H;
        cnt -= H;
    } else if (cnt > H) {
        cnt = H;
    }
}

template <int NV, class V, class Add, class Shfl>
__device__ __forceinline__ void warp_reduce_scatter(V (&v)[NV], V zero, int lane, Add add, Shfl shfl, int &base,
                                                    int &cnt) {
    constexpr int H1 = (NV + 1) / 2, H2 = (H1 + 1) / 2, H3 = (H2 + 1) / 2, H4 = (H3 + 1) / 2;
    base = 0;
    cnt = NV;
    rs_step<NV, 16>(v, lane, zero, add, shfl, base, cnt);
    rs_step<H1, 8>(v, lane, zero, add, shfl, base, cnt);
    rs_step<H2, 4>(v, lane, zero, add, shfl, base, cnt);
    rs_step<H3, 2>(v, lane, zero, add, shfl, base, cnt);
    rs_step<H4, 1>(v, lane, zero, add, shfl, base, cnt);
    if (cnt < 0) cnt = 0;
}

// ------------------------------------------------------------------ multipoles in fixed point
// exponent of a box whose multipoles are not all finite
constexpr int kFxNaNExp = 1 << 20;
// The scale 2^(x - 1023) of v.  Where it is no normal number v is scaled instead, in two
// steps that round once, and the scale is 1 (strengths near the ends of the range,
// whose sums are still finite); NaN for a box of kFxNaNExp.
static __device__ __forceinline__ double fx_scale(double &v, int x) {
    if ((unsigned)(x - 1) < 2046u) return __longlong_as_double((long long)x << 52);
    const int n = max(x - 1023, -1500), h = n >> 1;   // (a box of zeros: far below)
    if (x > kFxNaNExp / 2) v = __longlong_as_double(0x7ff8000000000000ll);
    else v = v * __longlong_as_double((long long)(h + 1023) << 52) * __longlong_as_double((long long)(n - h + 1023) << 52);
    return 1.0;
}

// direct sums to the QBX centres in 64-bit fixed point (gq_near_fx.cu): Qout [nc][E.Q+1]
void gq_near_centres_fx(gq_ctx *ctx, const EvalView &E, int nwork, const int *work, double2 *Qout);
// direct potential at the point targets for S, likewise (gq_near_fx.cu)
void gq_near_points_fx(gq_ctx *ctx, const EvalView &E, int nwork, const int *work, double *pot);
// List 2 translations (M2L) of orders 16 .. 30 in fixed point (gq_m2l_fx.cu), added to L
void gq_m2l_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double2 *L);
void gq_m2l_fx_prepare(int dev);   // its tables on device dev
// the multipoles of the boxes in fixed point, into g->Mfx and g->Efx (gq_w_fx.cu)
void gq_mfix(gq_geom *g, gq_ctx *ctx, int P1, const double2 *M);
// List 3 far (gq_w_fx.cu), from g->Mfx and g->Efx: multipoles at the point targets, and to
// the QBX centres for p_qbx <= kWFxMaxQ, added to pot and Q
constexpr int kWFxMaxQ = 10;
void gq_w_points_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double *pot);
void gq_w_centres_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, const double2 *M, double2 *Q);
void gq_w_fx_prepare(int dev);     // its tables on device dev
// M2M of all levels in fixed point (gq_m2m_fx.cu)
void gq_m2m_fx(gq_geom *g, gq_ctx *ctx, const EvalView &E, double2 *M);
void gq_m2m_fx_prepare(int dev);   // its table on device dev
