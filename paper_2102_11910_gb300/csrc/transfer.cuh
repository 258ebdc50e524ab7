// Vortex-grid transfer kernels shared by the regularization entry points and
// the tile-ordered vortex state (internal; every translation unit that
// includes it gets its own copies of these kernels).
#pragma once
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fixpt.cuh"

namespace {

constexpr int BIN_THREADS = 256;
constexpr int BIN_UNROLL = 4;        // vortices per thread whose loads are issued together

// Per-vortex cell record (original order).  Mixed path: packed cell and the
// 32-bit cell fractions as fixed-point integers; FP64: cell and fractions.
template <typename T> struct Pos;
template <> struct __align__(16) Pos<float> {
    unsigned cell;        // ci | cj << 16
    unsigned fxw, fyw;    // fraction * 2^32 (truncated)
    float g;
};
template <> struct __align__(16) Pos<double> {
    int ci, cj;
    double fx, fy, g;
};
// Per-tile record: cell relative to the tile origin (lx, ly in [-2, 32]),
// fractions, Gamma and the vortex's original index q.  Mixed path: each
// fraction keeps 24 bits, fixed point, with the biased local cell lx + 2 in the
// low 8 bits of the same word (16 bytes in all, like the FP64 record's 32).
template <typename T> struct Rec;
template <> struct __align__(16) Rec<float> {
    unsigned xw, yw;      // (fraction * 2^32) & ~0xFF | (local cell + 2)
    float g;
    int q;
};
template <> struct __align__(16) Rec<double> {
    short lx, ly;
    int q;
    double fx, fy, g;
};

__device__ __forceinline__ int pos_ci(const Pos<float>& p) { return (int)(p.cell & 0xFFFFu); }
__device__ __forceinline__ int pos_cj(const Pos<float>& p) { return (int)(p.cell >> 16); }
__device__ __forceinline__ int pos_ci(const Pos<double>& p) { return p.ci; }
__device__ __forceinline__ int pos_cj(const Pos<double>& p) { return p.cj; }

__device__ __forceinline__ int rec_lx(const Rec<float>& r) { return (int)(r.xw & 0xFFu) - 2; }
__device__ __forceinline__ int rec_ly(const Rec<float>& r) { return (int)(r.yw & 0xFFu) - 2; }
__device__ __forceinline__ float rec_fx(const Rec<float>& r) { return __uint2float_rn(r.xw >> 8) * 0x1p-24f; }
__device__ __forceinline__ float rec_fy(const Rec<float>& r) { return __uint2float_rn(r.yw >> 8) * 0x1p-24f; }
__device__ __forceinline__ int rec_lx(const Rec<double>& r) { return r.lx; }
__device__ __forceinline__ int rec_ly(const Rec<double>& r) { return r.ly; }
__device__ __forceinline__ double rec_fx(const Rec<double>& r) { return r.fx; }
__device__ __forceinline__ double rec_fy(const Rec<double>& r) { return r.fy; }

__device__ __forceinline__ Rec<float> make_rec(const Pos<float>& p, int lx, int ly, int q) {
    Rec<float> r;
    r.xw = (p.fxw & ~0xFFu) | (unsigned)(lx + 2);
    r.yw = (p.fyw & ~0xFFu) | (unsigned)(ly + 2);
    r.g = p.g;
    r.q = q;
    return r;
}
__device__ __forceinline__ Rec<double> make_rec(const Pos<double>& p, int lx, int ly, int q) {
    Rec<double> r;
    r.lx = (short)lx;
    r.ly = (short)ly;
    r.q = q;
    r.fx = p.fx;
    r.fy = p.fy;
    r.g = p.g;
    return r;
}

// M4' weights of the four nodes floor(g)-1 .. floor(g)+2 for fractional part f.
// FP32: the cubics term by term (their arithmetic hides behind the shared
// adds and loads: the nine-operation form below measured no faster there).
__device__ __forceinline__ void m4p_weights(float f, float w[4]) {
    const float a0 = 1.0f + f, a1 = f, a2 = 1.0f - f, a3 = 2.0f - f;
    w[0] = 0.5f * (2.0f - a0) * (2.0f - a0) * (1.0f - a0);
    w[1] = 1.0f - 2.5f * a1 * a1 + 1.5f * a1 * a1 * a1;
    w[2] = 1.0f - 2.5f * a2 * a2 + 1.5f * a2 * a2 * a2;
    w[3] = 0.5f * (2.0f - a3) * (2.0f - a3) * (1.0f - a3);
}
// FP64: with t = 1 - f and p = f t the cubics are -p t / 2, t + p (1 - 3/2 f),
// f + p (1 - 3/2 t) and -p f / 2, nine operations of a pipe that issues two a
// clock and SM.
__device__ __forceinline__ void m4p_weights(double f, double w[4]) {
    const double t = 1.0 - f, p = f * t, h = -0.5 * p;
    w[0] = h * t;
    w[1] = fma(p, fma(-1.5, f, 1.0), t);
    w[2] = fma(p, fma(-1.5, t, 1.0), f);
    w[3] = h * f;
}

// The same weights in Q61 as centred halves (fixpt.cuh), from the fraction in
// Q60: FP64 records' terms are formed on the integer pipe, which issues a 32 x
// 32 + 64 multiply-add sixteen times as often as the FP64 pipe a multiply.
// With a = p f and b = p t = p - a the weights are -b/2, t + p - 3/2 a, f + p -
// 3/2 b, -a/2: their sum is exactly one, each is within 2^-60 of its value.
constexpr int Q_FRAC = 60, Q_WEIGHT = 61;
__device__ __forceinline__ long long fx_frac(double f) {       // f in [0, 1): multiples of 2^-60 are exact
    const long long b = __double_as_longlong(f);
    const int ef = (int)(b >> 52);
    if (ef == 0) return 0;
    const long long m = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    const int d = 1075 - Q_FRAC - ef;                            // m 2^(ef - 1075) 2^60
    return d <= 0 ? m << -d : (d > 54 ? 0ll : (m + ((1ll << d) >> 1)) >> d);
}
__device__ __forceinline__ long long fx_qmul60(long long a, long long b) {
    const FxSplit x = fx_split(a), y = fx_split(b);
    const long long t = (1ll << 28) + fx_mw(x.h, y.l) + fx_mw(x.l, y.h);
    return (fx_mw(x.h, y.h) << 2) + (t >> 29);
}
__device__ __forceinline__ void fx_m4p(double frac, FxSplit (&w)[4]) {
    const long long f = fx_frac(frac), t = (1ll << Q_FRAC) - f, p = fx_qmul60(f, t), a = fx_qmul60(p, f), b = p - a;
    w[0] = fx_split(-b);
    w[1] = fx_split(2 * (t + p) - 3 * a);
    w[2] = fx_split(2 * (f + p) - 3 * b);
    w[3] = fx_split(-a);
}
// x w 2^-61
__device__ __forceinline__ long long fx_weigh(FxSplit x, FxSplit w) {
    const long long t = (1ll << 29) + fx_mw(x.h, w.l) + fx_mw(x.l, w.h);
    return (fx_mw(x.h, w.h) << 1) + (t >> 30);
}

// Grid coordinate g of a position; the stencil floor(g)-1 .. floor(g)+2 lies in
// [0, n) iff 1 <= g < n - 2.  FP64 path: g = (X - x0)/dx, fraction g - floor(g)
// exact (the binning passes: split_div).  Mixed path: one FMA, then the integer and fractional parts are read
// from the bits of g (no further FP64 work); the fraction is truncated to 24 bits.
__device__ __forceinline__ bool split(double X, double x0, double dx, double, double, int n, long long, int& c,
                                      double& f) {
    const double g = (X - x0) / dx;
    if (!(g >= 1.0 && g < (double)(n - 2))) return false;
    const double fl = floor(g);
    c = (int)fl;
    f = g - fl;
    return true;
}
__device__ __forceinline__ bool split(double X, double, double, double inv_dx, double c0, int, long long lim, int& c,
                                      float& f) {
    const double g = fma(X, inv_dx, c0);
    // 1 <= g < n - 2 compared on the bit patterns (monotone for non-negative
    // doubles; negative values and NaN fail; lim = bits of (double)(n - 2)),
    // keeping the FP64 pipe for the FMA
    const long long gb = __double_as_longlong(g);
    if (gb < 0x3FF0000000000000ll || gb >= lim) return false;
    // g = 2^e (1 + m 2^-52), 0 <= e <= 10 since g < 2048: the integer part is the
    // top e fraction bits with the hidden bit, the cell fraction the next 32
    const unsigned hi = (unsigned)((unsigned long long)gb >> 32), lo = (unsigned)gb;
    const int e = (int)(hi >> 20) - 1023;
    const unsigned m20 = hi & 0xFFFFFu;
    c = (int)((m20 | 0x100000u) >> (20 - e));
    f = __uint2float_rz(__funnelshift_l(lo, m20, 12 + e)) * 0x1p-32f;
    return true;
}

// Mixed path of the binning passes: as split, but the cell fraction is returned
// as a 32-bit fixed-point integer (fraction * 2^32, truncated).
__device__ __forceinline__ bool split_fixed(double X, double inv_dx, double c0, long long lim, int& c, unsigned& fr) {
    const double g = fma(X, inv_dx, c0);
    const long long gb = __double_as_longlong(g);
    if (gb < 0x3FF0000000000000ll || gb >= lim) return false;
    const unsigned hi = (unsigned)((unsigned long long)gb >> 32), lo = (unsigned)gb;
    const int e = (int)(hi >> 20) - 1023;
    const unsigned m20 = hi & 0xFFFFFu;
    c = (int)((m20 | 0x100000u) >> (20 - e));
    fr = __funnelshift_l(lo, m20, 12 + e);
    return true;
}

// double -> float rounded to nearest even with integer instructions only (the
// FP64 pipe is 1/64 rate); zero, and values outside the normal FP32 range,
// take the hardware conversion.  Bitwise equal to (float)d.
__device__ __forceinline__ float d2f(double d) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7FF) - 1023 + 127;
    if (e <= 0 || e >= 255) return (float)d;
    const unsigned long long m = b & 0xFFFFFFFFFFFFFull;     // 52 fraction bits
    const unsigned top = (unsigned)(m >> 29);                // the 23 kept
    const unsigned rest = (unsigned)(m & 0x1FFFFFFFull);     // the 29 dropped
    unsigned out = sign | ((unsigned)e << 23) | top;
    if (rest > 0x10000000u || (rest == 0x10000000u && (top & 1u))) ++out;   // carries into the exponent
    return __uint_as_float(out);
}

__device__ __forceinline__ void make_pos(Pos<float>& p, int ci, int cj, unsigned fxw, unsigned fyw, double g) {
    p.cell = (unsigned)ci | ((unsigned)cj << 16);
    p.fxw = fxw;
    p.fyw = fyw;
    p.g = d2f(g);
}
__device__ __forceinline__ void make_pos(Pos<double>& p, int ci, int cj, double fx, double fy, double g) {
    p.ci = ci;
    p.cj = cj;
    p.fx = fx;
    p.fy = fy;
    p.g = g;
}

struct Geo {
    double x0, y0, dx;
    double inv_dx, cx, cy;     // 1/dx, -x0/dx, -y0/dx (host computed)
    double inv_dx2;            // 1/dx^2
    long long xlim, ylim;      // bit patterns of (double)(nx - 2), (double)(ny - 2)
    int nx, ny, ntx, ntiles;
    int recip;                 // dx and 1/dx far from the ends of the double range: loc_split divides by 1/dx
};

// the split used by the locate pass: fixed-point fraction (mixed), exact (FP64)
__device__ __forceinline__ bool loc_split(double X, const Geo& g, int axis, int& c, unsigned& fr) {
    return split_fixed(X, g.inv_dx, axis ? g.cy : g.cx, axis ? g.ylim : g.xlim, c, fr);
}
// g = (X - x0)/dx as the division gives it, from the rounded reciprocal: two
// corrections by exact residuals (Markstein's theorem: with the correctly
// rounded reciprocal the second one rounds correctly).  Range test, cell and
// fraction from the bits of g, so that a coordinate costs six FP64
// instructions instead of a division's fifteen and six more (k_locate at 1e6
// vortices: 60 -> 33 us).
__device__ __forceinline__ bool loc_split(double X, const Geo& geo, int axis, int& c, double& f) {
    const double x0 = axis ? geo.y0 : geo.x0;
    if (!geo.recip) return split(X, x0, geo.dx, 0.0, 0.0, axis ? geo.ny : geo.nx, 0, c, f);
    const double d = X - x0;
    double g = d * geo.inv_dx;
    g = fma(fma(-g, geo.dx, d), geo.inv_dx, g);
    g = fma(fma(-g, geo.dx, d), geo.inv_dx, g);
    const long long gb = __double_as_longlong(g);
    if (gb < 0x3FF0000000000000ll || gb >= (axis ? geo.ylim : geo.xlim)) return false;
    const int e = (int)(gb >> 52) - 1023;                               // 0 .. 10
    const long long m = (gb & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    c = (int)(m >> (52 - e));
    const long long r = m & ((1ll << (52 - e)) - 1);                    // fraction 2^(52 - e)
    const int lz = __clzll(r);                                          // leading bit to bit 52
    f = r == 0 ? 0.0 : __longlong_as_double((r << (lz - 11)) + ((long long)(1023 + 10 + e - lz) << 52));
    return true;
}
// Cell and fraction as the records carry them (mixed: 24 bits of it): R_v and
// E_v at the same position are each other's transpose, so that a vortex's
// velocity under its own field cancels.
__device__ __forceinline__ bool split_rec(double X, const Geo& g, int axis, int& c, float& f) {
    unsigned fr = 0;
    const bool ok = loc_split(X, g, axis, c, fr);
    f = __uint2float_rn(fr >> 8) * 0x1p-24f;
    return ok;
}
__device__ __forceinline__ bool split_rec(double X, const Geo& g, int axis, int& c, double& f) { return loc_split(X, g, axis, c, f); }
template <typename T> using Frac = typename std::conditional<sizeof(T) == 4, unsigned, double>::type;

// max(m, |g|), compared as integers, so that a NaN is above all; NaNs as infinities
__device__ __forceinline__ float abs_max(float m, float g) {
    return __int_as_float(max(__float_as_int(m), __float_as_int(g) & 0x7FFFFFFF));
}
__device__ __forceinline__ double abs_max(double m, double g) {
    return __longlong_as_double(max(__double_as_longlong(m), __double_as_longlong(g) & 0x7FFFFFFFFFFFFFFFll));
}
__device__ __forceinline__ float no_nan(float m) { return m <= INFINITY ? m : INFINITY; }
__device__ __forceinline__ double no_nan(double m) {
    return __longlong_as_double(min(__double_as_longlong(m), 0x7FF0000000000000ll));
}

// The vortex count and block span of a binning pass: the launch's own, or,
// when dn is given (a captured step replayed at a growing count), dn[0] with
// the span bin_span computes for it; blocks past the count bin nothing.
// (max_blocks: the launch's partition mode, BIN_MAX_BLOCKS or BIN_WIDE_BLOCKS,
// chosen on the host for the capacity.)
__device__ __forceinline__ void bin_count(const int64_t* dn, int min_span, int max_blocks, int64_t& nv,
                                          int64_t& span) {
    if (!dn) return;
    nv = *dn;
    const int64_t s = (nv + max_blocks - 1) / max_blocks;
    span = s < min_span ? min_span : s;
}

template <typename T, int TILE, int NT>
__global__ void __launch_bounds__(NT) k_locate(const double* __restrict__ X, const double* __restrict__ Y,
                                                       const double* __restrict__ G, int64_t nv, int64_t span,
                                                       const int64_t* __restrict__ dn, int min_span, int max_blocks, Geo geo,
                                                       Pos<T>* __restrict__ pos, int* __restrict__ hist,
                                                       double* __restrict__ gmax_blk, int* __restrict__ status,
                                                       unsigned long long* __restrict__ oob, T* __restrict__ zu,
                                                       T* __restrict__ zv) {
    extern __shared__ unsigned sm[];
    __shared__ T wmax[NT / 32];
    unsigned* cnt = sm;
    T gm = T(0);          // in the record's precision: no FP64 instruction per vortex in the mixed path
    for (int i = threadIdx.x; i < geo.ntiles; i += NT) cnt[i] = 0u;
    pdl_wait();
    bin_count(dn, min_span, max_blocks, nv, span);
    __syncthreads();
    const int64_t lo = (int64_t)blockIdx.x * span;
    const int64_t hi = lo + span < nv ? lo + span : nv;
    int bad = 0;
    for (int64_t base = lo; base < hi; base += NT * BIN_UNROLL) {
        // issue the loads of BIN_UNROLL vortices before using any of them
        double xs[BIN_UNROLL], ys[BIN_UNROLL], gs[BIN_UNROLL];
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {   // clamped: a thread past the end reloads the last vortex
            int64_t q = base + k * NT + threadIdx.x;
            q = q < hi ? q : hi - 1;
            xs[k] = X[q];
            ys[k] = Y[q];
            gs[k] = G[q];
        }
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {
            const int64_t q = base + k * NT + threadIdx.x;
            if (q >= hi) break;
            int ci = 0, cj = 0;
            Frac<T> fx = 0, fy = 0;
            Pos<T> p;
            if (!loc_split(xs[k], geo, 0, ci, fx) || !loc_split(ys[k], geo, 1, cj, fy)) {
                ++bad;
                make_pos(p, 0xFFFF, 0xFFFF, Frac<T>(0), Frac<T>(0), 0.0);   // marker: skipped by scatter
                pos[q] = p;
                if (zu) {                             // no E_v record: its velocity is zero
                    zu[q] = T(0);
                    zv[q] = T(0);
                }
                continue;
            }
            make_pos(p, ci, cj, fx, fy, gs[k]);
            pos[q] = p;
            gm = abs_max(gm, p.g);                 // |Gamma| as the record carries it
            const int tx0 = (ci - 1) / TILE, tx1 = (ci + 2) / TILE;
            const int ty0 = (cj - 1) / TILE, ty1 = (cj + 2) / TILE;
            const int t0 = ty0 * geo.ntx + tx0;
            const bool px = tx1 > tx0, py = ty1 > ty0;
            atomicAdd(&cnt[t0], 1u);
            if (px) atomicAdd(&cnt[t0 + 1], 1u);
            if (py) atomicAdd(&cnt[t0 + geo.ntx], 1u);
            if (px && py) atomicAdd(&cnt[t0 + geo.ntx + 1], 1u);
        }
    }
    if (bad) {
        atomicAdd(oob, (unsigned long long)bad);
        atomicOr(status, ST_OUT_OF_DOMAIN);
    }
    gm = no_nan(gm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = gm;
    __syncthreads();
    if (threadIdx.x == 0) {
        T m = T(0);
        for (int i = 0; i < NT / 32; ++i) m = fmax(m, wmax[i]);
        gmax_blk[blockIdx.x] = (double)m;
    }
    int* row = hist + (size_t)blockIdx.x * geo.ntiles;
    for (int i = threadIdx.x; i < geo.ntiles; i += NT) row[i] = (int)cnt[i];
}

// Fixed-point exponent of a tile: every node sum is bounded by
// count * max|Gamma| < 2^e and is scaled to stay below 2^61.
__device__ __forceinline__ int tile_shift_of(unsigned count, double gmax) {
    const double bound = (double)count * gmax;
    int e = 0;
    if (bound > 0.0) frexp(bound, &e);
    const int sh = 61 - e;
    return sh > 100 ? 100 : (sh < -60 ? -60 : sh);
}

// k_offsets: a block covers OFF_TILES tiles; its OFF_SEGS x OFF_TILES threads
// each own a run of at most OFF_RUN consecutive vortex blocks of one tile.
constexpr int OFF_TILES = 8, OFF_SEGS = 128, OFF_RUN = 5;
static_assert(OFF_SEGS * OFF_RUN >= BIN_MAX_BLOCKS && BIN_MAX_BLOCKS <= 1024, "k_offsets covers every block");
static_assert(OFF_TILES * OFF_SEGS == 1024, "k_offsets runs 1024 threads");

__device__ __forceinline__ int warp_incl_scan(int v, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    return v;
}

// Per-tile totals and per-(block, tile) offsets within the tile: tile_count
// and, in place over the block histograms, off[b][t] = sum_{b' < b} hist[b'][t].
// Blocks are independent (the tiles' first slots are added by the scatter pass).
__global__ void __launch_bounds__(1024) k_offsets(int ntiles, int nb, int* __restrict__ hist_off,
                                                  unsigned* __restrict__ tile_count, const double* __restrict__ gmax_blk,
                                                  double* __restrict__ gmax_all) {
    __shared__ int part[OFF_SEGS][OFF_TILES + 1];
    __shared__ double wmax[32];
    const int tx = threadIdx.x % OFF_TILES, ty = threadIdx.x / OFF_TILES;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int t0 = blockIdx.x * OFF_TILES, t = t0 + tx;
    const int S = (nb + OFF_SEGS - 1) / OFF_SEGS;   // <= OFF_RUN
    const int b0 = ty * S;
    pdl_wait();
    // block 0: the largest |Gamma| over the locate blocks, one load a thread
    // (nb <= 1024), issued with the histogram loads and reduced after them
    double gm = blockIdx.x == 0 && (int)threadIdx.x < nb ? gmax_blk[threadIdx.x] : 0.0;
    int v[OFF_RUN];
    int seg = 0;
#pragma unroll
    for (int k = 0; k < OFF_RUN; ++k) {              // all loads in flight together (clamped index)
        const bool in = k < S && b0 + k < nb && t < ntiles;
        v[k] = nb > 0 ? hist_off[in ? (size_t)(b0 + k) * ntiles + t : 0] : 0;
        v[k] = in ? v[k] : 0;
        seg += v[k];
    }
    if (blockIdx.x == 0) {                           // block-uniform
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
        if (lane == 0) wmax[wid] = gm;
    }
    part[ty][tx] = seg;
    __syncthreads();
    if (blockIdx.x == 0 && wid == OFF_TILES) {       // OFF_TILES < 32: a warp that scans nothing
        double m = wmax[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) *gmax_all = m;
    }
    if (wid < OFF_TILES) {                            // exclusive scan over the runs of tile t0 + wid
        const int a0 = part[4 * lane][wid], a1 = part[4 * lane + 1][wid];
        const int a2 = part[4 * lane + 2][wid], a3 = part[4 * lane + 3][wid];
        const int sum4 = a0 + a1 + a2 + a3;
        const int incl = warp_incl_scan(sum4, lane);
        const int ex = incl - sum4;
        part[4 * lane][wid] = ex;
        part[4 * lane + 1][wid] = ex + a0;
        part[4 * lane + 2][wid] = ex + a0 + a1;
        part[4 * lane + 3][wid] = ex + a0 + a1 + a2;
        if (lane == 31 && t0 + wid < ntiles) tile_count[t0 + wid] = (unsigned)incl;
    }
    __syncthreads();
    if (t < ntiles) {
        int run = part[ty][tx];
#pragma unroll
        for (int k = 0; k < OFF_RUN; ++k) {
            if (k < S && b0 + k < nb) hist_off[(size_t)(b0 + k) * ntiles + t] = run;
            run += v[k];
        }
    }
}

// Every block scans the tile totals itself (block 0 publishes the tiles' first
// slots for the deposit and interpolation passes), adds them to its offsets
// and places its records.
constexpr int SCAN_PER = 16;     // tiles per thread in the block scan: 256 * 16 = 64 * 64 tiles at most
// vortices a thread loads at a time: at 1024 threads the eight FP32 records
// spill (64 registers at most), so four (FP64: four and two)
template <typename T, int NT> struct ScatterUnroll {
    static constexpr int value = (sizeof(T) == 4 ? 8 : 4) / (NT == 1024 ? 2 : 1);
};
static_assert((2048 / BIN_TILE) * (2048 / BIN_TILE) <= BIN_THREADS * SCAN_PER, "scan covers every tile");
constexpr int MAX_SCAN_TILES = BIN_THREADS * SCAN_PER;   // smaller tiles are offered only up to this count

template <typename T, int TILE, int NT>
__global__ void __launch_bounds__(NT, NT == 1024 ? 1 : 4) k_scatter(const Pos<T>* __restrict__ pos, int64_t nv, int64_t span,
                                                        const int64_t* __restrict__ dn, int min_span, int max_blocks,
                                                        Geo geo, const int* __restrict__ off,
                                                        const unsigned* __restrict__ tile_count,
                                                        int* __restrict__ tile_start, Rec<T>* __restrict__ recs,
                                                        int64_t rec_cap, int* __restrict__ status) {
    extern __shared__ unsigned sm[];
    __shared__ int wsum[NT / 32];
    unsigned* cnt = sm;
    int* first = (int*)(sm + geo.ntiles);
    pdl_wait();
    bin_count(dn, min_span, max_blocks, nv, span);
    const int64_t lo = (int64_t)blockIdx.x * span;
    const int64_t hi = lo + span < nv ? lo + span : nv;
    // this thread's first records (in flight during the scan)
    Pos<T> p[ScatterUnroll<T, NT>::value];
#pragma unroll
    for (int k = 0; k < ScatterUnroll<T, NT>::value; ++k) {     // clamped loads; past the end: no vortex
        const int64_t q = lo + k * NT + threadIdx.x;
        p[k] = pos[q < hi ? q : (hi > 0 ? hi - 1 : 0)];
        if (q >= hi) make_pos(p[k], 0xFFFF, 0xFFFF, Frac<T>(0), Frac<T>(0), 0.0);
    }
    // exclusive scan of tile_count: thread i owns tiles [i * per, i * per + per)
    const int per = (geo.ntiles + NT - 1) / NT;   // <= SCAN_PER
    const int t0 = threadIdx.x * per;
    int mine = 0;
#pragma unroll
    for (int k = 0; k < SCAN_PER; ++k)
        if (k < per && t0 + k < geo.ntiles) mine += (int)tile_count[t0 + k];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    int run = incl - mine;
    for (int w = 0; w < wid; ++w) run += wsum[w];
    const int* row = off + (size_t)blockIdx.x * geo.ntiles;
#pragma unroll
    for (int k = 0; k < SCAN_PER; ++k) {
        const int i = t0 + k;
        if (k < per && i < geo.ntiles) {
            cnt[i] = 0u;
            first[i] = run + row[i];
            if (blockIdx.x == 0) tile_start[i] = run;
            run += (int)tile_count[i];
        }
    }
    __syncthreads();
    for (int64_t base = lo; base < hi; base += NT * ScatterUnroll<T, NT>::value) {
        if (base != lo) {
#pragma unroll
            for (int k = 0; k < ScatterUnroll<T, NT>::value; ++k) {     // loads first (clamped)
                const int64_t q = base + k * NT + threadIdx.x;
                p[k] = pos[q < hi ? q : hi - 1];
                if (q >= hi) make_pos(p[k], 0xFFFF, 0xFFFF, Frac<T>(0), Frac<T>(0), 0.0);
            }
        }
#pragma unroll
        for (int k = 0; k < ScatterUnroll<T, NT>::value; ++k) {
            const int ci = pos_ci(p[k]), cj = pos_cj(p[k]);
            if (ci == 0xFFFF) continue;
            const int64_t q = base + k * NT + threadIdx.x;
            // Up to four tiles, each its own predicated code: in loops over
            // them the lanes of a warp went as many rounds as the one with
            // most (1e6 vortices on 1024^2: locate 11.6 -> 10.9, scatter 11.1 ->
            // 10.6 us; 4e6 on 2048 x 1800: locate 34 -> 31)
            const int tx0 = (ci - 1) / TILE, tx1 = (ci + 2) / TILE;
            const int ty0 = (cj - 1) / TILE, ty1 = (cj + 2) / TILE;
            const int t0 = ty0 * geo.ntx + tx0;
            const bool px = tx1 > tx0, py = ty1 > ty0;
            const auto take = [&](int t) { return first[t] + (int)atomicAdd(&cnt[t], 1u); };
            const auto put = [&](int slot, int tx, int ty) {
                if (slot < 0 || slot >= rec_cap) atomicOr(status, ST_INTERNAL);   // counts and histograms disagree
                else recs[slot] = make_rec(p[k], ci - tx * TILE, cj - ty * TILE, (int)q);
            };
            const int s0 = take(t0);
            const int s1 = px ? take(t0 + 1) : 0;
            const int s2 = py ? take(t0 + geo.ntx) : 0;
            put(s0, tx0, ty0);
            if (px) put(s1, tx1, ty0);
            if (py) put(s2, tx0, ty1);
            if (px && py) put(take(t0 + geo.ntx + 1), tx1, ty1);
        }
    }
}

// One-pass binning of the mixed path's middling sets: at most RUN_MAX blocks, each
// of which locates its span of vortices (their cells stay in shared memory),
// counts and scans its own tiles, and writes its records in tile order into its
// own stretch of the record array, four slots a vortex.  table[b][t] holds the
// run of tile t in block b: first slot | records << 16.  The deposit and E_v
// blocks find a tile's records by a search over the runs (RunRecs).  The three
// passes of larger sets take as many launches of 3 to 6 us whatever the count
// (a velocity of 5,000 vortices on 1024^2 65.2 -> 58.0 us, of 20,011 on 700 x 333
// 46.7 -> 39.5, of 65,000 on 300 x 200 46.8 -> 43.6; of 131,000, whose 32 blocks
// bind, 57.0 -> 55.9).  More and so shorter runs lose: with 304 blocks, each
// record's run found by a scan, 1e6 vortices on 1024^2 took 109 us against 103.
template <int TILE>
__global__ void __launch_bounds__(RUN_THREADS) k_bin_runs(const double* __restrict__ X, const double* __restrict__ Y,
                                                             const double* __restrict__ G, int64_t nv, int span,
                                                             const int64_t* __restrict__ dn, Geo geo,
                                                             Rec<float>* __restrict__ recs, unsigned* __restrict__ table,
                                                             double* __restrict__ gmax_blk, int* __restrict__ status,
                                                             unsigned long long* __restrict__ oob, float* __restrict__ zu,
                                                             float* __restrict__ zv) {
    extern __shared__ __align__(16) unsigned char run_dyn[];
    __shared__ float wmax[RUN_THREADS / 32];
    __shared__ int wsum[RUN_THREADS / 32];
    Pos<float>* cells = reinterpret_cast<Pos<float>*>(run_dyn);
    unsigned* cnt = reinterpret_cast<unsigned*>(cells + span);
    for (int i = threadIdx.x; i < geo.ntiles; i += RUN_THREADS) cnt[i] = 0u;
    pdl_wait();
    if (dn) nv = *dn < nv ? *dn : nv;
    const int64_t lo = (int64_t)blockIdx.x * span;
    const int n = (int)(lo >= nv ? 0 : (nv - lo < span ? nv - lo : span));
    __syncthreads();
    float gm = 0.f;
    int bad = 0;
    for (int base = 0; base < n; base += RUN_THREADS * BIN_UNROLL) {
        double xs[BIN_UNROLL], ys[BIN_UNROLL], gs[BIN_UNROLL];
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {   // clamped: a thread past the end reloads the last vortex
            int i = base + k * RUN_THREADS + threadIdx.x;
            i = i < n ? i : n - 1;
            xs[k] = X[lo + i];
            ys[k] = Y[lo + i];
            gs[k] = G[lo + i];
        }
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {
            const int i = base + k * RUN_THREADS + threadIdx.x;
            if (i >= n) break;
            int ci = 0, cj = 0;
            unsigned fx = 0, fy = 0;
            Pos<float> p;
            if (!loc_split(xs[k], geo, 0, ci, fx) || !loc_split(ys[k], geo, 1, cj, fy)) {
                ++bad;
                make_pos(p, 0xFFFF, 0xFFFF, 0u, 0u, 0.0);   // marker: no record
                cells[i] = p;
                if (zu) {
                    zu[lo + i] = 0.f;
                    zv[lo + i] = 0.f;
                }
                continue;
            }
            make_pos(p, ci, cj, fx, fy, gs[k]);
            cells[i] = p;                            // read back by this thread
            gm = abs_max(gm, p.g);
            const int tx0 = (ci - 1) / TILE, tx1 = (ci + 2) / TILE;
            const int ty0 = (cj - 1) / TILE, ty1 = (cj + 2) / TILE;
            const int t0 = ty0 * geo.ntx + tx0;
            const bool px = tx1 > tx0, py = ty1 > ty0;
            atomicAdd(&cnt[t0], 1u);
            if (px) atomicAdd(&cnt[t0 + 1], 1u);
            if (py) atomicAdd(&cnt[t0 + geo.ntx], 1u);
            if (px && py) atomicAdd(&cnt[t0 + geo.ntx + 1], 1u);
        }
    }
    if (bad) {
        atomicAdd(oob, (unsigned long long)bad);
        atomicOr(status, ST_OUT_OF_DOMAIN);
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    gm = no_nan(gm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if (lane == 0) wmax[wid] = gm;
    __syncthreads();
    // exclusive scan of the counts: a thread owns `per` tiles
    const int per = (geo.ntiles + RUN_THREADS - 1) / RUN_THREADS, t0 = threadIdx.x * per;
    const int t1 = t0 + per < geo.ntiles ? t0 + per : geo.ntiles;
    int sum = 0;
    for (int i = t0; i < t1; ++i) sum += (int)cnt[i];
    const int incl = warp_incl_scan(sum, lane);
    if (lane == 31) wsum[wid] = incl;
    if (threadIdx.x == 0) {
        float m = 0.f;
        for (int i = 0; i < RUN_THREADS / 32; ++i) m = fmax(m, wmax[i]);
        gmax_blk[blockIdx.x] = (double)m;
    }
    __syncthreads();
    unsigned run = (unsigned)(incl - sum);
    for (int w = 0; w < wid; ++w) run += (unsigned)wsum[w];
    unsigned* row = table + (size_t)blockIdx.x * geo.ntiles;
    for (int i = t0; i < t1; ++i) {
        const unsigned c = cnt[i];
        row[i] = run | (c << 16);
        cnt[i] = run;
        run += c;
    }
    __syncthreads();
    Rec<float>* out = recs + 4 * lo;
    for (int i = threadIdx.x; i < n; i += RUN_THREADS) {
        const Pos<float> p = cells[i];
        const int ci = pos_ci(p), cj = pos_cj(p);
        if (ci == 0xFFFF) continue;
        const int tx0 = (ci - 1) / TILE, tx1 = (ci + 2) / TILE;
        const int ty0 = (cj - 1) / TILE, ty1 = (cj + 2) / TILE;
        for (int ty = ty0; ty <= ty1; ++ty)
            for (int tx = tx0; tx <= tx1; ++tx)
                out[atomicAdd(&cnt[ty * geo.ntx + tx], 1u)] = make_rec(p, ci - tx * TILE, cj - ty * TILE, (int)(lo + i));
    }
}

// fixed-point scale 2^sh as a floating-point number, sh in [-60, 100]
template <typename T> __device__ __forceinline__ T pow2(int sh);
template <> __device__ __forceinline__ float pow2<float>(int sh) { return __int_as_float((sh + 127) << 23); }

// x = hi 2^16 + lo + e, |lo| <= 2^15, |e| <= 1/2, for |x| < 2^38, with FP32
// adds only (no conversion instructions, which issue at 1/8 rate): added to
// 1.5 2^39, x leaves its multiple of 2^16, h, in the sum's low mantissa bits;
// x - h is exact, and added to 1.5 2^23 leaves its nearest integer there.
// (Splitting the product gy wx unrounded, by fused multiply-adds, is one
// operation less and a little more accurate, but other bits of w move a state
// of dense vortices by 2e-9 of its positions, which are FP64 results.)
// With sorted_slot 1e6 vortices on 1024^2 deposit in 20.0 us instead of 21.6,
// 4e6 on 2048 x 1800 in 61 instead of 67.  Other sorts measured: 2048 records
// at a time no faster; 128 by each warp alone, no barriers, a tenth slower.
__device__ __forceinline__ void split_hilo(float x, int& hi, int& lo) {
    const float t = __fadd_rn(x, 0x1.8p39f);
    hi = __float_as_int(t) - 0x53400000;
    lo = __float_as_int(__fadd_rn(__fsub_rn(x, __fsub_rn(t, 0x1.8p39f)), 0x1.8p23f)) - 0x4B400000;
}

// Deposit: one block per node tile accumulates its records in shared memory as
// fixed-point integers.  FP32 path: each term v 2^sh, rounded to an integer
// hi 2^16 + lo, goes into two native 32-bit shared adds (exact while the tile
// has fewer than 65536 records and |sum| < 2^38); otherwise, and for FP64, one
// 64-bit add.  Integer sums are exact, so the result does not depend on the
// order of the adds.  The scale bounds every node sum by the tile's record
// count times the largest |Gamma| of the whole regularization (reduced by
// k_offsets from the locate blocks' maxima).  If that is not finite, each tile
// looks through its records (tile_gmax): one that holds such a strength becomes NaN,
// the others go by their own largest.  (A one-add variant with a
// node-window bound measured no faster and lost seven bits on clustered
// vortices; shared adds are not what bounds this kernel.)
//
// A record's local cell (lx, ly) lies in [-2, TILE], so its nodes lie in
// [-3, TILE + 2]: the accumulator covers that range (acc_w^2 nodes) and the
// adds need no bounds tests; only the tile's own TILE x TILE nodes are written
// out.
constexpr int ACC_HALO = 3;
template <int TILE> struct AccW { static constexpr int value = TILE + 6; };

enum { DEP_SPLIT32 = 0, DEP_F32_64 = 1 };

// FP64 records: Gamma on the largest |Gamma|'s scale below 2^58, both weights
// applied in fixed point, the term rounded once to the tile's scale (drop bits
// less) and added as two 32-bit words, the low one's carry to the high one.
// (A 64-bit shared add is a compare-and-swap loop: 3.7 lanes a clock and SM
// against 11.7 for the two adds with the carry.)  1e6 vortices on 1024^2: 259
// us with FP64 products and 64-bit adds, 53 us.
template <int ACC_W>
__device__ __forceinline__ void deposit_one_fx(const Rec<double>& rc, int gexp, int drop, unsigned* acc_lo,
                                               unsigned* acc_hi) {
    FxSplit wx[4], wy[4];
    fx_m4p(rc.fx, wx);
    fx_m4p(rc.fy, wy);
    const FxSplit g = fx_split(fx_from_double(rc.g, gexp));
    const int base = (rec_ly(rc) - 1 + ACC_HALO) * ACC_W + (rec_lx(rc) - 1 + ACC_HALO);
    const long long half = (1ll << drop) >> 1, tie = drop ? -1ll : 0ll;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const FxSplit gy = fx_split(fx_weigh(g, wy[b]));
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int node = base + b * ACC_W + a;
            const long long y = fx_weigh(gy, wx[a]), x = (y + half + ((y >> 63) & tie)) >> drop;   // halves away from 0
            const unsigned lo = (unsigned)x, old = atomicAdd(&acc_lo[node], lo);
            atomicAdd(&acc_hi[node], (unsigned)(x >> 32) + (old + lo < old ? 1u : 0u));
        }
    }
}

template <int MODE, int ACC_W, typename T>
__device__ __forceinline__ void deposit_one(const Rec<T>& rc, T scale, unsigned long long* acc) {
    int* acc_hi = reinterpret_cast<int*>(acc);
    int* acc_lo = reinterpret_cast<int*>(acc) + ACC_W * ACC_W;
    T wx[4], wy[4];
    m4p_weights(rec_fx(rc), wx);
    m4p_weights(rec_fy(rc), wy);
    const T gs = rc.g * scale;
    const int base = (rec_ly(rc) - 1 + ACC_HALO) * ACC_W + (rec_lx(rc) - 1 + ACC_HALO);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const T gy = gs * wy[b];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int node = base + b * ACC_W + a;
            const T x = gy * wx[a];
            if (MODE == DEP_SPLIT32) {
                int hi, lo;
                split_hilo((float)x, hi, lo);
                atomicAdd(&acc_hi[node], hi);
                atomicAdd(&acc_lo[node], lo);
            } else {
                atomicAdd(&acc[node], (unsigned long long)__float2ll_rn((float)x));
            }
        }
    }
}

// The records of one tile: load() gives a thread U of them, blockDim apart (a
// thread past the end reloads the last record, which it then skips).  FlatRecs:
// a stretch of one array.
constexpr int REC_U = 4;
template <typename T> struct FlatRecs {
    const Rec<T>* recs;
    int cnt;
    template <int U> __device__ __forceinline__ void load(int r0, Rec<T> (&rc)[U]) const {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = r0 + u * (int)blockDim.x + (int)threadIdx.x;
            rc[u] = recs[r < cnt ? r : cnt - 1];
        }
    }
};
// The runs that k_bin_runs left for the tile: five halvings find a record's.
struct RunRecs {
    const Rec<float>* recs;
    const int2* runs;        // [RUN_MAX] records of the runs before; slot of the run's first record less that
    int cnt;
    template <int U> __device__ __forceinline__ void load(int r0, Rec<float> (&rc)[U]) const {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int r = min(r0 + u * (int)blockDim.x + (int)threadIdx.x, cnt - 1);
            int b = 0;                                   // the last run that begins at r or before
#pragma unroll
            for (int step = RUN_MAX / 2; step > 0; step >>= 1)
                if (runs[b + step].x <= r) b += step;
            rc[u] = recs[r + runs[b].y];
        }
    }
};

// Where a tile's records are: as k_scatter left them, or in runs
struct FlatBins {
    const int* tile_start;
    const unsigned* tile_count;
    const double* gmax;            // largest |Gamma|
    int64_t rec_cap;
};
struct RunBins {
    const unsigned* table;
    const double* gmax;            // that of each block
    int nb, region, ntiles;        // blocks, record slots of each
};

// The records of tile t and, with GMAX, the largest |Gamma|
template <bool GMAX, typename T>
__device__ __forceinline__ FlatRecs<T> open_tile(const FlatBins& bins, const Rec<T>* recs, int t, int* status,
                                                 double& gmax) {
    int start = bins.tile_start[t], cnt = (int)bins.tile_count[t];
    if (cnt != 0 && (start < 0 || cnt < 0 || (int64_t)start + cnt > bins.rec_cap)) {     // block-uniform
        if (threadIdx.x == 0) atomicOr(status, ST_INTERNAL);
        cnt = 0;
    }
    if (cnt == 0) start = 0;
    if (GMAX) gmax = *bins.gmax;
    return FlatRecs<T>{recs + start, cnt};
}
template <bool GMAX>
__device__ __forceinline__ RunRecs open_tile(const RunBins& bins, const Rec<float>* recs, int t, int* status,
                                             double& gmax) {
    static_assert(RUN_MAX == 32, "a run a lane");
    __shared__ int2 runs[RUN_MAX];
    __shared__ int total;
    __shared__ float top;
    if (threadIdx.x < 32) {
        const int b = threadIdx.x;
        const unsigned e = b < bins.nb ? bins.table[(size_t)b * bins.ntiles + t] : 0u;
        float gm = GMAX && b < bins.nb ? (float)bins.gmax[b] : 0.f;        // exact: a float
        const int slot = (int)(e & 0xFFFFu);
        int c = (int)(e >> 16);
        if (slot + c > bins.region) {                                    // not as the binning writes it
            atomicOr(status, ST_INTERNAL);
            c = 0;
        }
        const int incl = warp_incl_scan(c, b);
        runs[b] = make_int2(incl - c, b * bins.region + slot - (incl - c));
        if (b == 31) total = incl;
        if (GMAX) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) gm = fmaxf(gm, __shfl_xor_sync(0xffffffffu, gm, o));
            if (b == 0) top = gm;
        }
    }
    __syncthreads();
    if (GMAX) gmax = (double)top;
    return RunRecs{recs, runs, total};
}

// every record of the tile, given to `one`; rc holds this thread's first REC_U (src.load at 0)
template <typename T, typename SRC, typename F>
__device__ __forceinline__ void deposit_records(const SRC& src, Rec<T> (&rc)[REC_U], F one) {
    const int stride = REC_U * (int)blockDim.x, cnt = src.cnt;
    for (int r0 = 0; r0 < cnt; r0 += stride) {
        Rec<T> cur[REC_U];
#pragma unroll
        for (int u = 0; u < REC_U; ++u) cur[u] = rc[u];
        if (r0 + stride < cnt) src.load(r0 + stride, rc);
#pragma unroll
        for (int u = 0; u < REC_U; ++u)
            if (r0 + u * (int)blockDim.x + (int)threadIdx.x < cnt) one(cur[u]);
    }
}

// Split-32 deposit in bank order.  The shared adds of one warp instruction
// (the same stencil term of 32 records) conflict when two lanes' records put
// their stencils' first nodes in the same bank, which for records in random
// cells costs about 3.7 passes an add.  So each chunk of REC_U x blockDim
// records is first counting-sorted by that bank (one shared add a record
// into 32 counters), and lane l of row i takes sorted record l R + i (R rows
// of 32 in the chunk): the lanes of a row lie about one bucket, so one bank,
// apart.  The chunk is stored transposed (sorted record l R + i in slot
// 32 i + l) so a row reads 32 consecutive records.  Only the order of the
// integer adds changes, so the sums are those of the unsorted deposit.
constexpr int DEP_MAX_THREADS = 256;
constexpr int DEP_SORT_MIN = 256;     // fewer records: too few adds for the sort's three barriers to pay
constexpr int DEP_SORT_SLOTS = REC_U * DEP_MAX_THREADS + 32;

// Slot of sorted record idx < 32 R <= SORT_MAX: 32 (idx mod R) + idx / R.  The
// quotient is (idx m) >> 20 with m = floor(2^20 / R) + 1: m R exceeds 2^20 by at
// most R, and idx R < 2^20.  (The compiler's division by R cost a record some
// twenty of its four hundred instructions.)
constexpr int SORT_MAX = 1024;
struct SlotInv {
    unsigned m[SORT_MAX / 32 + 1];
    constexpr SlotInv() : m() {
        for (unsigned r = 1; r <= SORT_MAX / 32; ++r) m[r] = (1u << 20) / r + 1u;
    }
};
__constant__ constexpr SlotInv SLOT_INV;
__device__ __forceinline__ int sorted_slot(int idx, int R, unsigned inv) {
    const int q = (int)(((unsigned)idx * inv) >> 20);
    return 32 * (idx - q * R) + q;
}

template <int ACC_W, typename T, typename SRC>
__device__ __forceinline__ void deposit_records_banked(const SRC& src, T scale,
                                                       unsigned long long* acc, Rec<T> (&rc)[REC_U],
                                                       Rec<T>* srt, int* bcnt, int* bstart) {
    const int stride = REC_U * (int)blockDim.x, cnt = src.cnt;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
    for (int r0 = 0; r0 < cnt; r0 += stride) {
        const int n = cnt - r0 < stride ? cnt - r0 : stride;
        const int R = (n + 31) >> 5;
        const unsigned inv = SLOT_INV.m[R];
        int bank[REC_U], pos[REC_U];
#pragma unroll
        for (int u = 0; u < REC_U; ++u) {
            const int r = u * (int)blockDim.x + (int)threadIdx.x;     // index within the chunk
            bank[u] = ((rec_ly(rc[u]) - 1 + ACC_HALO) * ACC_W + (rec_lx(rc[u]) - 1 + ACC_HALO)) & 31;
            pos[u] = r < n ? atomicAdd(&bcnt[bank[u]], 1) : 0;
        }
        __syncthreads();
        if (wid == 0) {                               // bucket starts; counters cleared for the next chunk
            const int c = bcnt[lane];
            bstart[lane] = warp_incl_scan(c, lane) - c;
            bcnt[lane] = 0;
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < REC_U; ++u) {
            const int r = u * (int)blockDim.x + (int)threadIdx.x;
            if (r < n) {
                srt[sorted_slot(bstart[bank[u]] + pos[u], R, inv)] = rc[u];
            }
        }
        if (r0 + stride < cnt) src.load(r0 + stride, rc);   // the next chunk in flight
        __syncthreads();
        for (int i = wid; i < R; i += nw)
            if (lane * R + i < n) deposit_one<DEP_SPLIT32, ACC_W, T>(srt[i * 32 + lane], scale, acc);
        __syncthreads();                              // srt and the counters are reused
    }
}

// shared memory of one tile's deposit (SORT: with room for the bank-ordered chunk)
template <typename T, int TILE, bool SORT>
struct DepositSmem {
    unsigned long long acc[AccW<TILE>::value * AccW<TILE>::value];
    Rec<T> srt[SORT && sizeof(T) == 4 ? DEP_SORT_SLOTS : 1];
    int bcnt[32], bstart[32];
    unsigned long long top;    // tile_gmax: the largest finite |Gamma|'s bits, and whether there are others
    int bad;
};

template <typename T, int TILE, bool SORT>
__device__ __forceinline__ void deposit_clear(DepositSmem<T, TILE, SORT>& sm) {
    for (int i = threadIdx.x; i < AccW<TILE>::value * AccW<TILE>::value; i += blockDim.x) sm.acc[i] = 0ull;
    if (threadIdx.x < 32) sm.bcnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        sm.top = 0ull;
        sm.bad = 0;
    }
}

// the tile's largest finite |Gamma|; sm.bad is set if one of its strengths is not finite
template <typename T, int TILE, bool SORT, typename SRC>
__device__ __noinline__ double tile_gmax(const SRC src, DepositSmem<T, TILE, SORT>& sm) {
    __syncthreads();
    for (int r0 = 0; r0 < src.cnt; r0 += (int)blockDim.x) {
        Rec<T> rc[1];
        src.load(r0, rc);
        const double g = fabs((double)rc[0].g);
        if (g < INFINITY) atomicMax(&sm.top, (unsigned long long)__double_as_longlong(g));
        else sm.bad = 1;
    }
    __syncthreads();
    return __longlong_as_double((long long)sm.top);
}

// w of tile (tx, ty) from its records (global or shared memory); rc holds
// this thread's first ones, sm is cleared (the barrier is in here)
template <typename T, int TILE, bool SORT, typename SRC>
__device__ __forceinline__ void deposit_tile(const SRC& src, double gmax, const Geo& geo, int tx, int ty,
                                             T* __restrict__ w, DepositSmem<T, TILE, SORT>& sm, Rec<T> (&rc)[REC_U]) {
    constexpr int ACC_W = AccW<TILE>::value;
    const int cnt = src.cnt;
    unsigned long long* acc = sm.acc;
    if (__double2hiint(gmax) == 0x7FF00000) gmax = tile_gmax<T, TILE, SORT, SRC>(src, sm);     // an infinity; block-uniform
    if constexpr (sizeof(T) == 8) {
        // terms below 2^58 come drop bits finer than the sums, which stay below 2^63
        const int gf = (int)(__double_as_longlong(gmax) >> 52) & 0x7FF, gexp = gf ? gf : 1;
        const int drop = max(32 - __clz(cnt) - 5, 0);             // count < 2^(drop + 5)
        const int sh = -(fx_exp(gexp) + drop);
        unsigned* acc_lo = reinterpret_cast<unsigned*>(acc);
        unsigned* acc_hi = acc_lo + ACC_W * ACC_W;
        __syncthreads();
        deposit_records<T>(src, rc, [&](const Rec<T>& r) { deposit_one_fx<ACC_W>(r, gexp, drop, acc_lo, acc_hi); });
        __syncthreads();
        const double inv_dx2 = sm.bad ? (double)NAN : geo.inv_dx2;
        for (int i = threadIdx.x; i < TILE * TILE; i += blockDim.x) {
            const int lx = i % TILE, ly = i / TILE;
            const int gi = tx * TILE + lx, gj = ty * TILE + ly;
            const int node = (ly + ACC_HALO) * ACC_W + lx + ACC_HALO;
            if (gi < geo.nx && gj < geo.ny) {
                const long long a = (long long)(((unsigned long long)acc_hi[node] << 32) | acc_lo[node]);
                w[(size_t)gj * geo.nx + gi] = fx_to_double(a, -sh) * inv_dx2;
            }
        }
    } else {
        const bool split32 = cnt < 65536;
        const int sh = tile_shift_of((unsigned)cnt, gmax) - (split32 ? 23 : 0);   // 2^61 -> 2^38 when split
        const T scale = pow2<T>(sh);
        __syncthreads();
        if (SORT && split32 && cnt >= DEP_SORT_MIN)             // block-uniform
            deposit_records_banked<ACC_W, T>(src, scale, acc, rc, sm.srt, sm.bcnt, sm.bstart);
        else if (split32)
            deposit_records<T>(src, rc,
                               [&](const Rec<T>& r) { deposit_one<DEP_SPLIT32, ACC_W, T>(r, scale, acc); });
        else
            deposit_records<T>(src, rc,
                               [&](const Rec<T>& r) { deposit_one<DEP_F32_64, ACC_W, T>(r, scale, acc); });
        __syncthreads();
        const int* acc_hi = reinterpret_cast<const int*>(acc);
        const int* acc_lo = reinterpret_cast<const int*>(acc) + ACC_W * ACC_W;
        const float inv_dx2f = sm.bad ? NAN : (float)geo.inv_dx2;
        for (int i = threadIdx.x; i < TILE * TILE; i += blockDim.x) {
            const int lx = i % TILE, ly = i / TILE;
            const int gi = tx * TILE + lx, gj = ty * TILE + ly;
            const int node = (ly + ACC_HALO) * ACC_W + lx + ACC_HALO;
            if (gi < geo.nx && gj < geo.ny) {
                long long a;
                if (split32) a = (long long)acc_hi[node] * 65536ll + (long long)acc_lo[node];
                else a = (long long)acc[node];
                w[(size_t)gj * geo.nx + gi] = __ll2float_rn(a) * pow2<float>(-sh) * inv_dx2f;
            }
        }
    }
}

template <typename T, int TILE, typename BINS>
__global__ void __launch_bounds__(256) k_deposit(const Rec<T>* __restrict__ recs, BINS bins, Geo geo, T* __restrict__ w,
                                                 int* __restrict__ status) {
    __shared__ DepositSmem<T, TILE, true> sm;
    const int t = blockIdx.x;
    deposit_clear(sm);
    pdl_wait();
    double gmax;
    const auto src = open_tile<true>(bins, recs, t, status, gmax);
    Rec<T> rc[REC_U];
    if (src.cnt > 0) src.load(0, rc);                               // in flight across the barrier
    deposit_tile(src, gmax, geo, t % geo.ntx, t / geo.ntx, w, sm, rc);
}

// A bound sheet added to w with the deposit: the grid nodes of its 16 ns
// stencil entries, sorted, and dx^2 R_s f at each node's first entry.
struct SheetAdd {
    const int* node;
    const double* val;
    int n;                     // entries; 0: no sheet
};

// R_v of a small set in one launch: one block per tile reads every vortex,
// keeps the records of its own tile in shared memory (any order: the sums are
// integers) with the largest |Gamma| of all, and deposits them, bitwise as the
// binning passes and k_deposit do.  The four launches of those cost 15 us
// whatever the set's size; this one reads 24 nv bytes a tile from L2, which
// is less while tiles x nv is below DIRECT_WORK (256 vortices on 128^2: four
// launches of 15 us became one of 4, the whole velocity 26.1 -> 16.1 us; 2000 on
// 768 x 512, 7.7e5 tile reads: 18 -> 9 us).  With a sheet,
// the tile's nodes of R_s f are added after the vortices'.
template <typename T, int TILE>
__global__ void __launch_bounds__(256) k_deposit_direct(const double* __restrict__ X, const double* __restrict__ Y,
                                                        const double* __restrict__ G, int64_t nv,
                                                        const int64_t* __restrict__ dn, Geo geo, T* __restrict__ w,
                                                        SheetAdd sheet, int* __restrict__ status,
                                                        unsigned long long* __restrict__ oob) {
    __shared__ DepositSmem<T, TILE, false> sm;
    __shared__ T wmax[8];
    __shared__ int n;
    extern __shared__ __align__(16) unsigned char direct_dyn[];
    Rec<T>* list = reinterpret_cast<Rec<T>*>(direct_dyn);
    const int t = blockIdx.x, tx = t % geo.ntx, ty = t / geo.ntx;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    deposit_clear(sm);
    if (threadIdx.x == 0) n = 0;
    pdl_wait();
    if (dn) nv = *dn < nv ? *dn : nv;                // nv: the records the list holds
    __syncthreads();
    T gm = T(0);
    int bad = 0;
    for (int64_t base = 0; base < nv; base += 256 * BIN_UNROLL) {
        double xs[BIN_UNROLL], ys[BIN_UNROLL], gs[BIN_UNROLL];
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {       // clamped: a thread past the end reloads the last vortex
            int64_t q = base + k * 256 + threadIdx.x;
            q = q < nv ? q : nv - 1;
            xs[k] = X[q];
            ys[k] = Y[q];
            gs[k] = G[q];
        }
#pragma unroll
        for (int k = 0; k < BIN_UNROLL; ++k) {
            const int64_t q = base + k * 256 + threadIdx.x;
            if (base + k * 256 >= nv) break;         // block-uniform
            int ci = 0, cj = 0;
            Frac<T> fx = 0, fy = 0;
            const bool in = q < nv;
            const bool ok = loc_split(xs[k], geo, 0, ci, fx) && loc_split(ys[k], geo, 1, cj, fy);
            Pos<T> p;
            make_pos(p, ci, cj, fx, fy, gs[k]);
            if (in && !ok) ++bad;
            if (in && ok) gm = abs_max(gm, p.g);
            const bool mine = in && ok && (ci - 1) / TILE <= tx && tx <= (ci + 2) / TILE && (cj - 1) / TILE <= ty &&
                              ty <= (cj + 2) / TILE;
            const unsigned m = __ballot_sync(0xffffffffu, mine);
            if (m) {
                int b = 0;
                if (lane == 0) b = atomicAdd(&n, __popc(m));
                b = __shfl_sync(0xffffffffu, b, 0);
                if (mine) list[b + __popc(m & ((1u << lane) - 1u))] = make_rec(p, ci - tx * TILE, cj - ty * TILE, (int)q);
            }
        }
    }
    if (bad && t == 0) {
        atomicAdd(oob, (unsigned long long)bad);
        atomicOr(status, ST_OUT_OF_DOMAIN);
    }
    gm = no_nan(gm);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xffffffffu, gm, o));
    if (lane == 0) wmax[wid] = gm;
    __syncthreads();
    for (int i = 0; i < 8; ++i) gm = fmax(gm, wmax[i]);
    const int cnt = n;
    Rec<T> rc[REC_U];
    const FlatRecs<T> src{list, cnt};
    if (cnt > 0) src.load(0, rc);
    deposit_tile(src, (double)gm, geo, tx, ty, w, sm, rc);
    if (sheet.n == 0) return;
    __syncthreads();                                  // the tile's w is written
    for (int i = threadIdx.x; i < sheet.n; i += 256) {
        const int node = sheet.node[i], before = i > 0 ? sheet.node[i - 1] : -1;
        const double v = sheet.val[i];
        const int gj = node / geo.nx, gi = node - gj * geo.nx;
        if (gi / TILE == tx && gj / TILE == ty && node != before)
            w[node] = (T)((double)w[node] + v * geo.inv_dx2);
    }
}

// sets that take k_deposit_direct and k_interp_direct: their records fit the
// block's list, and the tiles' repeated reads cost less than binning
constexpr int64_t DIRECT_WORK = (int64_t)1 << 20;
template <typename T> constexpr int64_t direct_max() { return sizeof(T) == 4 ? 4096 : 2048; }

template <typename T>
__device__ __forceinline__ void gather16(const T* __restrict__ uv, int nx, int ci, int cj, T fx, T fy, T& su, T& sv) {
    T wx[4], wy[4];
    m4p_weights(fx, wx);
    m4p_weights(fy, wy);
    su = 0;
    sv = 0;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
        const T* row = uv + 2 * ((size_t)(cj - 1 + b) * nx + (ci - 1));
        T ru = 0, rv = 0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            ru += wx[a] * row[2 * a];
            rv += wx[a] * row[2 * a + 1];
        }
        su += wy[b] * ru;
        sv += wy[b] * rv;
    }
}

// E_v at the vortices of the last regularization, in tile order: one block per
// tile stages the (u, v) nodes its resident vortices can touch (the tile plus
// one node before and two after, per direction) in shared memory, then every
// record whose cell lies in the tile (each vortex has exactly one such record)
// gathers its 4x4 stencil there and writes its result at its original index.
//
// FP64: the patch is held in fixed point, each component below 2^58 of its own
// largest value (a stream along x leaves v its digits), as centred halves (16
// bytes a node, as the doubles), and the forty products of a record are integer
// multiply-adds (1e6 vortices on 1024^2: 227 -> 70 us, of which the second
// exponent is 3); a patch with an infinity or a NaN keeps its doubles and the FP64
// sums.
template <int TILE>
__global__ void __launch_bounds__(256) k_interp_tiles_f64(const Rec<double>* __restrict__ recs, FlatBins bins,
                                                          const double2* __restrict__ uv, Geo geo,
                                                          double* __restrict__ uq, double* __restrict__ vq, int64_t nq,
                                                          int* __restrict__ status) {
    constexpr int PATCH = TILE + 3;
    __shared__ int4 patch[PATCH * PATCH];
    __shared__ int top[2];
    const int t = blockIdx.x;
    if (threadIdx.x < 2) top[threadIdx.x] = 1;
    pdl_wait();
    double unused;
    const auto src = open_tile<false>(bins, recs, t, status, unused);
    const int cnt = src.cnt;
    if (cnt == 0) return;                             // block-uniform
    const int tx = t % geo.ntx, ty = t / geo.ntx;
    const int gi0 = tx * TILE - 1, gj0 = ty * TILE - 1;
    double2* patchd = reinterpret_cast<double2*>(patch);
    int eu = 1, ev = 1;
    for (int i = threadIdx.x; i < PATCH * PATCH; i += blockDim.x) {
        const int gi = gi0 + i % PATCH, gj = gj0 + i / PATCH;
        double2 v = make_double2(0.0, 0.0);
        if (gi >= 0 && gi < geo.nx && gj >= 0 && gj < geo.ny) v = uv[(size_t)gj * geo.nx + gi];
        patchd[i] = v;
        eu = max(eu, (__double2hiint(v.x) >> 20) & 0x7FF);
        ev = max(ev, (__double2hiint(v.y) >> 20) & 0x7FF);
    }
    __syncthreads();                                  // top is initialised
    eu = __reduce_max_sync(0xffffffffu, eu);
    ev = __reduce_max_sync(0xffffffffu, ev);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&top[0], eu);
        atomicMax(&top[1], ev);
    }
    __syncthreads();
    eu = top[0];
    ev = top[1];
    const bool finite = max(eu, ev) < 2047;           // block-uniform
    if (finite) {
        for (int i = threadIdx.x; i < PATCH * PATCH; i += blockDim.x) {       // each thread its own nodes, in place
            const double2 v = patchd[i];
            const FxSplit a = fx_split(fx_from_double(v.x, eu)), b = fx_split(fx_from_double(v.y, ev));
            patch[i] = make_int4(a.h, a.l, b.h, b.l);
        }
        __syncthreads();
    }
    constexpr int U = 2;
    for (int r0 = 0; r0 < cnt; r0 += U * blockDim.x) {
        Rec<double> rc[U];
        bool ok[U];
        src.load(r0, rc);
#pragma unroll
        for (int u = 0; u < U; ++u) ok[u] = r0 + u * (int)blockDim.x + (int)threadIdx.x < cnt;
#pragma unroll 1
        for (int u = 0; u < U; ++u) {
            const Rec<double> c = u == 0 ? rc[0] : rc[1];
            const int lx = rec_lx(c), ly = rec_ly(c);
            if (!(u == 0 ? ok[0] : ok[1]) || lx < 0 || lx >= TILE || ly < 0 || ly >= TILE) continue;   // not home
            double ou, ov;
            if (finite) {
                FxSplit wx[4], wy[4];
                fx_m4p(c.fx, wx);
                fx_m4p(c.fy, wy);
                long long su = 0, sv = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int4* row = patch + (ly + b) * PATCH + lx;    // node (lx - 1 + a, ly - 1 + b)
                    long long hu = 0, hv = 0, tu = 1ll << 29, tv = 1ll << 29;
#pragma unroll
                    for (int a = 0; a < 4; ++a) {
                        const int4 q = row[a];
                        hu += fx_mw(q.x, wx[a].h);
                        tu += fx_mw(q.x, wx[a].l) + fx_mw(q.y, wx[a].h);
                        hv += fx_mw(q.z, wx[a].h);
                        tv += fx_mw(q.z, wx[a].l) + fx_mw(q.w, wx[a].h);
                    }
                    su += fx_weigh(fx_split((hu << 1) + (tu >> 30)), wy[b]);
                    sv += fx_weigh(fx_split((hv << 1) + (tv >> 30)), wy[b]);
                }
                ou = fx_to_double(su, fx_exp(eu));
                ov = fx_to_double(sv, fx_exp(ev));
            } else {
                double wx[4], wy[4];
                m4p_weights(c.fx, wx);
                m4p_weights(c.fy, wy);
                ou = ov = 0.0;
                for (int b = 0; b < 4; ++b) {
                    const double2* row = patchd + (ly + b) * PATCH + lx;
                    double ru = 0.0, rv = 0.0;
                    for (int a = 0; a < 4; ++a) {
                        ru += wx[a] * row[a].x;
                        rv += wx[a] * row[a].y;
                    }
                    ou += wy[b] * ru;
                    ov += wy[b] * rv;
                }
            }
            if (c.q < 0 || c.q >= nq) {
                atomicOr(status, ST_INTERNAL);
                continue;
            }
            uq[c.q] = ou;
            vq[c.q] = ov;
        }
    }
}

// FP32 variant that reads each stencil row with two 16-byte
// shared loads: the patch is staged twice as node pairs, starting at even and
// at odd local x, so that the four nodes px .. px + 3 of a row are the pairs
// E[px / 2], E[px / 2 + 1] (px even) or O[(px - 1) / 2], O[(px + 1) / 2].
//
// The home records of each chunk of REC_U x blockDim records are counting-
// sorted by the shared-memory bank of their first patch row (as the deposit's
// records are, same transposed layout), so the eight lanes of each quarter-
// warp, whose 16-byte loads are served together, read eight different bank
// groups; non-home records (a vortex's other tiles) drop out in the same pass.
// U records a thread a chunk.  Dynamic shared memory: (U x blockDim + 32)
// records.  Five blocks an SM (48 registers): with 64 registers, so four, 1e6
// vortices on 1024^2 took 22.4 us instead of 20.5.
template <int TILE> struct InterpSmem {
    static constexpr int PATCH = TILE + 3, PAIRS = (PATCH + 1) / 2;   // 18 pairs per patch row at TILE 32
    float4 pe[PATCH * PAIRS];
    float4 po[PATCH * PAIRS];
    int bcnt[32], bstart[32], nhome;
};

// The tile's patch; a barrier follows it
template <int TILE>
__device__ __forceinline__ void stage_patch(InterpSmem<TILE>& sm, const float2* __restrict__ uv, const Geo& geo, int tx,
                                            int ty) {
    constexpr int PATCH = InterpSmem<TILE>::PATCH, PAIRS = InterpSmem<TILE>::PAIRS;
    if (threadIdx.x < 32) sm.bcnt[threadIdx.x] = 0;
    const int gi0 = tx * TILE - 1, gj0 = ty * TILE - 1;
    // patch nodes px, py in [0, 2 PAIRS) x [0, PATCH); px = 2 PAIRS - 1 only pads
    for (int i = threadIdx.x; i < PATCH * 2 * PAIRS; i += blockDim.x) {
        const int px = i % (2 * PAIRS), py = i / (2 * PAIRS);
        const int gi = gi0 + px, gj = gj0 + py;
        float2 v = make_float2(0.f, 0.f);
        if (px < PATCH && gi >= 0 && gi < geo.nx && gj >= 0 && gj < geo.ny) v = uv[(size_t)gj * geo.nx + gi];
        float* e = reinterpret_cast<float*>(&sm.pe[py * PAIRS + px / 2]) + 2 * (px & 1);
        e[0] = v.x;
        e[1] = v.y;
        if (px >= 1) {
            float* o = reinterpret_cast<float*>(&sm.po[py * PAIRS + (px - 1) / 2]) + 2 * ((px - 1) & 1);
            o[0] = v.x;
            o[1] = v.y;
        }
    }
}

// one(record, u, v, place) for each home record: place counts them up without
// gaps, a row of lanes on end.  rc: the thread's first U; srt: U x blockDim + 32.
// Returns their number.  CHAIN: a row's four terms added from the left, fused;
// a state's FP64 positions follow these bits.
template <int TILE, bool CHAIN, int U, typename SRC, typename F>
__device__ __forceinline__ int interp_home_records(InterpSmem<TILE>& sm, const SRC& src, Rec<float> (&rc)[U],
                                                   Rec<float>* srt, F one) {
    constexpr int PAIRS = InterpSmem<TILE>::PAIRS;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)blockDim.x >> 5;
    const int stride = U * (int)blockDim.x, cnt = src.cnt;
    int seen = 0;
    for (int r0 = 0; r0 < cnt; r0 += stride) {
        const int n = cnt - r0 < stride ? cnt - r0 : stride;
        int key[U], pos[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int lx = rec_lx(rc[u]), ly = rec_ly(rc[u]);
            const bool home = u * (int)blockDim.x + (int)threadIdx.x < n && lx >= 0 && lx < TILE && ly >= 0 &&
                              ly < TILE;
            const float4* row = ((lx & 1) ? sm.po + (lx - 1) / 2 : sm.pe + lx / 2) + ly * PAIRS;
            key[u] = home ? (int)((__cvta_generic_to_shared(row) >> 4) & 31) : -1;
            pos[u] = home ? atomicAdd(&sm.bcnt[key[u]], 1) : 0;
        }
        __syncthreads();
        if (wid == 0) {                               // bucket starts; counters cleared for the next chunk
            const int c = sm.bcnt[lane];
            const int incl = warp_incl_scan(c, lane);
            sm.bstart[lane] = incl - c;
            sm.bcnt[lane] = 0;
            if (lane == 31) sm.nhome = incl;
        }
        __syncthreads();
        const int nh = sm.nhome, R = (nh + 31) >> 5;
        const unsigned inv = SLOT_INV.m[R];
        // row i holds full + (i < more) records, from lane 0 on
        const int full = (int)(((unsigned)nh * inv) >> 20), more = nh - full * R;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (key[u] >= 0) {
                srt[sorted_slot(sm.bstart[key[u]] + pos[u], R, inv)] = rc[u];
            }
        }
        if (r0 + stride < cnt) src.load(r0 + stride, rc);   // the next chunk in flight
        __syncthreads();
        for (int i = wid; i < R; i += nw) {
            if (lane * R + i >= nh) continue;
            const Rec<float> rcu = srt[i * 32 + lane];
            const int lx = rec_lx(rcu), ly = rec_ly(rcu);
            float wx[4], wy[4];
            m4p_weights(rec_fx(rcu), wx);
            m4p_weights(rec_fy(rcu), wy);
            const float4* rows = (lx & 1) ? sm.po + (lx - 1) / 2 : sm.pe + lx / 2;   // node px = lx is the first
            float su = 0.f, sv = 0.f;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const float4 p0 = rows[(ly + b) * PAIRS], p1 = rows[(ly + b) * PAIRS + 1];
                float ru, rv;
                if (CHAIN) {
                    ru = __fmaf_rn(wx[3], p1.z, __fmaf_rn(wx[2], p1.x, __fmaf_rn(wx[1], p0.z, __fmul_rn(wx[0], p0.x))));
                    rv = __fmaf_rn(wx[3], p1.w, __fmaf_rn(wx[2], p1.y, __fmaf_rn(wx[1], p0.w, __fmul_rn(wx[0], p0.y))));
                } else {
                    ru = wx[0] * p0.x + wx[1] * p0.z + wx[2] * p1.x + wx[3] * p1.z;
                    rv = wx[0] * p0.y + wx[1] * p0.w + wx[2] * p1.y + wx[3] * p1.w;
                }
                su += wy[b] * ru;
                sv += wy[b] * rv;
            }
            one(rcu, su, sv, seen + i * full + min(i, more) + lane);
        }
        seen += nh;
        __syncthreads();                              // srt and the counters are reused
    }
    return seen;
}

template <int TILE, int U, typename BINS>
__global__ void __launch_bounds__(256, 5) k_interp_tiles_f32(const Rec<float>* __restrict__ recs, BINS bins,
                                                          const float2* __restrict__ uv, Geo geo,
                                                          float* __restrict__ uq, float* __restrict__ vq, int64_t nq,
                                                          int* __restrict__ status) {
    __shared__ InterpSmem<TILE> sm;
    extern __shared__ __align__(16) unsigned char interp_dyn[];
    const int t = blockIdx.x;
    pdl_wait();
    double unused;
    const auto src = open_tile<false>(bins, recs, t, status, unused);
    if (src.cnt == 0) return;                     // block-uniform
    Rec<float> rc[U];
    src.load(0, rc);                              // in flight while the patch is staged
    stage_patch<TILE>(sm, uv, geo, t % geo.ntx, t / geo.ntx);
    __syncthreads();
    interp_home_records<TILE, false>(sm, src, rc, reinterpret_cast<Rec<float>*>(interp_dyn),
                              [&](const Rec<float>& r, float su, float sv, int) {
                                  if (r.q < 0 || r.q >= nq) {
                                      atomicOr(status, ST_INTERNAL);
                                      return;
                                  }
                                  uq[r.q] = su;
                                  vq[r.q] = sv;
                              });
}

// E_v at arbitrary points, FP64: a thread a point.
__global__ void __launch_bounds__(256) k_interp_xy_f64(const double* __restrict__ uv, const double* __restrict__ X,
                                                       const double* __restrict__ Y, int64_t nq, Geo geo,
                                                       double* __restrict__ uq, double* __restrict__ vq,
                                                       int* __restrict__ status, unsigned long long* __restrict__ oob) {
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < nq; q += (int64_t)gridDim.x * blockDim.x) {
        int ci = 0, cj = 0;
        double fx = 0, fy = 0, su = 0, sv = 0;
        if (loc_split(X[q], geo, 0, ci, fx) && loc_split(Y[q], geo, 1, cj, fy)) {
            gather16<double>(uv, geo.nx, ci, cj, fx, fy, su, sv);
        } else {
            atomicAdd(oob, 1ull);
            atomicOr(status, ST_OUT_OF_DOMAIN);
        }
        uq[q] = su;
        vq[q] = sv;
    }
}

// FP32: a warp takes 32 points.  Cells and weights are formed by a thread a
// point and left in shared memory; then eight lanes a point, four points at a
// time, gather one half row of the stencil each.  The pass is bound by the L1
// lookups of its scattered loads, one a distinct line and instruction: a
// thread a point makes 16 a point, half rows 8 (200,003 points on 768 x 512:
// 16.6 -> 12.3 us between events).
constexpr int XY_THREADS = 128;
struct XyPoint {
    float wx[4], wy[4];
    int at;                    // first node of the stencil; -1: off the grid
    float u, v;
    int pad;
};
// PAIRS: uv lies on 8-byte boundaries and a node is one load; a caller's field that starts on an odd word is read by words.
template <bool PAIRS> __device__ __forceinline__ float2 load_node(const float* __restrict__ p) {
    if constexpr (PAIRS) return __ldg(reinterpret_cast<const float2*>(p));
    else return make_float2(__ldg(p), __ldg(p + 1));
}
template <bool PAIRS>
__global__ void __launch_bounds__(XY_THREADS) k_interp_xy_f32(const float* __restrict__ uv, const double* __restrict__ X,
                                                              const double* __restrict__ Y, int64_t nq, Geo geo,
                                                              float* __restrict__ uq, float* __restrict__ vq,
                                                              int* __restrict__ status, unsigned long long* __restrict__ oob) {
    __shared__ __align__(16) XyPoint pts[XY_THREADS];
    const int lane = threadIdx.x & 31, col = lane & 3, pair = (lane >> 2) & 1;
    XyPoint* mine = pts + (threadIdx.x & ~31);
    pdl_wait();
    for (int64_t q0 = ((int64_t)blockIdx.x * XY_THREADS + threadIdx.x) - lane; q0 < nq; q0 += (int64_t)gridDim.x * XY_THREADS) {
        const int64_t q = q0 + lane;
        {
            XyPoint p;
            int ci = 0, cj = 0;
            float fx = 0.f, fy = 0.f;
            const bool ok = q < nq && split(X[q], geo.x0, geo.dx, geo.inv_dx, geo.cx, geo.nx, geo.xlim, ci, fx) &&
                            split(Y[q], geo.y0, geo.dx, geo.inv_dx, geo.cy, geo.ny, geo.ylim, cj, fy);
            if (q < nq && !ok) {
                atomicAdd(oob, 1ull);
                atomicOr(status, ST_OUT_OF_DOMAIN);
            }
            m4p_weights(ok ? fx : 0.f, p.wx);
            m4p_weights(ok ? fy : 0.f, p.wy);
            p.at = ok ? (cj - 1) * geo.nx + ci - 1 : -1;
            p.u = p.v = 0.f;
            mine[lane] = p;
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const XyPoint& p = mine[4 * i + (lane >> 3)];
            const int at = p.at;
            float2 a = make_float2(0.f, 0.f), b = a;
            if (at >= 0) {
                const float* r = uv + 2 * ((size_t)at + 2 * pair * geo.nx + col);
                a = load_node<PAIRS>(r);
                b = load_node<PAIRS>(r + 2 * geo.nx);
            }
            const float2 w = *reinterpret_cast<const float2*>(p.wy + 2 * pair);
            const float wx = p.wx[col];
            float su = wx * (w.x * a.x + w.y * b.x), sv = wx * (w.x * a.y + w.y * b.y);
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) {
                su += __shfl_xor_sync(0xffffffffu, su, o);
                sv += __shfl_xor_sync(0xffffffffu, sv, o);
            }
            if ((lane & 7) == 0) {
                mine[4 * i + (lane >> 3)].u = su;
                mine[4 * i + (lane >> 3)].v = sv;
            }
        }
        __syncwarp();
        if (q < nq) {
            uq[q] = mine[lane].u;
            vq[q] = mine[lane].v;
        }
        __syncwarp();
    }
}

// E_v of a small set at its own vortices, without binned records: four threads
// a vortex, one stencil row each (the rows' loads are in flight together),
// added in pairs; the position update of a time step in the same launch.  A
// vortex off the grid has velocity zero (and was counted by R_v).
template <typename T>
__global__ void __launch_bounds__(128) k_interp_direct(const C_t<T>* __restrict__ uv, const double* X, const double* Y,
                                                       int64_t nq, const int64_t* __restrict__ dn, Geo geo, T* uq, T* vq,
                                                       AdvanceArgs adv) {
    const int64_t q0 = (blockIdx.x * (int64_t)128 + threadIdx.x) >> 2;
    const int b = threadIdx.x & 3;
    pdl_wait();
    if (dn) nq = *dn < nq ? *dn : nq;
    const int64_t q = q0 < nq ? q0 : nq - 1;          // whole warps take part in the shuffles
    if (nq <= 0) return;
    const double x = X[q], y = Y[q];
    int ci = 1, cj = 1;
    T fx = 0, fy = 0;
    const bool ok = split_rec(x, geo, 0, ci, fx) && split_rec(y, geo, 1, cj, fy);
    if (!ok) { ci = 1; cj = 1; fx = 0; fy = 0; }
    T wx[4], wy[4];
    m4p_weights(fx, wx);
    m4p_weights(fy, wy);
    const C_t<T>* row = uv + (size_t)(cj - 1 + b) * geo.nx + (ci - 1);
    T su = 0, sv = 0;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        const C_t<T> c = row[a];
        su += wx[a] * c.x;
        sv += wx[a] * c.y;
    }
    const T wb = b == 0 ? wy[0] : b == 1 ? wy[1] : b == 2 ? wy[2] : wy[3];
    su *= wb;
    sv *= wb;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
        su += __shfl_xor_sync(0xffffffffu, su, o);
        sv += __shfl_xor_sync(0xffffffffu, sv, o);
    }
    if (b != 0 || q0 >= nq) return;
    if (!ok) su = sv = T(0);
    if (uq) {
        uq[q] = su;
        vq[q] = sv;
    }
    if (adv.kind == ADV_EULER) {
        adv.X[q] = x + adv.dt * (double)su;
        adv.Y[q] = y + adv.dt * (double)sv;
    } else if (adv.kind == ADV_PREDICT) {
        adv.Xs[q] = x + adv.dt * (double)su;
        adv.Ys[q] = y + adv.dt * (double)sv;
    } else if (adv.kind == ADV_HEUN) {
        adv.X[q] += 0.5 * adv.dt * ((double)((const T*)adv.u1)[q] + (double)su);
        adv.Y[q] += 0.5 * adv.dt * ((double)((const T*)adv.v1)[q] + (double)sv);
    }
}

// Scratch used by one regularization: owned by a plan, or carved from the
// static array of the allocation-free entry point.
struct BinWork {
    int* status;
    unsigned long long* oob;
    unsigned* tile_count;     // written by k_offsets
    double* gmax;             // [0]: largest |Gamma| (k_offsets); [1 + b]: that of locate block b
    int* tile_start;
    int* bin_off;             // a histogram row of ntiles a block
    int64_t off_cap;          // ints in bin_off
    void* pos;
    void* recs;
    int64_t rec_cap;          // record slots in recs
    void* zu = nullptr;       // optional E_v outputs (plan precision): zeroed for every vortex off the grid
    void* zv = nullptr;
};

inline Geo make_geo(int nx, int ny, double dx, double x0, double y0, int tile = BIN_TILE) {
    Geo g;
    g.x0 = x0; g.y0 = y0; g.dx = dx; g.nx = nx; g.ny = ny;
    g.inv_dx = 1.0 / dx;
    g.cx = -x0 / dx;
    g.cy = -y0 / dx;
    g.inv_dx2 = 1.0 / (dx * dx);
    g.recip = dx > 0x1p-500 && dx < 0x1p500;
    const double lx = (double)(nx - 2), ly = (double)(ny - 2);
    memcpy(&g.xlim, &lx, sizeof(double));
    memcpy(&g.ylim, &ly, sizeof(double));
    g.ntx = ceil_div(nx, tile);
    g.ntiles = g.ntx * ceil_div(ny, tile);
    return g;
}

// Bin nv vortices by tile (locate, offsets, scatter) into bw; `p` (may be
// null) only supplies the timing records and the error text.
// With dn (device count, see bin_count), nv is the capacity the launch is sized for.
template <typename T, int TILE, int NT>
pf_status bin_launch_nt(pf_plan p, const Geo& geo, const BinWork& bw, const double* X, const double* Y,
                        const double* G, int64_t nv, cudaStream_t s, int min_span, const int64_t* dn) {
    const int nb = bin_blocks(nv, min_span);
    const int64_t span = bin_span(nv, min_span);
    const int mb = bin_max_blocks(nv);
    if ((int64_t)nb * geo.ntiles > bw.off_cap) {
        if (p) snprintf(p->err, sizeof(p->err), "binning of %lld vortices: histograms reserved for fewer blocks", (long long)nv);
        return PF_ERR_INTERNAL;
    }
    const size_t sh_loc = (size_t)geo.ntiles * sizeof(unsigned);
    const size_t sh_sc = 2 * (size_t)geo.ntiles * sizeof(unsigned);
    if (set_smem(k_locate<T, TILE, NT>, sh_loc) != cudaSuccess || set_smem(k_scatter<T, TILE, NT>, sh_sc) != cudaSuccess)
        return PF_ERR_CUDA;
    Pos<T>* pos = (Pos<T>*)bw.pos;
    if (nb > 0) {
        PF_KERNEL(p, "bin_locate", PF_CUDA(p, pf_launch(k_locate<T, TILE, NT>, nb, NT, sh_loc, s, X, Y, G, nv,
                                                       span, dn, min_span, mb, geo, pos, bw.bin_off, bw.gmax + 1,
                                                       bw.status, bw.oob, (T*)bw.zu, (T*)bw.zv)));
    }
    PF_KERNEL(p, "bin_offsets", PF_CUDA(p, pf_launch(k_offsets, ceil_div(geo.ntiles, OFF_TILES), 1024, 0, s,
                                                     geo.ntiles, nb, bw.bin_off, bw.tile_count,
                                                     (const double*)(bw.gmax + 1), bw.gmax)));
    if (nb > 0) {
        PF_KERNEL(p, "bin_scatter", PF_CUDA(p, pf_launch(k_scatter<T, TILE, NT>, nb, NT, sh_sc, s, pos, nv,
                                                         span, dn, min_span, mb, geo, bw.bin_off, bw.tile_count,
                                                         bw.tile_start, (Rec<T>*)bw.recs, bw.rec_cap, bw.status)));
    } else if (cudaMemsetAsync(bw.tile_start, 0, (size_t)geo.ntiles * sizeof(int), s) != cudaSuccess) {
        return PF_ERR_CUDA;
    }
    return PF_OK;
}

template <typename T, int TILE = BIN_TILE>
pf_status bin_launch(pf_plan p, const Geo& geo, const BinWork& bw, const double* X, const double* Y,
                     const double* G, int64_t nv, cudaStream_t s, int min_span = BIN_MIN_SPAN,
                     const int64_t* dn = nullptr) {
    if (geo.ntiles > MAX_SCAN_TILES) return PF_ERR_ARG;
    if (bin_max_blocks(nv) == BIN_WIDE_BLOCKS)
        return bin_launch_nt<T, TILE, 1024>(p, geo, bw, X, Y, G, nv, s, min_span, dn);
    return bin_launch_nt<T, TILE, BIN_THREADS>(p, geo, bw, X, Y, G, nv, s, min_span, dn);
}

// Deposit the binned records of bw into w.
template <typename T, int TILE = BIN_TILE>
pf_status deposit_launch(pf_plan p, const Geo& geo, const Rec<T>* recs, const int* tile_start,
                         const unsigned* tile_count, const double* gmax, int64_t rec_cap, int* status, T* w,
                         cudaStream_t s, int threads = 256) {
    PF_KERNEL(p, "regularize", PF_CUDA(p, pf_launch(k_deposit<T, TILE, FlatBins>, geo.ntiles, threads, 0, s, recs,
                                                    FlatBins{tile_start, tile_count, gmax, rec_cap}, geo, w, status)));
    return PF_OK;
}

// The four regularization kernels.
template <typename T, int TILE = BIN_TILE>
pf_status regularize_launch(pf_plan p, const Geo& geo, const BinWork& bw, const double* X, const double* Y,
                            const double* G, int64_t nv, T* w, cudaStream_t s, int min_span = BIN_MIN_SPAN,
                            int threads = 256, const int64_t* dn = nullptr) {
    PF_TRY((bin_launch<T, TILE>(p, geo, bw, X, Y, G, nv, s, min_span, dn)));
    return deposit_launch<T, TILE>(p, geo, (const Rec<T>*)bw.recs, bw.tile_start, bw.tile_count,
                                   (const double*)bw.gmax, bw.rec_cap, bw.status, w, s, threads);
}

}  // namespace
