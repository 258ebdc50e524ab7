// The zero-padded convolution of fft.cu (same three passes, same half-spectrum
// layout) in block fixed point (fixpt.cuh): the passes of FP64 plans, and the
// FP64-class streamfunction that the sheet solves of mixed plans read.
//
// Every transform carries its own power-of-two exponent.  A row transform's
// is stored per row pair, a column's per column and component; the next pass
// aligns what it loads to the largest of them, so a value keeps at least the
// bits that matter against the largest one, as it does in a floating-point
// FFT, whose rounding noise is white and scaled by the largest values too.
// A NaN or an infinity in the input makes every output a NaN (as it spreads
// in floating point).
//
// Bound by the integer ALU (half its issue slots in the column pass) and the
// latencies between them at 24 warps an SM.  Measured against the same passes
// in FP64 (radix 16, FP64 pipe 90 % busy), 1024^2 nodes, velocity: rows 92 ->
// 28 us, columns 417 -> 134 us, inverse rows 157 -> 45 us; streamfunction of
// 512 x 384: 120 -> 44 us; and against double-float passes on the FP32 pipe
// (48 bits) for the surface right-hand side of 768 x 512: 102 -> 66 us.  The
// error is below that of the FP64 passes: against transforms in 80 bits, five grids of
// 128^2 to 1024^2 and three random fields each, psi 1.3e-16 to 4.3e-15 of its norm
// (FP64 passes 2.2e-16 to 6.9e-15, larger in each case), u and v 1.4 to 2.3e-16 (3.0 to 5.1e-16).
//
// A thread holds eight points (radix 8, T = N / 8 threads a transform), and
// every kernel has one copy of the transform's code, its passes and its
// directions (forward, and the inverse with real and imaginary parts
// exchanged) being loops: with sixteen points a thread and every pass inlined,
// a warp ran 11,000 instructions straight through and waited two thirds of its
// time for the instruction cache.
#include <algorithm>
#include <utility>

#include "fft_reg.cuh"

namespace {

__device__ __forceinline__ size_t spec_at(int j, int k, int nk) {
    return ((size_t)(j >> 2) * nk + k) * 4 + (j & 3);
}

// A transform's reductions over its threads (whole warps): slots in shared
// memory, each zero (FX_ZERO for exponents) before its one use.
__device__ __forceinline__ void group_or(unsigned* slot, unsigned v) {
    v = __reduce_or_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicOr(slot, v);
}
__device__ __forceinline__ void group_max(int* slot, int v) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(slot, v);
}

// one pad element per eight: the first pass's stores, eight elements apart,
// and all its other accesses are free of bank conflicts
__device__ __forceinline__ int pad8(int i) { return i + (i >> 3); }
template <int N> struct FxBuf { static constexpr int size = N + N / 8; };

// all of v brought below 2^FX_TOP for a mask gathered from it; e follows
template <int N>
__device__ __forceinline__ void rescale(fxc (&v)[N], unsigned mask, int& e) {
    const int sh = fx_shift_of(mask);
    e += sh;
    if (sh > 0) {                              // uniform over the transform's threads
        const long long h = (1ll << sh) >> 1;
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = fxc{fx_round(v[r].x, h, sh), fx_round(v[r].y, h, sh)};
    } else if (sh < 0) {
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = fxc{v[r].x << -sh, v[r].y << -sh};
    }
}

template <int N>
__device__ __forceinline__ unsigned mask_of(const fxc (&v)[N]) {
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < N; ++r) m |= fx_mask(v[r]);
    return m;
}

// Length-N transform (N = 8 8 8 R, or 8 8 4 for N = 256) by T = N / 8 threads,
// thread t holding x[t + T r] on input and output: inputs below 2^FX_TOP,
// outputs below 2^(FX_TOP + 3.5), v 2^e on both sides.  twN[m] = exp(-2 pi i
// m / N).  slot: three zeroed words.  Every thread of the block calls it.
template <int N>
__device__ __forceinline__ void fx_fft(fxc (&v)[8], fxc* buf, int t, const int4* __restrict__ twN, unsigned* slot,
                                       int& e) {
    constexpr int T = N / 8;
    constexpr int R = N == 256 ? 4 : N / 512;          // last pass; 1: none
    constexpr int NS_END = N / R;                       // the radix-8 passes cover Ns = 1, 8, .. < NS_END
#pragma unroll 1
    for (int Ns = 1; Ns < NS_END; Ns *= 8) {
        const int k = t & (Ns - 1);
        if (Ns > 1) {
            const int step = k * (T / Ns);              // r k N / (8 Ns)
#pragma unroll
            for (int r = 1; r < 8; ++r) v[r] = fx_cmul(v[r], __ldg(twN + r * step));
        }
        dft8<fxc, false>(v);
        if (R == 1 && Ns * 8 == N) return;              // outputs t + T r are in place
        group_or(slot, mask_of(v));
        __syncthreads();                                // buf is free, the mask complete after the next barrier
        const int d = (t - k) * 8 + k;
#pragma unroll
        for (int r = 0; r < 8; ++r) buf[pad8(d + r * Ns)] = v[r];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < 8; ++r) v[r] = buf[pad8(t + T * r)];
        rescale(v, *slot, e);
        ++slot;
    }
    if (R > 1) {
        constexpr int M = 8 / R;                        // butterflies j = t + m T, inputs j + r N / R
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const int j = t + m * T;
            fxc u[R];
#pragma unroll
            for (int r = 0; r < R; ++r) u[r] = v[m + r * M];
#pragma unroll
            for (int r = 1; r < R; ++r) u[r] = fx_cmul(u[r], __ldg(twN + r * j));
            dft_r<fxc, false, R>(u);
#pragma unroll
            for (int r = 0; r < R; ++r) v[m + r * M] = u[r];
        }
    }
}

// exponent field of a value (0 for zero and denormals; 2047: not finite)
__device__ __forceinline__ int exp_field(double d) { return (int)(((unsigned)__double2hiint(d) >> 20) & 0x7FF); }

// transforms a block of the row passes: 128 threads at least
template <int P> struct FxGroups { static constexpr int value = P >= 1024 ? 1 : 1024 / P; };

// Forward row pass: rows j, j + 1 as one complex transform, split into their
// half spectra.  The two rows' integers share the exponent rowE[j / 2].  The
// inputs' upper half (n >= P / 2 >= nx) is zero padding.
template <typename T, int P>
__global__ void __launch_bounds__(P / 8 * FxGroups<P>::value) k_fx_rows_fwd(const T* __restrict__ w, fxc* __restrict__ T1,
                                                                      int nx, int ny, const int4* __restrict__ twP,
                                                                      int* __restrict__ rowE, int* __restrict__ colmax) {
    constexpr int TP = P / 8, SB = FxBuf<P>::size, NK = P / 2 + 1, G = FxGroups<P>::value;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fxc* bufs = reinterpret_cast<fxc*>(smem_raw);
    __shared__ unsigned slots[G][4];
    const int g = threadIdx.x / TP, t = threadIdx.x % TP;
    fxc* buf = bufs + g * SB;
    const int r0 = 2 * G * blockIdx.x, j0 = r0 + 2 * g;
    const bool h0 = j0 < ny, h1 = j0 + 1 < ny;
    if (threadIdx.x < 4 * G) slots[threadIdx.x >> 2][threadIdx.x & 3] = 0u;
    pdl_wait();
    if (blockIdx.x == 0 && threadIdx.x == 0) *colmax = FX_ZERO;     // for the column pass
    double a[4], b[4];
    const int ja = h0 ? j0 : ny - 1, jb = h1 ? j0 + 1 : ny - 1;     // clamped: loads never branch
    int ef = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int n = t + TP * r, nc = n < nx ? n : nx - 1;
        const T x = w[(size_t)ja * nx + nc], y = w[(size_t)jb * nx + nc];
        a[r] = n < nx && h0 ? (double)x : 0.0;
        b[r] = n < nx && h1 ? (double)y : 0.0;
        // 0: zeros only; denormals count with the smallest normal exponent
        const int ea = exp_field(a[r]), eb = exp_field(b[r]);
        ef = max(ef, max(ea, eb));
        if (ef == 0 && ((__double_as_longlong(a[r]) | __double_as_longlong(b[r])) << 1) != 0) ef = 1;
    }
    __syncthreads();
    group_max((int*)&slots[g][3], ef);
    __syncthreads();
    const int emax = (int)slots[g][3], eu = max(emax, 1);
    fxc v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r)
        v[r] = r < 4 ? fxc{fx_from_double(a[r], eu), fx_from_double(b[r], eu)} : fxc{0, 0};
    int e = fx_exp(eu);
    fx_fft<P>(v, buf, t, twP, slots[g], e);
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 8; ++r) buf[pad8(t + TP * r)] = v[r];
    if (t == 0 && h0) rowE[j0 >> 1] = emax >= 2047 ? FX_NAN : emax == 0 ? FX_ZERO : e - 1;   // halves: below
    __syncthreads();
    fxc* dst = T1 + (size_t)(r0 >> 2) * NK * 4 + (r0 & 3);
    for (int i = threadIdx.x; i < NK * G; i += blockDim.x) {
        const int k = i / G, gg = i % G;
        const fxc* bz = bufs + gg * SB;
        const fxc z1 = bz[pad8(k)];
        fxc z2 = bz[pad8((P - k) & (P - 1))];
        z2.y = -z2.y;
        const fxc s = z1 + z2, d = z1 - z2;         // twice the half spectra: the exponent is one less
        const size_t at = ((size_t)((2 * gg) >> 2) * NK + k) * 4 + ((2 * gg) & 3);
        if (r0 + 2 * gg < ny) {
            dst[at] = s;
            dst[at + 1] = fxc{d.y, -d.x};
        }
    }
}

// leading bit position of a product with exponent eh, as the common scale needs it
__device__ __forceinline__ int lead_of(fxc p, int eh) { return 32 - __clz((int)fx_mask(p)) + eh; }

struct HVal {              // a spectrum value as a Q62 mantissa in [1/2, 1) and an exponent
    int bh, bl, e;
};
__device__ __forceinline__ HVal h_of(double h, bool neg) {
    const long long b = __double_as_longlong(h);
    const int ef = (int)((b >> 52) & 0x7FF);
    const long long m = ((b & 0xFFFFFFFFFFFFFll) | (1ll << 52)) << 9;
    HVal v;
    v.e = ef ? ef - 1022 : 0;
    const int hi = ef ? (int)(m >> 31) : 0, lo = ef ? (int)(m & 0x7FFFFFFF) : 0;
    const bool n = (b < 0) != neg;
    v.bh = n ? -hi : hi;
    v.bl = n ? -lo : lo;
    return v;
}

// Column pass: one column a block; forward transform, then per component the
// product with its spectrum and the inverse (real and imaginary parts
// exchanged on both sides of a forward transform).  768 threads an SM at 80
// registers: what the velocity's two shared buffers admit at Q = 2048.
template <int Q, bool UV>
__global__ void __launch_bounds__(Q / 8, 6144 / Q) k_fx_cols(const fxc* __restrict__ T1, fxc* __restrict__ T2a, fxc* __restrict__ T2b,
                                                   int ny, int nk, const double* __restrict__ Ha,
                                                   const double* __restrict__ Hb, int Hld, const int4* __restrict__ twQ,
                                                   const int* __restrict__ rowE, int* __restrict__ colEa,
                                                   int* __restrict__ colEb, int* __restrict__ colmax,
                                                   const int* __restrict__ rows) {
    constexpr int TQ = Q / 8, SB = FxBuf<Q>::size;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fxc* buf = reinterpret_cast<fxc*>(smem_raw);
    fxc* keep = buf + SB;
    __shared__ unsigned slots[12];
    __shared__ int tops[3];
    const int k = blockIdx.x, t = threadIdx.x;
    if (t < 12) slots[t] = 0u;
    if (t < 3) tops[t] = FX_ZERO;
    pdl_wait();
    // rows (nullable, psi): only output rows rows[0] .. rows[1] are needed, in whole pairs (k_fx_rows_inv)
    const int jlo = rows ? max(rows[0], 0) & ~1 : 0, jhi = rows ? min(rows[1] | 1, ny - 1) : ny - 1;
    fxc v[8];
    int d[4];
    int gE = FX_ZERO;
    for (int i = t; i < (ny + 1) / 2; i += TQ) gE = max(gE, rowE[i]);
#pragma unroll
    for (int r = 0; r < 8; ++r) {             // rows from Q / 2 on are padding
        v[r] = fxc{0, 0};
        if (r < 4) {
            const int l = t + TQ * r, lc = l < ny ? l : ny - 1;
            const fxc x = T1[spec_at(lc, k, nk)];
            d[r] = rowE[lc >> 1];
            if (l < ny) v[r] = x;
        }
    }
    __syncthreads();
    group_max(&tops[0], gE);
    __syncthreads();
    gE = tops[0];
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        v[r] = fx_align(v[r], min(gE - d[r], 63));
        m |= fx_mask(v[r]);
    }
    group_or(&slots[0], m);
    __syncthreads();
    int e = gE, ez = 0, etop = FX_ZERO;
    rescale(v, slots[0], e);
#pragma unroll 1
    for (int ph = 0; ph < (UV ? 3 : 2); ++ph) {
        if (ph > 0) {
            // i z h (velocity) or z h, parts exchanged; the products' common exponent from their largest
            const double* h = (ph == 1 ? Ha : Hb) + (size_t)k * Hld;
            const bool odd = UV && ph == 1;                       // u: odd in l; v, psi: even
            int eh[8], lead = FX_ZERO;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int l = t + TQ * r;
                const bool lo = l <= Q / 2;
                const HVal hv = h_of(__ldg(h + (lo ? l : Q - l)), odd && !lo);
                fxc z = v[r];
                if (UV) {
                    if (ph == 1) keep[pad8(l)] = z;                // read back by this thread
                    else z = keep[pad8(l)];
                    z = fxc{z.x, -z.y};
                } else {
                    z = fxc{z.y, z.x};
                }
                v[r] = fxc{fx_rmul(z.x, hv.bh, hv.bl), fx_rmul(z.y, hv.bh, hv.bl)};
                eh[r] = hv.e;
                if (v[r].x | v[r].y) lead = max(lead, lead_of(v[r], hv.e));
            }
            group_max(&tops[ph], lead);
            __syncthreads();
            const int top = tops[ph];
            e = top == FX_ZERO ? FX_ZERO : ez + top + 32 - FX_TOP;
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = fx_align(v[r], top + 32 - FX_TOP - eh[r]);
        }
        fx_fft<Q>(v, buf, t, twQ, slots + 1 + 3 * ph, e);
        if (ph == 0) {
            ez = e;
        } else {
            fxc* out = ph == 1 ? T2a : T2b;
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int l = t + TQ * r;
                if (l >= jlo && l <= jhi) out[spec_at(l, k, nk)] = fxc{v[r].y, v[r].x};
            }
            e = gE >= FX_NAN ? FX_NAN : max(e, FX_ZERO);
            etop = max(etop, e);
            if (t == 0) (ph == 1 ? colEa : colEb)[k] = e;
        }
    }
    if (t == 0) atomicMax(colmax, etop);
}

// Inverse row pass: u_j + i v_j (one row) or psi_j + i psi_{j+1} (two rows) a
// transform; out FP64.
// (Two rows a block at P = 2048, which read T2's sectors whole, measured 55 us
// against 45: the pass is bound by the integer pipe, not by those reads.)
template <int P, bool UV>
__global__ void __launch_bounds__(P / 8 * FxGroups<P>::value) k_fx_rows_inv(
    const fxc* __restrict__ T2a, const fxc* __restrict__ T2b, double* __restrict__ out, int nx, int ny, double Uinf,
    double Vinf, const int4* __restrict__ twP, const int* __restrict__ colEa, const int* __restrict__ colEb,
    const int* __restrict__ colmax, const int* __restrict__ rows) {
    constexpr int TP = P / 8, SB = FxBuf<P>::size, NK = P / 2 + 1, G = FxGroups<P>::value;
    constexpr int h = P / 2;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    fxc* bufs = reinterpret_cast<fxc*>(smem_raw);
    __shared__ unsigned slots[G][4];
    const int g = threadIdx.x / TP, t = threadIdx.x % TP;
    fxc* buf = bufs + g * SB;
    if (threadIdx.x < 4 * G) slots[threadIdx.x >> 2][threadIdx.x & 3] = 0u;
    const int j = (UV ? 1 : 2) * (G * blockIdx.x + g), jb = UV ? j : j + 1;
    const fxc* Sb = UV ? T2b : T2a;
    pdl_wait();
    // rows (nullable, psi): blocks whose rows are not read later do nothing
    if (rows) {
        const int lo = 2 * G * blockIdx.x;
        if (lo + 2 * G - 1 < rows[0] || lo > rows[1]) return;
    }
    const int E = *colmax;
    const bool ha = j < ny && (!rows || ((j | 1) >= rows[0] && (j & ~1) <= rows[1])), hb = jb < ny && ha;
    __syncthreads();
    unsigned m = 0;
    // k = t + TP i, i < 4, and the last one (k = P / 2) by thread 0; parts exchanged
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int k = i < 4 ? t + TP * i : h;
        if (i == 4 && t != 0) break;
        const int ea = colEa[k], eb = UV ? colEb[k] : ea;
        fxc a = fxc{0, 0}, b = fxc{0, 0};
        if (ha) a = T2a[spec_at(j, k, NK)];
        if (hb) b = Sb[spec_at(jb, k, NK)];
        a = fx_align(a, min(E - ea, 63));
        b = fx_align(b, min(E - eb, 63));
        if (k == 0 || k == h) { a.y = 0; b.y = 0; }
        const fxc z = fxc{a.y + b.x, a.x - b.y};                 // a + i b
        buf[pad8(k)] = z;
        m |= fx_mask(z);
        if (k > 0 && k < h) {
            const fxc c = fxc{b.x - a.y, a.x + b.y};             // conj(a) + i conj(b)
            buf[pad8(P - k)] = c;
            m |= fx_mask(c);
        }
    }
    __syncwarp();
    group_or(&slots[g][0], m);
    __syncthreads();
    fxc v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = buf[pad8(t + TP * r)];
    int e = E;
    rescale(v, slots[g][0], e);
    fx_fft<P>(v, buf, t, twP, &slots[g][1], e);
    const bool bad = E >= FX_NAN;
    const double nan = __longlong_as_double(0x7FF8000000000000ll);
    const bool add = UV && (Uinf != 0.0 || Vinf != 0.0);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int n = t + TP * r;
        const double x = bad ? nan : fx_to_double(v[r].y, e), y = bad ? nan : fx_to_double(v[r].x, e);
        if (n >= nx) continue;
        if (UV) {
            if (ha)
                reinterpret_cast<double2*>(out)[(size_t)j * nx + n] = add ? make_double2(x + Uinf, y + Vinf) : make_double2(x, y);
        } else {
            if (ha) out[(size_t)j * nx + n] = x;
            if (hb) out[(size_t)jb * nx + n] = y;
        }
    }
}

struct FxArgs {
    const void* w;
    double* out;
    double U, V;
    fxc *T1, *T2a, *T2b;
    const int* rows;
};

template <typename T, int P>
pf_status fx_rows_fwd(pf_plan p, const FxArgs& a) {
    constexpr int G = FxGroups<P>::value;
    const size_t sm = G * (size_t)FxBuf<P>::size * sizeof(fxc);
    PF_CUDA(p, set_smem(k_fx_rows_fwd<T, P>, sm));
    PF_KERNEL(p, "fft_rows_fwd", PF_CUDA(p, pf_launch(k_fx_rows_fwd<T, P>, ceil_div(p->ny, 2 * G), P / 8 * G, sm, p->stream,
                                                      (const T*)a.w, a.T1, p->nx, p->ny, p->twP_fx, p->fx_exp + FXE_ROW,
                                                      p->fx_exp)));
    return PF_OK;
}

template <int Q, bool UV>
pf_status fx_cols(pf_plan p, const FxArgs& a) {
    const size_t sm = (UV ? 2 : 1) * (size_t)FxBuf<Q>::size * sizeof(fxc);
    const int nk = p->P / 2 + 1;
    PF_CUDA(p, set_smem(k_fx_cols<Q, UV>, sm));
    PF_KERNEL(p, "fft_cols_conv", PF_CUDA(p, pf_launch(k_fx_cols<Q, UV>, nk, Q / 8, sm, p->stream, a.T1, a.T2a, a.T2b, p->ny, nk,
                                                       UV ? p->Hu64 : p->H64, p->Hv64, p->Hld, p->twQ_fx,
                                                       p->fx_exp + FXE_ROW, p->fx_exp + FXE_COLA, p->fx_exp + FXE_COLB,
                                                       p->fx_exp, a.rows)));
    return PF_OK;
}

template <int P, bool UV>
pf_status fx_rows_inv(pf_plan p, const FxArgs& a) {
    constexpr int G = FxGroups<P>::value;
    const size_t sm = G * (size_t)FxBuf<P>::size * sizeof(fxc);
    PF_CUDA(p, set_smem(k_fx_rows_inv<P, UV>, sm));
    PF_KERNEL(p, "fft_rows_inv", PF_CUDA(p, pf_launch(k_fx_rows_inv<P, UV>, ceil_div(p->ny, (UV ? 1 : 2) * G), P / 8 * G, sm,
                                                      p->stream, a.T2a, a.T2b, a.out, p->nx, p->ny, a.U, a.V, p->twP_fx,
                                                      p->fx_exp + FXE_COLA, p->fx_exp + FXE_COLB, p->fx_exp, a.rows)));
    return PF_OK;
}

#define FX_SIZE(n, ...)                                                   \
    switch (n) {                                                          \
        case 256: { constexpr int N = 256; PF_TRY((__VA_ARGS__)); break; }   \
        case 512: { constexpr int N = 512; PF_TRY((__VA_ARGS__)); break; }   \
        case 1024: { constexpr int N = 1024; PF_TRY((__VA_ARGS__)); break; } \
        case 2048: { constexpr int N = 2048; PF_TRY((__VA_ARGS__)); break; } \
        case 4096: { constexpr int N = 4096; PF_TRY((__VA_ARGS__)); break; } \
        default: return PF_ERR_ARG;                                       \
    }

template <typename T, bool UV>
pf_status fx_conv(pf_plan p, const FxArgs& a) {
    FX_SIZE(p->P, fx_rows_fwd<T, N>(p, a))
    FX_SIZE(p->Q, fx_cols<N, UV>(p, a))
    FX_SIZE(p->P, fx_rows_inv<N, UV>(p, a))
    return PF_OK;
}

// ---- twiddles in Q62, by Taylor series in 128-bit integers on the host
typedef __int128 i128;

// cos and sin of 2 pi m / N, 0 <= m <= N / 8 (below pi / 4), in Q62 to a few units
void octant(int m, int N, long long& c, long long& s) {
    const unsigned long long PI62 = 14488038916154245684ull;          // pi 2^62
    const i128 th = (i128)PI62 * (2 * (i128)m) / N;
    const i128 t2 = (th * th) >> 62;
    i128 ct = (i128)1 << 62, st = th, cs = ct, ss = st;
    for (int k = 1; k < 16; ++k) {
        ct = -((ct * t2) >> 62) / ((2 * k - 1) * (2 * k));
        st = -((st * t2) >> 62) / ((2 * k) * (2 * k + 1));
        cs += ct;
        ss += st;
    }
    c = (long long)cs;
    s = (long long)ss;
}

}  // namespace

// appends exp(-2 pi i m / N), m in [0, N), to v: centred halves (fx_high, fx_low) of the Q62 parts
void fx_twiddles(std::vector<int4>& v, int N) {
    const long long one = (1ll << 62) - 1;                                // so that the high half fits
    std::vector<long long> cs(N / 8 + 1), sn(N / 8 + 1);
    for (int m = 0; m <= N / 8; ++m) octant(m, N, cs[m], sn[m]);
    for (int m = 0; m < N; ++m) {
        const int q = m % (N / 4), in = q > N / 8 ? N / 4 - q : q;
        long long a = cs[in], b = sn[in], c, s;
        if (q > N / 8) std::swap(a, b);                                   // first quadrant: (a, b) = (cos, sin) of q
        switch (m / (N / 4)) {
            case 0: c = a; s = b; break;
            case 1: c = -b; s = a; break;
            case 2: c = -a; s = -b; break;
            default: c = b; s = -a; break;
        }
        c = std::min(std::max(c, -one), one);
        s = std::min(std::max(-s, -one), one);
        v.push_back(make_int4(fx_high(c), fx_low(c), fx_high(s), fx_low(s)));
    }
}

// node velocity (mode CONV_UV) or streamfunction of an FP64 plan's w; P, Q >= 256
pf_status conv_fx(pf_plan p, const double* w, double* out, int mode, double Uinf, double Vinf) {
    const FxArgs a{w, out, Uinf, Vinf, (fxc*)p->T1, (fxc*)p->T2a, (fxc*)p->T2b, nullptr};
    return mode == CONV_UV ? fx_conv<double, true>(p, a) : fx_conv<double, false>(p, a);
}

// psi = -L^-1 w as doubles for either precision of plan, of which only rows
// rows[0] .. rows[1] (device, within [0, ny)) are computed; T1, T2: ldT x ldK
// FP64-sized complex each
pf_status conv_psi_fx(pf_plan p, const void* w, double* psi, void* T1, void* T2, const int* rows) {
    if (p->P < 256 || p->Q < 256) return PF_ERR_ARG;
    const FxArgs a{w, psi, 0.0, 0.0, (fxc*)T1, (fxc*)T2, (fxc*)T2, rows};
    return p->prec == PF_FP64 ? fx_conv<double, false>(p, a) : fx_conv<float, false>(p, a);
}
