// The sheet solve of a body step on a small surface, in two launches:
//
//   k_vortex_rhs   E_s L^-1 R_v Gamma straight from the vortices (and E_s L^-1
//                  d_j of the vortices being released, at positions it works
//                  out itself, and the partial sums of Gamma);
//   k_sheet_small  right-hand side, S^-1 with one refinement, constraint rows,
//                  sheet, release, and R_s f node by node, in one cluster.
//
// The chain they replace was sixteen launches of 2 to 17 us, each too small to
// fill the GPU (128^2 nodes, 64 points, 256 vortices: 81 us of kernels a stage
// with the R_v they needed; these two 22 us).
#include <cooperative_groups.h>

#include "body.cuh"
#include "transfer.cuh"

namespace cg = cooperative_groups;

namespace {

// a weight |w| < 2 in Q61
__device__ __forceinline__ long long fx_q61(double w) {
    const long long b = __double_as_longlong(w);
    const int ef = (int)((b >> 52) & 0x7FF);
    if (ef == 0) return 0;
    const long long m = (b & 0xFFFFFFFFFFFFFll) | (1ll << 52);
    const long long v = fx_align1(m, 1014 - ef);                // m 2^(ef - 1075) 2^61
    return b < 0 ? -v : v;
}
// a table value in Q61 (0 at the origin, else 1/4 .. 1.53, at the corner of 2048 x 2048 nodes): its mantissa shifted
__device__ __forceinline__ long long fx_lgf(double g) {
    const long long b = __double_as_longlong(g);
    const int ef = (int)(b >> 52);
    return ef ? ((b & 0xFFFFFFFFFFFFFll) | (1ll << 52)) << (ef - 1014) : 0ll;
}

// Sum over a chunk of the vortices (blockIdx.y) of Gamma_q sum_{16 x 16 node
// pairs} d_p G M4'M4' for surface point p = blockIdx.x.  The pairs collapse to
// 7 x 7 node offsets with convolved weights (stencil_pair_lgf); a round of 64
// vortices has its weights formed by a thread per vortex and axis, then eight
// lanes a vortex take one column of the offsets each, so that a table row's
// seven values are one or two lines for the lanes together (a thread a vortex
// would touch 49).  Weights, table and products in Q61 on the integer pipe
// (FP64 has two multiply-adds a clock and SM), the sum over vortices in FP64
// in a fixed order.  p = 0 also sums the chunk's Gamma.  A last row of blocks
// forms, for each released vortex j, e_j[p] (position: given, or by the
// placement rule).
constexpr int VR_THREADS = 128, VR_ROUND = 64;

struct VortexRhs {
    const double *X, *Y, *G;
    int64_t nv;
    const int64_t* dn;
    int pairs;                 // 0: only the sums of Gamma and the released vortices
    const int *six, *siy;
    const double *swx, *swy, *table;
    int ns, ne, chunks, place; // place: released positions from e, written to newx, newy; else read there
    EdgeGeo e;
    double *newx, *newy;
    unsigned long long* oob;       // if not null: += the vortices off the grid
    double *part, *gpart, *unit;   // part[p * chunks + c], gpart[c], unit[j * ns + p]
};

struct VrShared {
    FxSplit c[VR_ROUND][2][8];
    int base[VR_ROUND][2];
    double g[VR_ROUND];
    FxSplit sw[2][4];
    double red[VR_THREADS / 32];
    double redg[VR_THREADS / 32];
};

// weights of one axis of a vortex against the surface point's: seven node offsets from base
__device__ __forceinline__ bool vr_weights(double z, const Geo& geo, int axis, int surf0, const FxSplit (&sw)[4], FxSplit* c,
                                           int& base) {
    int ci = 1;
    double f = 0.0;
    const bool ok = loc_split(z, geo, axis, ci, f);
    FxSplit wv[4];
    fx_m4p(ok ? f : 0.0, wv);
#pragma unroll
    for (int d = 0; d < 7; ++d) {
        long long h = 0, t = 1ll << 29;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int a2 = a + 3 - d;
            if (a2 < 0 || a2 > 3) continue;
            h += fx_mw(sw[a].h, wv[a2].h);
            t += fx_mw(sw[a].h, wv[a2].l) + fx_mw(sw[a].l, wv[a2].h);
        }
        c[d] = fx_split((h << 1) + (t >> 30));
    }
    c[7] = FxSplit{0, 0};
    base = surf0 - (ci - 1) - 3;
    return ok;
}

// This lane's column d of the pair sum, in Q61: cx[d] sum_e cy[e] G(base + (d, e)).
// The middle sum is taken in two parts, t0 over four entries and t1 over three:
// low halves are at most 2^30, the table's high halves 1.53 x 2^30 and the seven
// |cy| add up to at most 1.25, so t0 is at most (4 x 1.53 + 1.25) 2^60 = 7.4 x
// 2^60 < 2^63, where all seven together pass 2^63 from offsets of about 100 nodes on.
// (With the table in Q60 one sum holds them, and a bit is lost.)
__device__ __forceinline__ long long vr_column(const FxSplit (*c)[8], const int* base, int d, const double* __restrict__ G,
                                               int ld) {
    if (d == 7) return 0;
    int m = base[0] + d;
    m = m < 0 ? -m : m;
    long long h = 0, t0 = 1ll << 29, t1 = 0;
#pragma unroll
    for (int e = 0; e < 7; ++e) {
        int n = base[1] + e;
        n = n < 0 ? -n : n;
        const FxSplit g = fx_split(fx_lgf(__ldg(G + (size_t)n * ld + m))), w = c[1][e];
        h += fx_mw(g.h, w.h);
        (e < 4 ? t0 : t1) += fx_mw(g.h, w.l) + fx_mw(g.l, w.h);
    }
    const long long low = (1ll << 30) - 1, t = (t0 >> 30) + (t1 >> 30) + (((t0 & low) + (t1 & low)) >> 30);
    return fx_weigh(fx_split((h << 1) + t), c[0][d]);
}

// Q61 to double
__device__ __forceinline__ double fx_q61_double(long long v) { return fx_to_double(v, -61); }

// e_j[p] of the released vortices, eight lanes each
__device__ __forceinline__ void released(const VortexRhs& A, const Geo& geo, int p, const int (&surf)[2], VrShared& s,
                                         int* status) {
    const int tid = threadIdx.x, lane8 = tid & 7;
    if (tid < 2 * A.ne) {                       // a thread per released vortex and axis
        const int j = tid >> 1, axis = tid & 1;
        double z;
        if (A.place) {
            const int64_t last = A.dn ? A.dn[1 + j] : A.e.last[j];
            const double ez = axis ? A.e.ey[j] : A.e.ex[j];
            z = last < 0 ? ez + A.e.first_dist * (axis ? A.e.ny[j] : A.e.nx[j]) : ez + ((axis ? A.Y : A.X)[last] - ez) / 3.0;
            if (p == 0) (axis ? A.newy : A.newx)[j] = z;
        } else {
            z = (axis ? A.newy : A.newx)[j];
        }
        int base = 0;
        const bool ok = vr_weights(z, geo, axis, surf[axis], s.sw[axis], s.c[j][axis], base);
        s.base[j][axis] = ok ? base : 1 << 24;
    }
    __syncthreads();
    const int j = tid >> 3;                      // ne <= 2 PF_MAX_BODIES = 8 groups of eight lanes
    double u = 0.0;
    const bool ok = j < A.ne && s.base[j][0] < 1 << 20 && s.base[j][1] < 1 << 20;
    if (ok) u = fx_q61_double(vr_column(s.c[j], s.base[j], lane8, A.table, geo.nx + 1));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
    if (j < A.ne && lane8 == 0) {
        A.unit[(size_t)j * A.ns + p] = u;
        if (!ok && p == 0) atomicOr(status, ST_OUT_OF_DOMAIN);
    }
}

__global__ void __launch_bounds__(VR_THREADS) k_vortex_rhs(VortexRhs A, Geo geo, int* __restrict__ status) {
    __shared__ VrShared s;
    const int p = blockIdx.x, chunk = blockIdx.y, nchunk = A.chunks, tid = threadIdx.x, lane8 = tid & 7;
    pdl_wait();
    const int64_t n = A.dn ? *A.dn : A.nv;
    const int64_t per = (n + nchunk - 1) / nchunk, q0 = chunk * per, q1 = q0 + per < n ? q0 + per : n;
    if (tid < 8) s.sw[tid >> 2][tid & 3] = fx_split(fx_q61((tid < 4 ? A.swx : A.swy)[4 * p + (tid & 3)]));
    const int surf[2] = {A.six[4 * p], A.siy[4 * p]};
    __syncthreads();
    if (chunk == nchunk) {
        released(A, geo, p, surf, s, status);
        return;
    }
    double acc = 0.0;
    if (A.pairs) {
        for (int64_t r0 = q0; r0 < q1; r0 += VR_ROUND) {
            {
                const int v = tid & (VR_ROUND - 1), axis = tid / VR_ROUND;     // a thread per vortex and axis
                const int64_t q = r0 + v;
                int base = 0;
                bool ok = false;
                if (q < q1) ok = vr_weights(axis ? A.Y[q] : A.X[q], geo, axis, surf[axis], s.sw[axis], s.c[v][axis], base);
                s.base[v][axis] = ok ? base : 1 << 24;                        // marks a vortex that is left out
                if (axis == 0) s.g[v] = q < q1 ? A.G[q] : 0.0;
            }
            __syncthreads();
            if (p == 0 && A.oob && tid < VR_ROUND && r0 + tid < q1 &&
                (s.base[tid][0] >= 1 << 20 || s.base[tid][1] >= 1 << 20)) {
                atomicAdd(A.oob, 1ull);
                atomicOr(status, ST_OUT_OF_DOMAIN);
            }
#pragma unroll 1
            for (int v = tid >> 3; v < VR_ROUND; v += VR_THREADS / 8)
                if (s.base[v][0] < 1 << 20 && s.base[v][1] < 1 << 20)
                    acc += s.g[v] * fx_q61_double(vr_column(s.c[v], s.base[v], lane8, A.table, geo.nx + 1));
            __syncthreads();
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if ((tid & 31) == 0) s.red[tid >> 5] = acc;
        __syncthreads();
        if (tid == 0) A.part[(size_t)p * nchunk + chunk] = (s.red[0] + s.red[1]) + (s.red[2] + s.red[3]);
    }
    if (p == 0) {
        double g = 0.0;
        for (int64_t q = q0 + tid; q < q1; q += VR_THREADS) g += A.G[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
        if ((tid & 31) == 0) s.redg[tid >> 5] = g;
        __syncthreads();
        if (tid == 0) A.gpart[chunk] = (s.redg[0] + s.redg[1]) + (s.redg[2] + s.redg[3]);
    }
}
static_assert(2 * PF_MAX_BODIES * 8 <= VR_THREADS, "a group of lanes per released vortex");

// ---------------------------------------------------------------------------
// One cluster of eight blocks: block c takes rows c, c + 8, ... of the three
// products (S^-1 rhs, the residual against S, its correction), eight lanes a
// row and right-hand side, and every result goes to all blocks' shared memory
// over the cluster's network; block 0 then closes the constraint rows.  At two
// FP64 multiply-adds a clock and SM, 9 ns^2 of them take 0.4 us (ns 64) to 7 us
// (ns 256) on eight SMs; past SHEET_SMALL points one block per row fills more
// of the GPU (sheet_solve_device).
constexpr int SC_BLOCKS = 8, SC_THREADS = 256;
constexpr int SHEET_F0 = -1;         // mode: f0 of a new factor instead of a sheet

struct ScShared {
    double v[3][SHEET_SMALL], y[3][SHEET_SMALL], r[3][SHEET_SMALL], z[3][SHEET_SMALL];
    double ds[SHEET_SMALL], f0[SHEET_SMALL], f[SHEET_SMALL];
    double param, shift, sum[3];
};

__host__ __device__ constexpr int sc_rows(int ns) { return (ns + SC_BLOCKS - 1) / SC_BLOCKS; }
inline size_t sc_smem(int ns) {      // two blocks of rows, or the sheet's 16 ns terms and nodes
    return std::max(2 * (size_t)sc_rows(ns) * ns * sizeof(double), (size_t)16 * ns * (sizeof(double) + sizeof(int)));
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}

// A warp's FP64 instruction occupies its quarter of the SM for 64 clocks
// whether one lane or all are active, so sums are left to one warp each, and
// scalars are worked out by as many lanes as there are of them.
__device__ __forceinline__ double warp_sum(double a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}
__device__ __forceinline__ double lane_val(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }

// s0, Gamma1, Gamma2 of the constraint rows (k_constraints, body.cu), by one
// warp; h: f0hat^T ft*, ft_1, ft_2
__device__ __forceinline__ void constraint_rows(const SheetSmall& A, const ScShared& s, double param, double Gamma0, double& s0,
                                                double& G1, double& G2) {
    const int lane = threadIdx.x & 31;
    G1 = G2 = 0.0;
    if (A.mode == PF_SHEET_GIVEN_S0) {
        s0 = param;
        return;
    }
    if (A.mode == PF_SHEET_CIRCULATION) {
        s0 = (s.sum[0] - param) / Gamma0;
        return;
    }
    // lane 3 e + c: y_c / f0 at edge e
    const int e = lane < 3 ? 0 : 1, c = lane < 3 ? lane : lane < 6 ? lane - 3 : 0, k = e ? A.k2 : A.k1;
    const double at = c < A.nc ? s.z[c][k] / s.f0[k] : 0.0;
    if (A.mode == PF_SHEET_KUTTA_STEADY) {
        s0 = lane_val(at, 0);
        return;
    }
    const EdgeBounds& eb = A.eb;
    // lane 3 e + c, c > 0: A_ec = 1 + h_c - Gamma0 t_ec; c = 0: b_e = -(param + h_0 - Gamma0 fs_e + Gamma0 target_e)
    const double lo = e ? eb.lo[1] : eb.lo[0], hi = e ? eb.hi[1] : eb.hi[0];
    const double fs = __shfl_sync(0xffffffffu, at, 3 * e);
    const double tg = eb.on ? (fs < lo ? lo : hi) : 0.0;
    const bool act = !eb.on || !(lo <= fs && fs <= hi);
    double x = (c ? 1.0 : param) + s.sum[c] - Gamma0 * at;
    if (c == 0) x = -(x + Gamma0 * tg);
    const double b1 = lane_val(x, 0), A11 = lane_val(x, 1), A12 = lane_val(x, 2);
    const double b2 = lane_val(x, 3), A21 = lane_val(x, 4), A22 = lane_val(x, 5);
    const double t1 = lane_val(tg, 0), t2 = lane_val(tg, 3);
    const bool on1 = __shfl_sync(0xffffffffu, act, 0), on2 = A.nedge == 2 && __shfl_sync(0xffffffffu, act, 3);
    // lane 0: Gamma1, lane 1: Gamma2
    double num, den;
    if (on1 && on2) {
        num = lane ? A11 * b2 - A21 * b1 : b1 * A22 - A12 * b2;
        den = A11 * A22 - A12 * A21;
    } else if (on1) {
        num = lane ? 0.0 : b1;
        den = A11;
    } else if (on2) {
        num = lane ? b2 : 0.0;
        den = A22;
    } else {
        num = s.sum[0] + param;
        den = Gamma0;
    }
    const double q = num / den;
    if (!on1 && !on2) {
        s0 = q;
        return;
    }
    G1 = lane_val(q, 0);
    G2 = lane_val(q, 1);
    // s0: the active edges' g_k - target, averaged; lanes 0 and 3 hold the edges
    double g = __shfl_sync(0xffffffffu, at, 3 * e) + G1 * __shfl_sync(0xffffffffu, at, 3 * e + 1) +
               G2 * __shfl_sync(0xffffffffu, at, 3 * e + 2) - (e ? t2 : t1);
    const double g1 = lane_val(g, 0), g2 = lane_val(g, 3);
    s0 = on1 && on2 ? 0.5 * (g1 + g2) : on1 ? g1 : g2;
}

__global__ void __launch_bounds__(SC_THREADS) __cluster_dims__(SC_BLOCKS, 1, 1) k_sheet_small(SheetSmall A) {
    __shared__ ScShared s;
    extern __shared__ __align__(16) double sc_dyn[];
    cg::cluster_group cl = cg::this_cluster();
    const int me = (int)cl.block_rank(), tid = threadIdx.x, ns = A.ns, nc = A.nc;
    const int rows = (ns - me + SC_BLOCKS - 1) / SC_BLOCKS;   // rows me, me + 8, ...
    double* minv = sc_dyn;                                // this block's rows of S^-1 and S
    double* mat = minv + sc_rows(ns) * ns;
    pdl_wait();
    for (int i = tid; i < rows * ns; i += SC_THREADS) {   // in flight while the right-hand side is formed
        const size_t at = (size_t)(me + SC_BLOCKS * (i / ns)) * ns + i % ns;
        cp_async8(minv + i, A.Sinv + at);
        cp_async8(mat + i, A.S + at);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const double Gamma0 = A.mode == SHEET_F0 ? 1.0 : *A.gamma0;
    const int p = tid, lane = tid & 31, wid = tid >> 5;   // ns <= SC_THREADS
    if (wid == SC_THREADS / 32 - 1) {                     // the last warp: param, +- the sum of Gamma
        double g = A.param_d ? *A.param_d : A.param_h;
        if (A.gpart) g = A.gsign * warp_sum(lane < A.ngpart ? A.gpart[lane] : 0.0);
        if (lane == 0) s.param = g;
    }
    // right-hand side 0 (every block its own copy): s'_b - shift + E L^-1 w
    double sb = 0.0, ew = 0.0;
    if (A.mode == SHEET_F0) {
        if (p < ns) {
            sb = 1.0;
            s.ds[p] = A.ds[p];
        }
    } else if (p < ns) {
        const double x = A.x[p], y = A.y[p], fh = A.f0hat[p];
        s.ds[p] = A.ds[p];
        s.f0[p] = A.f0[p];
        double part[EW_SPLIT_MAX];
#pragma unroll
        for (int c = 0; c < EW_SPLIT_MAX; ++c) part[c] = c < A.chunks ? A.part[(size_t)p * A.chunks + c] : 0.0;
        for (int c = 1; c < nc; ++c) s.v[c][p] = A.unit[(size_t)(c - 1) * ns + p];
        sb = (A.m.U - A.m.Uinf) * y - (A.m.V - A.m.Vinf) * x;
        if (A.m.Omega != 0.0) sb -= 0.5 * A.m.Omega * (x * x + y * y);
#pragma unroll
        for (int c = 0; c < EW_SPLIT_MAX; ++c)
            if (c < A.chunks) ew += part[c];
        s.f[p] = fh * sb;                                 // terms of f0hat^T s'_b
    }
    __syncthreads();
    if (wid == 0) {
        double sh = 0.0;
        if (A.mode == PF_SHEET_GIVEN_S0) {
            sh = s.param;
        } else if (A.mode != PF_SHEET_CIRCULATION && A.mode != SHEET_F0) {
            for (int q = lane; q < ns; q += 32) sh += s.f[q];
            sh = warp_sum(sh) / Gamma0;
        }
        if (lane == 0) s.shift = sh;
    }
    __syncthreads();
    const double param = s.param;
    if (p < ns) s.v[0][p] = sb - s.shift + ew;
    asm volatile("cp.async.wait_all;" ::: "memory");
    cl.sync();                                            // every block has started: its shared memory can be written
    // out_c = (MODE 1: in2_c -) A in_c (MODE 2: + in2_c) for this block's rows, to every block
    const int lane8 = tid & 7, grp = tid >> 3;
    auto product = [&](int mode, const double* M, double (*in)[SHEET_SMALL], double (*in2)[SHEET_SMALL],
                       double (*out)[SHEET_SMALL]) {
        for (int i0 = 0; i0 < rows * nc; i0 += SC_THREADS / 8) {
            const int i = i0 + grp, c = i % nc, row = me + SC_BLOCKS * (i / nc);
            const bool on = i < rows * nc;
            double a0 = 0.0, a1 = 0.0;
            if (on) {
                const double* mr = M + (i / nc) * ns;
                int q = lane8;
                for (; q + 8 < ns; q += 16) {
                    a0 += mr[q] * in[c][q];
                    a1 += mr[q + 8] * in[c][q + 8];
                }
                if (q < ns) a0 += mr[q] * in[c][q];
            }
            double a = a0 + a1;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (on) {
                if (mode == 1) a = in2[c][row] - a;
                else if (mode == 2) a += in2[c][row];
                cl.map_shared_rank(&out[c][row], lane8)[0] = a;     // lane l writes to block l
            }
        }
        cl.sync();
    };
    product(0, minv, s.v, s.v, s.y);
    product(1, mat, s.y, s.v, s.r);
    product(2, minv, s.r, s.y, s.z);
    if (A.mode == SHEET_F0) {                             // f0, f0hat = dS f0, Gamma0 = <1, f0>
        if (me != 0) return;
        if (p < ns) {
            const double f0 = s.z[0][p], h = s.ds[p] * f0;
            A.f[p] = f0;
            A.f0hat_out[p] = h;
            s.f[p] = h;
        }
        __syncthreads();
        if (wid == 0) {
            double g = 0.0;
            for (int q = lane; q < ns; q += 32) g += s.f[q];
            g = warp_sum(g);
            if (lane == 0) A.scal[0] = g;
        }
        return;
    }
    // (no remote access after the last barrier.)  Every block closes the
    // constraint rows for itself and adds its share of R_s f's nodes.
    if (wid < 3 && A.mode != PF_SHEET_GIVEN_S0) {
        double h = 0.0;
        if (wid < nc)
            for (int q = lane; q < ns; q += 32) h += s.ds[q] * s.z[wid][q];
        h = warp_sum(h);
        if (lane == 0) s.sum[wid] = h;
    }
    __syncthreads();
    double s0, G1, G2;
    if (wid == 0) {
        constraint_rows(A, s, param, Gamma0, s0, G1, G2);
        if (lane == 0) {
            s.sum[0] = s0;
            s.sum[1] = G1;
            s.sum[2] = G2;
        }
    }
    __syncthreads();
    s0 = s.sum[0];
    G1 = s.sum[1];
    G2 = s.sum[2];
    if (p < ns) {
        double f = s.z[0][p];
        if (A.mode != PF_SHEET_GIVEN_S0) {                 // f0 o (ftilde* + sum G ft - s0)
            if (nc > 1) f += G1 * s.z[1][p];
            if (nc > 2) f += G2 * s.z[2][p];
            f -= s0 * s.f0[p];
        }
        if (me == 0) A.f[p] = f;
        s.f[p] = f;
    }
    if (me == 0 && tid == 0) {
        A.scal[0] = s0;
        A.scal[1] = G1;
        A.scal[2] = G2;
    }
    if (me == 0 && A.rel.n > 0 && tid < 32) {                          // the released vortices join the set (as k_append)
        int64_t nv = A.rel.nv;
        if (A.rel.use_dn) nv = A.rel.dn[0];
        const bool fits = nv >= 0 && nv + A.rel.n <= A.rel.cap;
        if (tid < A.rel.n && fits) {
            A.rel.X[nv + tid] = A.rel.newx[tid];
            A.rel.Y[nv + tid] = A.rel.newy[tid];
            A.rel.G[nv + tid] = tid ? G2 : G1;
            A.rel.dn[1 + tid] = nv + tid;
        }
        __syncwarp();
        if (tid == 0) {
            if (fits) A.rel.dn[0] = nv + A.rel.n;
            else atomicOr(A.rel.status, ST_CAPACITY);
        }
    }
    if (!A.sval) return;
    __syncthreads();                                       // f is complete; the matrices are done with
    // R_s f dx^2, one value per node's first sorted entry: this block's eighth of
    // the entries and the runs that leave it (a node has at most 16 ns of them)
    const int per = 2 * ns, i0 = me * per, i1 = min(i0 + per, 16 * ns);
    double* term = sc_dyn;
    int* node = reinterpret_cast<int*>(term + 16 * ns);
    int end = i1;
    if (i1 < 16 * ns) {                                    // the run that i1 - 1 belongs to
        const int last = A.snode[i1 - 1];
        while (end < 16 * ns && A.snode[end] == last) ++end;
    }
    for (int i = i0 + tid; i < end; i += SC_THREADS) {
        const int e = A.sorder[i], q = e >> 4;
        node[i] = A.snode[i];
        term[i] = s.ds[q] * s.f[q] * A.swx[4 * q + (e & 3)] * A.swy[4 * q + ((e >> 2) & 3)];
    }
    const int before = i0 > 0 ? A.snode[i0 - 1] : -1;
    __syncthreads();
    for (int i = i0 + tid; i < i1; i += SC_THREADS) {
        double acc = 0.0;
        if ((i == i0 ? before : node[i - 1]) != node[i])
            for (int k = i; k < end && node[k] == node[i]; ++k) acc += term[k];
        A.sval[i] = acc;
    }
}

}  // namespace

// partial sums a surface point: about seven blocks an SM, whose table reads
// hide one another's latency, and a round of vortices each (a function of ns
// and the capacity, so that a captured step and pf_step add in the same order)
int vortex_rhs_chunks(int ns, int64_t cap) {
    const int64_t rounds = (cap + VR_ROUND - 1) / VR_ROUND;
    return (int)std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>(EW_SPLIT_MAX, ceil_div(7 * 152, ns)), rounds));
}

pf_status vortex_rhs(pf_plan p, pf_schur s, const VortexSource& vs, int ne, const EdgeGeo* place, double* newx, double* newy,
                     double* unit) {
    VortexRhs A{};
    A.X = vs.X;
    A.Y = vs.Y;
    A.G = vs.G;
    A.nv = vs.n;
    A.dn = vs.dn;
    A.pairs = vs.pairs;
    A.oob = vs.oob;
    A.six = s->six;
    A.siy = s->siy;
    A.swx = s->swx;
    A.swy = s->swy;
    A.table = p->G;
    A.ns = s->ns;
    A.ne = ne;
    A.chunks = vortex_rhs_chunks(s->ns, vs.cap);
    A.place = place != nullptr;
    if (place) A.e = *place;
    A.newx = newx;
    A.newy = newy;
    A.part = s->ewpart;
    A.gpart = s->gpart;
    A.unit = unit;
    const Geo geo = make_geo(p->nx, p->ny, p->dx, p->x0, p->y0);
    PF_KERNEL(p, "vortex_rhs", PF_CUDA(p, pf_launch(k_vortex_rhs, dim3(s->ns, A.chunks + (ne > 0)), VR_THREADS, 0, p->stream,
                                                    A, geo, p->d_status)));
    return PF_OK;
}

// f0 = S^-1 1 refined, f0hat and Gamma0 of a new factor
pf_status sheet_f0_small(pf_plan p, pf_schur s) {
    SheetSmall a{};
    a.mode = SHEET_F0;
    a.ns = s->ns;
    a.nc = 1;
    a.ds = s->ds;
    a.S = s->S;
    a.Sinv = s->Sinv;
    a.f = s->f0;
    a.f0hat_out = s->f0hat;
    a.scal = s->dgamma0;
    return sheet_small(p, a);
}

pf_status sheet_small(pf_plan p, const SheetSmall& a) {
    PF_CUDA(p, set_smem(k_sheet_small, sc_smem(SHEET_SMALL)));
    PF_KERNEL(p, "sheet_small", PF_CUDA(p, pf_launch(k_sheet_small, SC_BLOCKS, SC_THREADS, sc_smem(a.ns), p->stream, a)));
    return PF_OK;
}
