// Unbounded Poisson solve psi = -L^{-1} w by zero-padded FFT convolution with
// the real, even LGF spectrum (Sec. 2.1), and the spectral node velocity.
//
// Layout of the three passes (w real, ny rows of nx nodes; torus P x Q):
//   1. rows:    two real rows j, j+1 packed as one complex row, length-P FFT,
//               split into the two half spectra A_j(k), k in [0, P/2]; the
//               generic kernels store them column-major T1[k*ny + j], the
//               register-resident ones in groups of four rows (see below).
//   2. columns: for each k, length-Q FFT of T1[k, 0..ny) (zero padded),
//               multiply by the kernel spectrum (psi: -dx^2 Ghat/(PQ); for the
//               node velocity the spectra of the centred-differenced LGF,
//               u: -dx/2 D_y G, v: +dx/2 D_x G, which is exactly the central
//               difference of psi), inverse FFT, keep rows [0, ny).
//   3. rows:    rebuild full Hermitian rows from the half spectra of two real
//               outputs (psi_j + i psi_{j+1}, or u_j + i v_j), inverse FFT,
//               keep nodes [0, nx).
#include <type_traits>

#include "fft.cuh"
#include "fft_reg.cuh"

template <typename T>
__global__ void __launch_bounds__(256) k_rows_fwd(const T* __restrict__ w, C_t<T>* __restrict__ T1, int nx, int ny,
                                                  int P, const C_t<T>* __restrict__ tw) {
    using C = C_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    C* B = A + P;
    const int j0 = 2 * blockIdx.x;
    const bool has2 = (j0 + 1) < ny;
    for (int n = threadIdx.x; n < P; n += blockDim.x) {
        T a = 0, b = 0;
        if (n < nx) {
            a = w[(size_t)j0 * nx + n];
            if (has2) b = w[(size_t)(j0 + 1) * nx + n];
        }
        A[n] = cmake<C>(a, b);
    }
    __syncthreads();
    C* Z = block_fft<C, false>(A, B, P, tw);
    for (int k = threadIdx.x; k <= P / 2; k += blockDim.x) {
        const C z1 = Z[k], z2 = conjc(Z[(P - k) & (P - 1)]);
        T1[(size_t)k * ny + j0] = (z1 + z2) * T(0.5);
        if (has2) T1[(size_t)k * ny + j0 + 1] = mul_mi(z1 - z2) * T(0.5);
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_cols(const C_t<T>* __restrict__ T1, C_t<T>* __restrict__ T2a,
                                              C_t<T>* __restrict__ T2b, int ny, int Q, int mode,
                                              const T* __restrict__ H, const T* __restrict__ Hu,
                                              const T* __restrict__ Hv, int Hld, const C_t<T>* __restrict__ tw) {
    using C = C_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    C* B = A + Q;
    C* D = B + Q;
    const int k = blockIdx.x;
    for (int l = threadIdx.x; l < Q; l += blockDim.x)
        A[l] = l < ny ? T1[(size_t)k * ny + l] : cmake<C>(T(0), T(0));
    __syncthreads();
    C* Z = block_fft<C, false>(A, B, Q, tw);
    C* other = (Z == A) ? B : A;
    const size_t row = (size_t)k * Hld;
    if (mode == CONV_UV) {
        for (int l = threadIdx.x; l < Q; l += blockDim.x) {
            const bool lo = l <= Q / 2;
            const int lq = lo ? l : Q - l;
            const C iw = mul_i(Z[l]);
            const T hu = Hu[row + lq];
            D[l] = iw * (lo ? hu : -hu);      // odd in l
            Z[l] = iw * Hv[row + lq];         // even in l
        }
        __syncthreads();
        C* U = block_fft<C, true>(D, other, Q, tw);
        for (int j = threadIdx.x; j < ny; j += blockDim.x) T2a[(size_t)k * ny + j] = U[j];
        __syncthreads();
        C* scratch = (U == D) ? other : D;
        C* V = block_fft<C, true>(Z, scratch, Q, tw);
        for (int j = threadIdx.x; j < ny; j += blockDim.x) T2b[(size_t)k * ny + j] = V[j];
    } else {
        for (int l = threadIdx.x; l < Q; l += blockDim.x) Z[l] = Z[l] * H[row + (l <= Q / 2 ? l : Q - l)];
        __syncthreads();
        C* R = block_fft<C, true>(Z, other, Q, tw);
        for (int j = threadIdx.x; j < ny; j += blockDim.x) T2a[(size_t)k * ny + j] = R[j];
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_rows_inv(const C_t<T>* __restrict__ T2a, const C_t<T>* __restrict__ T2b,
                                                  T* __restrict__ out, int nx, int ny, int P, int mode, T Uinf,
                                                  T Vinf, const C_t<T>* __restrict__ tw) {
    using C = C_t<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    C* B = A + P;
    int ja, jb;
    const C_t<T>* Sb;
    bool has_b = true;
    if (mode == CONV_UV) {
        ja = jb = blockIdx.x;
        Sb = T2b;
    } else {
        ja = 2 * blockIdx.x;
        jb = ja + 1;
        has_b = jb < ny;
        Sb = T2a;
    }
    const int h = P / 2;
    for (int k = threadIdx.x; k <= h; k += blockDim.x) {
        C a = T2a[(size_t)k * ny + ja];
        C b = has_b ? Sb[(size_t)k * ny + jb] : cmake<C>(T(0), T(0));
        if (k == 0 || k == h) { a.y = 0; b.y = 0; }
        A[k] = a + mul_i(b);
        if (k > 0 && k < h) A[P - k] = conjc(a) + mul_i(conjc(b));
    }
    __syncthreads();
    C* Z = block_fft<C, true>(A, B, P, tw);
    if (mode == CONV_UV) {
        T* o = out + (size_t)2 * ja * nx;
        for (int n = threadIdx.x; n < nx; n += blockDim.x) {
            o[2 * n] = Z[n].x + Uinf;
            o[2 * n + 1] = Z[n].y + Vinf;
        }
    } else {
        for (int n = threadIdx.x; n < nx; n += blockDim.x) {
            out[(size_t)ja * nx + n] = Z[n].x;
            if (has_b) out[(size_t)jb * nx + n] = Z[n].y;
        }
    }
}

// generic in-place complex FFTs of a row-major (rows x len) array, used once per
// plan to transform the LGF torus
template <typename C>
__global__ void __launch_bounds__(256) k_fft_rows_inplace(C* data, int len, const C* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    C* B = A + len;
    C* row = data + (size_t)blockIdx.x * len;
    for (int n = threadIdx.x; n < len; n += blockDim.x) A[n] = row[n];
    __syncthreads();
    C* Z = block_fft<C, false>(A, B, len, tw);
    for (int n = threadIdx.x; n < len; n += blockDim.x) row[n] = Z[n];
}

template <typename C>
__global__ void __launch_bounds__(256) k_fft_cols_inplace(C* data, int width, int len, const C* __restrict__ tw) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* A = reinterpret_cast<C*>(smem_raw);
    C* B = A + len;
    const int c = blockIdx.x;
    for (int n = threadIdx.x; n < len; n += blockDim.x) A[n] = data[(size_t)n * width + c];
    __syncthreads();
    C* Z = block_fft<C, false>(A, B, len, tw);
    for (int n = threadIdx.x; n < len; n += blockDim.x) data[(size_t)n * width + c] = Z[n];
}

pf_status fft2d_inplace_f64(pf_plan p, double2* data) {
    const size_t sr = 2 * (size_t)p->P * sizeof(double2), sc = 2 * (size_t)p->Q * sizeof(double2);
    PF_CUDA(p, set_smem(k_fft_rows_inplace<double2>, sr));
    PF_CUDA(p, set_smem(k_fft_cols_inplace<double2>, sc));
    k_fft_rows_inplace<double2><<<p->Q, 256, sr, p->stream>>>(data, p->P, p->twP64);
    PF_LAUNCH_CHECK(p);
    k_fft_cols_inplace<double2><<<p->P, 256, sc, p->stream>>>(data, p->P, p->Q, p->twQ64);
    PF_LAUNCH_CHECK(p);
    return PF_OK;
}


// ---------------------------------------------------------------------------
// Register-resident variants for P, Q = 256 * R3 (256 <= P, Q <= 4096).
//
// Half-spectrum layout shared by T1, T2a, T2b: rows in groups of four,
// element (j, k) at ((j / 4) * nk + k) * 4 + j % 4 with nk = P/2 + 1.  The
// forward row pass (four rows per block) then writes one contiguous run, and
// a column k is read and written as full 32-byte sectors of four rows.
__device__ __forceinline__ size_t spec_at(int j, int k, int nk) {
    return ((size_t)(j >> 2) * nk + k) * 4 + (j & 3);
}

// Two consecutive rows j, j + 1 (j even) of a half spectrum are adjacent in
// this layout: one 16-byte access.
__device__ __forceinline__ void ld_pair(const float2* p, float2& a, float2& b) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void st_pair(float2* p, float2 a, float2 b) {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
}

// Rows a block of the forward pass: two transforms of two rows each, so that
// its 32-byte sectors of T1 are written whole by one block (measured faster
// than twice the blocks writing halves).
constexpr int FWD_GROUPS = 2;

// Transforms a block of the inverse row pass.  A 32-byte sector of T2 holds
// four rows' values of one k; a block that reads it for one row makes the pass
// wait on L2 (2048 x 1800 nodes, velocity: 84 us with one row a block, 28 with
// two, a tenth more with four; at 1024^2 all three the same, 9.2).
constexpr int INV_GROUPS = 2;

template <int R3>
__global__ void __launch_bounds__(16 * R3 * FWD_GROUPS) k_rows_fwd_r(const float* __restrict__ w,
                                                                                float2* __restrict__ T1, int nx,
                                                                                int ny, const float2* __restrict__ tw) {
    constexpr int P = 256 * R3, TP = P / 16, SB = SBuf<P>::size, NK = P / 2 + 1, G = FWD_GROUPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* bufs = reinterpret_cast<float2*>(smem_raw);
    const int g = threadIdx.x / TP, t = threadIdx.x % TP;
    float2* buf = bufs + g * SB;
    const int r0 = 2 * G * blockIdx.x;          // the block's first row (even)
    const int j0 = r0 + 2 * g;
    const bool h0 = j0 < ny, h1 = j0 + 1 < ny;
    pdl_wait();
    float2 v[16];
    const int ja = h0 ? j0 : ny - 1, jb = h1 ? j0 + 1 : ny - 1;     // clamped rows: loads never branch
#pragma unroll
    for (int r = 0; r < 16; ++r) {                   // n >= P / 2 >= nx: padding
        v[r] = make_float2(0.f, 0.f);
        if (r >= 8) continue;
        const int n = t + TP * r;
        const int nc = n < nx ? n : nx - 1;
        const float a = w[(size_t)ja * nx + nc], b = w[(size_t)jb * nx + nc];
        v[r] = make_float2(n < nx && h0 ? a : 0.f, n < nx && h1 ? b : 0.f);
    }
    fft_strided<float2, false, R3>(v, buf, t, tw);
#pragma unroll
    for (int r = 0; r < 16; ++r) buf[spad(t + TP * r)] = v[r];
    __syncthreads();
    // per k, the half spectra of the rows j0, j0 + 1 of each group are adjacent
    // (rows past ny get the zero spectrum of their zero input)
    float2* dst = T1 + (size_t)(r0 >> 2) * NK * 4 + (r0 & 3);
    for (int e = threadIdx.x; e < NK * G; e += blockDim.x) {
        const int k = e / G, gg = e % G;
        const float2* bz = bufs + gg * SB;
        const float2 z1 = bz[spad(k)], z2 = conjc(bz[spad((P - k) & (P - 1))]);
        st_pair(dst + 4 * k + 2 * gg, (z1 + z2) * 0.5f, mul_mi(z1 - z2) * 0.5f);
    }
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sa), "l"(gmem) : "memory");
}

// Column pass.  The block's rows of the kernel spectra (Hu and Hv, or H) are
// copied into shared memory by cp.async as the block starts, so their loads
// overlap the column load and the forward transform.  128 registers a thread
// hold the twiddles of all three transforms; loading them again in each (96
// registers, five blocks an SM instead of four) measured 18.3 us against 16.0 at
// 1024^2, 80 registers and six blocks 21.7, 168 and three 18.6.
template <int R3>
__global__ void __launch_bounds__(16 * R3, R3 > 1 ? 32 / R3 : 1) k_cols_r(
    const float2* __restrict__ T1, float2* __restrict__ T2a, float2* __restrict__ T2b, int ny, int nk, int mode,
    const float* __restrict__ H, const float* __restrict__ Hu, const float* __restrict__ Hv, int Hld,
    const float2* __restrict__ tw) {
    constexpr int Q = 256 * R3, TQ = Q / 16, SB = SBuf<Q>::size;
    constexpr int NH = (Q / 2 + 1 + 3) / 4 * 4, PER = 16 / sizeof(float);   // spectrum row length, elements per copy
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* buf = reinterpret_cast<float2*>(smem_raw);
    float2* keep = buf + SB;
    float* hs0 = reinterpret_cast<float*>(keep + SB);
    float* hs1 = hs0 + NH;
    const int k = blockIdx.x, t = threadIdx.x;
    const size_t row = (size_t)k * Hld;
    pdl_wait();
    {
        const float* s0 = mode == CONV_UV ? Hu : H;
        for (int i = PER * t; i < NH; i += PER * TQ) {
            cp_async16(hs0 + i, s0 + row + i);
            if (mode == CONV_UV) cp_async16(hs1 + i, Hv + row + i);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float2 v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) {            // clamped row: loads never branch; l >= Q / 2 >= ny: padding
        v[r] = make_float2(0.f, 0.f);
        if (r >= 8) continue;
        const int l = t + TQ * r;
        const float2 x = T1[spec_at(l < ny ? l : ny - 1, k, nk)];
        if (l < ny) v[r] = x;
    }
    fft_strided<float2, false, R3>(v, buf, t, tw);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (mode == CONV_UV) {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int l = t + TQ * r;
            const bool lo = l <= Q / 2;
            const int lq = lo ? l : Q - l;
            const float2 iw = mul_i(v[r]);
            const float hu = hs0[lq];
            keep[spad(l)] = iw * hs1[lq];          // even in l
            v[r] = iw * (lo ? hu : -hu);            // odd in l
        }
        fft_strided<float2, true, R3>(v, buf, t, tw);
#pragma unroll
        for (int r = 0; r < 16; ++r) {               // rows past Q / 2 are not kept
            const int l = t + TQ * r;
            if (r < 8 && l < ny) T2a[spec_at(l, k, nk)] = v[r];
            v[r] = keep[spad(l)];                    // written by this thread
        }
        fft_strided<float2, true, R3>(v, buf, t, tw);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int l = t + TQ * r;
            if (l < ny) T2b[spec_at(l, k, nk)] = v[r];
        }
    } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            const int l = t + TQ * r;
            v[r] = v[r] * hs0[l <= Q / 2 ? l : Q - l];
        }
        fft_strided<float2, true, R3>(v, buf, t, tw);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int l = t + TQ * r;
            if (l < ny) T2a[spec_at(l, k, nk)] = v[r];
        }
    }
}

// Inverse row pass.  A group's complex row is u_j + i v_j (node velocity: one
// row, half spectra from T2a and T2b) or psi_j + i psi_{j+1} (two rows of
// T2a).  Two rows' values of a k come as one 16-byte load.  At most 64
// registers a thread: 1024 threads an SM.
template <int R3>
__global__ void __launch_bounds__(16 * R3 * INV_GROUPS, R3 >= 4 ? 1024 / (16 * R3 * INV_GROUPS) : 1)
    k_rows_inv_r(const float2* __restrict__ T2a, const float2* __restrict__ T2b, float* __restrict__ out, int nx, int ny,
                 int mode, float Uinf, float Vinf, const float2* __restrict__ tw) {
    constexpr int P = 256 * R3, TP = P / 16, SB = SBuf<P>::size, NK = P / 2 + 1, G = INV_GROUPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* bufs = reinterpret_cast<float2*>(smem_raw);
    const int g = threadIdx.x / TP, t = threadIdx.x % TP;
    const bool uv = mode == CONV_UV;
    const int rows = uv ? G : 2 * G;                 // rows of the block
    const int r0 = rows * blockIdx.x;                // <= ny - 1: the rows read from it lie in stored groups of four
    const int h = P / 2;
    pdl_wait();
#pragma unroll 2
    for (int k = threadIdx.x; k <= h; k += blockDim.x) {
        float2 a[G], b[G];
        if (uv) {                                     // group gg takes row r0 + gg
            const size_t at = spec_at(r0, k, NK);       // r0 is even
            ld_pair(T2a + at, a[0], a[1]);
            ld_pair(T2b + at, b[0], b[1]);
#pragma unroll
            for (int gg = 0; gg < G; ++gg)
                if (r0 + gg >= ny) a[gg] = b[gg] = make_float2(0.f, 0.f);
        } else {                                      // group gg takes rows r0 + 2 gg, r0 + 2 gg + 1
#pragma unroll
            for (int gg = 0; gg < G; ++gg) {
                const int j = r0 + 2 * gg;
                ld_pair(T2a + spec_at(j < ny ? j : r0, k, NK), a[gg], b[gg]);
                if (j >= ny) a[gg] = make_float2(0.f, 0.f);
                if (j + 1 >= ny) b[gg] = make_float2(0.f, 0.f);
            }
        }
#pragma unroll
        for (int gg = 0; gg < G; ++gg) {
            float2 x = a[gg], y = b[gg];
            if (k == 0 || k == h) { x.y = 0; y.y = 0; }
            float2* buf = bufs + gg * SB;
            buf[spad(k)] = x + mul_i(y);
            if (k > 0 && k < h) buf[spad(P - k)] = conjc(x) + mul_i(conjc(y));
        }
    }
    __syncthreads();
    float2* buf = bufs + g * SB;
    float2 v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = buf[spad(t + TP * r)];
    __syncthreads();
    fft_strided<float2, true, R3>(v, buf, t, tw);
    if (uv) {
        const int j = r0 + g;
        if (j < ny) {
            float2* o = reinterpret_cast<float2*>(out) + (size_t)j * nx;
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int n = t + TP * r;
                if (n < nx) o[n] = make_float2(v[r].x + Uinf, v[r].y + Vinf);
            }
        }
    } else {
        const int ja = r0 + 2 * g, jb = ja + 1;
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const int n = t + TP * r;
            if (n < nx) {
                if (ja < ny) out[(size_t)ja * nx + n] = v[r].x;
                if (jb < ny) out[(size_t)jb * nx + n] = v[r].y;
            }
        }
    }
}

// workspaces of one convolution (half spectra of the rows, column outputs)
struct ConvWs {
    void* T1;
    void* T2a;
    void* T2b;
};

template <int R3P, int R3Q>
static pf_status conv_solve_r(pf_plan p, const float* w, float* out, int mode, float Uinf, float Vinf, const float* H, const float* Hu,
                              const float* Hv, const float2* twP, const float2* twQ, ConvWs ws) {
    constexpr int P = 256 * R3P, Q = 256 * R3Q;
    const int nx = p->nx, ny = p->ny;
    const size_t sf = FWD_GROUPS * (size_t)SBuf<P>::size * sizeof(float2);
    const size_t sc = 2 * (size_t)SBuf<Q>::size * sizeof(float2) + 2 * (size_t)((Q / 2 + 1 + 3) / 4 * 4) * sizeof(float);
    PF_CUDA(p, set_smem(k_rows_fwd_r<R3P>, sf));
    PF_CUDA(p, set_smem(k_cols_r<R3Q>, sc));
    float2* T1 = reinterpret_cast<float2*>(ws.T1);
    float2* T2a = reinterpret_cast<float2*>(ws.T2a);
    float2* T2b = reinterpret_cast<float2*>(ws.T2b);
    PF_KERNEL(p, "fft_rows_fwd", PF_CUDA(p, pf_launch(k_rows_fwd_r<R3P>, ceil_div(ny, 2 * FWD_GROUPS), 16 * R3P * FWD_GROUPS, sf, p->stream, w, T1,
                                                      nx, ny, twP)));
    PF_KERNEL(p, "fft_cols_conv", PF_CUDA(p, pf_launch(k_cols_r<R3Q>, P / 2 + 1, 16 * R3Q, sc, p->stream, T1, T2a,
                                                       T2b, ny, P / 2 + 1, mode, H, Hu, Hv, p->Hld, twQ)));
    const int nb = mode == CONV_UV ? ceil_div(ny, INV_GROUPS) : ceil_div(ny, 2 * INV_GROUPS);
    const size_t sr = INV_GROUPS * (size_t)SBuf<P>::size * sizeof(float2);
    PF_CUDA(p, set_smem(k_rows_inv_r<R3P>, sr));
    PF_KERNEL(p, "fft_rows_inv", PF_CUDA(p, pf_launch(k_rows_inv_r<R3P>, nb, 16 * R3P * INV_GROUPS, sr, p->stream, T2a, T2b,
                                                      out, nx, ny, mode, Uinf, Vinf, twP)));
    return PF_OK;
}

template <int R3P>
static pf_status conv_dispatch_q(pf_plan p, const float* w, float* out, int mode, float Uinf, float Vinf, const float* H, const float* Hu,
                                 const float* Hv, const float2* twP, const float2* twQ, ConvWs ws) {
    switch (p->Q) {
        case 256: return conv_solve_r<R3P, 1>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 512: return conv_solve_r<R3P, 2>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 1024: return conv_solve_r<R3P, 4>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 2048: return conv_solve_r<R3P, 8>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 4096: return conv_solve_r<R3P, 16>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
    }
    return PF_ERR_ARG;
}

static pf_status conv_dispatch(pf_plan p, const float* w, float* out, int mode, float Uinf, float Vinf, const float* H, const float* Hu,
                               const float* Hv, const float2* twP, const float2* twQ, ConvWs ws) {
    switch (p->P) {
        case 256: return conv_dispatch_q<1>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 512: return conv_dispatch_q<2>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 1024: return conv_dispatch_q<4>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 2048: return conv_dispatch_q<8>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
        case 4096: return conv_dispatch_q<16>(p, w, out, mode, Uinf, Vinf, H, Hu, Hv, twP, twQ, ws);
    }
    return PF_ERR_ARG;
}

template <typename T>
static pf_status conv_solve_t(pf_plan p, const T* w, T* out, int mode, T Uinf, T Vinf, const T* H, const T* Hu,
                              const T* Hv, const C_t<T>* twP, const C_t<T>* twQ, ConvWs ws) {
    using C = C_t<T>;
    const int P = p->P, Q = p->Q, nx = p->nx, ny = p->ny;
    // the third column buffer holds the second component (mode CONV_UV) only
    const size_t sr = 2 * (size_t)P * sizeof(C), sc = (mode == CONV_UV ? 3 : 2) * (size_t)Q * sizeof(C);
    PF_CUDA(p, set_smem(k_rows_fwd<T>, sr));
    PF_CUDA(p, set_smem(k_cols<T>, sc));
    PF_CUDA(p, set_smem(k_rows_inv<T>, sr));
    C* T1 = reinterpret_cast<C*>(ws.T1);
    C* T2a = reinterpret_cast<C*>(ws.T2a);
    C* T2b = reinterpret_cast<C*>(ws.T2b);
    PF_KERNEL(p, "fft_rows_fwd", k_rows_fwd<T><<<(ny + 1) / 2, 256, sr, p->stream>>>(w, T1, nx, ny, P, twP));
    PF_KERNEL(p, "fft_cols_conv", k_cols<T><<<P / 2 + 1, 256, sc, p->stream>>>(T1, T2a, T2b, ny, Q, mode, H, Hu, Hv, p->Hld, twQ));
    const int nb = mode == CONV_UV ? ny : (ny + 1) / 2;
    PF_KERNEL(p, "fft_rows_inv", k_rows_inv<T><<<nb, 256, sr, p->stream>>>(T2a, T2b, out, nx, ny, P, mode, Uinf, Vinf, twP));
    return PF_OK;
}

pf_status conv_solve(pf_plan p, const void* w, void* out, int mode, double Uinf, double Vinf) {
    // register-resident kernels unless the plan is configured for the shared-memory
    // ones; grids below 256 x 256 padded nodes always take the shared-memory ones
    const bool reg = p->fft_impl == 0 && p->P >= 256 && p->Q >= 256;
    const ConvWs ws{p->T1, p->T2a, p->T2b};
    if (p->prec == PF_FP64) {
        if (reg) return conv_fx(p, (const double*)w, (double*)out, mode, Uinf, Vinf);
        return conv_solve_t<double>(p, (const double*)w, (double*)out, mode, Uinf, Vinf, p->H64, p->Hu64, p->Hv64,
                                    p->twP64, p->twQ64, ws);
    }
    if (reg)
        return conv_dispatch(p, (const float*)w, (float*)out, mode, (float)Uinf, (float)Vinf, p->H32, p->Hu32,
                                    p->Hv32, p->twP32_r, p->twQ32_r, ws);
    return conv_solve_t<float>(p, (const float*)w, (float*)out, mode, (float)Uinf, (float)Vinf, p->H32, p->Hu32,
                               p->Hv32, p->twP32, p->twQ32, ws);
}
