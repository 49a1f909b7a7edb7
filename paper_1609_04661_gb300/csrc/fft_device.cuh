// Shared-memory FFT used by the detector-axis preconditioner H (Section 2.4,
// Eq. Aprecon) and the image-domain V^-1 (Algorithm 1, last step).
//
// The transform is a Stockham autosort FFT (natural order in and out,
// ping-pong between two shared-memory buffers) with radix-8 stages and one
// final radix-4 or radix-2 stage when log2 P is not a multiple of 3.  With
// Ns = the product of the radices already applied, butterfly j (of P/R)
// reads a[j + r P/R], r < R, multiplies input r by w^(r k) with k = j mod Ns
// and w = exp(-+ 2 pi i / (Ns R)), takes the R-point DFT in registers and
// writes output q to b[(j - k) R + k + q Ns].
//
// Shared-memory layout.  Element i of a buffer lives at fpad(i) = i + i/8
// (a buffer of P elements takes fft_buf_len(P) = P + P/8 slots): the first
// stage's stores b[8 j + q] and the second's fall on distinct banks for the
// 16 lanes of a 64-bit access, which without the padding collide 8- and
// 4-fold.  Twiddles are stored stage by stage (fft_twiddle_count(P) values):
// for every stage with Ns > 1, the (R - 1) Ns values exp(2 pi i r k / (Ns R))
// at [(r - 1) Ns + k], so the lanes of a warp read consecutive words.
#pragma once
#include "internal.cuh"

namespace dgct {

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// c * (dir i)
__device__ __forceinline__ float2 cmul_i(float2 c, float dir) { return make_float2(-dir * c.y, dir * c.x); }

// In-place R-point DFT X_q = sum_r v_r exp(dir 2 pi i r q / R), R = 2, 4, 8,
// by radix-2 splitting (even / odd inputs).
template <int R> __device__ __forceinline__ void dft_small(float2* v, float dir);

template <> __device__ __forceinline__ void dft_small<2>(float2* v, float) {
    const float2 t = v[0];
    v[0] = cadd(t, v[1]);
    v[1] = csub(t, v[1]);
}

__device__ __forceinline__ void dft4(float2 a0, float2 a1, float2 a2, float2 a3, float dir, float2* X) {
    const float2 e0 = cadd(a0, a2), e1 = csub(a0, a2);
    const float2 o0 = cadd(a1, a3), o1 = cmul_i(csub(a1, a3), dir);
    X[0] = cadd(e0, o0);
    X[1] = cadd(e1, o1);
    X[2] = csub(e0, o0);
    X[3] = csub(e1, o1);
}

template <> __device__ __forceinline__ void dft_small<4>(float2* v, float dir) {
    float2 X[4];
    dft4(v[0], v[1], v[2], v[3], dir, X);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = X[q];
}

template <> __device__ __forceinline__ void dft_small<8>(float2* v, float dir) {
    float2 E[4], O[4];
    dft4(v[0], v[2], v[4], v[6], dir, E);
    dft4(v[1], v[3], v[5], v[7], dir, O);
    const float s = 0.70710678118654752f;   // 1/sqrt(2)
    // W^q O_q with W = exp(dir 2 pi i / 8): W = (1 + dir i)/sqrt2, W^2 = dir i, W^3 = (-1 + dir i)/sqrt2
    const float2 t1 = make_float2(s * (O[1].x - dir * O[1].y), s * (dir * O[1].x + O[1].y));
    const float2 t2 = cmul_i(O[2], dir);
    const float2 t3 = make_float2(s * (-O[3].x - dir * O[3].y), s * (dir * O[3].x - O[3].y));
    v[0] = cadd(E[0], O[0]);
    v[4] = csub(E[0], O[0]);
    v[1] = cadd(E[1], t1);
    v[5] = csub(E[1], t1);
    v[2] = cadd(E[2], t2);
    v[6] = csub(E[2], t2);
    v[3] = cadd(E[3], t3);
    v[7] = csub(E[3], t3);
}

__host__ __device__ __forceinline__ int fpad(int i) { return i + (i >> 3); }
__host__ __device__ __forceinline__ int fft_buf_len(int P) { return P + P / 8 + 1; }

// Radices of the stages: 8 while Ns * 8 <= P, then 4 or 2 for the rest.
__host__ __device__ __forceinline__ int fft_stage_radix(int P, int Ns) {
    return Ns * 8 <= P ? 8 : (Ns * 4 == P ? 4 : (Ns * 2 == P ? 2 : 1));
}
__host__ __device__ __forceinline__ int fft_twiddle_count(int P) {
    int cnt = 0;
    for (int Ns = 1, R = fft_stage_radix(P, 1); R > 1; Ns *= R, R = fft_stage_radix(P, Ns))
        if (Ns > 1) cnt += (R - 1) * Ns;
    return cnt;
}

// One stage; tws = this stage's twiddles; dir = -1 forward, +1 inverse.
template <int R>
__device__ __forceinline__ void stockham_stage(const float2* a, float2* b, int P, int Ns,
                                               const float2* tws, float dir) {
    const int nb = P / R;
    for (int j = threadIdx.x; j < nb; j += blockDim.x) {
        const int k = j & (Ns - 1);
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = a[fpad(j + r * nb)];
        if (Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) {
                float2 w = tws[(r - 1) * Ns + k];
                w.y *= dir;
                v[r] = cmul(v[r], w);
            }
        }
        dft_small<R>(v, dir);
        const int o = (j - k) * R + k;
#pragma unroll
        for (int q = 0; q < R; ++q) b[fpad(o + q * Ns)] = v[q];
    }
}

// Transforms a[0..P) (P a power of two, padded layout); returns the buffer
// holding the result.  Every thread of the block takes part; tw (the
// stage-by-stage table) may point to global or shared memory.
__device__ __forceinline__ float2* fft_stockham(float2* a, float2* b, int P, const float2* tw, float dir) {
    int off = 0;
    for (int Ns = 1, R = fft_stage_radix(P, 1); R > 1; Ns *= R, R = fft_stage_radix(P, Ns)) {
        if (R == 8)
            stockham_stage<8>(a, b, P, Ns, tw + off, dir);
        else if (R == 4)
            stockham_stage<4>(a, b, P, Ns, tw + off, dir);
        else
            stockham_stage<2>(a, b, P, Ns, tw + off, dir);
        if (Ns > 1) off += (R - 1) * Ns;
        __syncthreads();
        float2* t = a;
        a = b;
        b = t;
    }
    return a;
}

// ------------------------------------------------ V^-1 / V of an image --
// The 2-D filter of an n x n real image on its m x m zero-padded grid, in three
// passes over the spectrum C [n][m], shared by the single and the batched
// kernels: rows, columns with the radial gain between their forward and inverse
// transforms, rows back.  A block takes NC neighbouring columns, so that the
// row-major spectrum is read in whole sectors.  The rows' conjugate symmetry is
// not used: two rows as one complex line and half the columns halve the work,
// but the error of V^-1 x against 64 bits grows by a quarter (2.0e-7 -> 2.5e-7
// over 64^2 .. 1024^2), since the discarded imaginary parts and the mirrored
// frequencies then no longer take their share of the rounding.
__host__ __device__ __forceinline__ int img_cols_per_block(int m) { return m <= 1024 ? 4 : (m <= 2048 ? 2 : 1); }

// row y of img -> C
__device__ __forceinline__ void img_rows_fwd_block(const float* __restrict__ img, int n, int m, int y,
                                                   const float2* __restrict__ tw, float2* __restrict__ C,
                                                   float2* smem) {
    float2* a = smem;
    float2* b = smem + fft_buf_len(m);
    for (int i = threadIdx.x; i < m; i += blockDim.x)
        a[fpad(i)] = make_float2(i < n ? img[(size_t)y * n + i] : 0.f, 0.f);
    __syncthreads();
    const float2* r = fft_stockham(a, b, m, tw, -1.f);
    for (int i = threadIdx.x; i < m; i += blockDim.x) C[(size_t)y * m + i] = r[fpad(i)];
}

// columns NC bx + threadIdx.y (blockDim.y = NC, which divides m): forward
// transform over the rows (rows >= n are zero), radial gain sqrt(max(rho, f0))
// or its reciprocal, inverse transform; rows < n are stored back.
__device__ __forceinline__ void img_cols_block(float2* __restrict__ C, int n, int m, int bx,
                                               const float2* __restrict__ tw, float f0, int inverse_gain,
                                               float2* smem) {
    const int NC = blockDim.y, kx0 = bx * NC, BL = fft_buf_len(m);
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nt = blockDim.x * NC, sh = __ffs(NC) - 1;   // NC = 1, 2, 4
    for (int j = tid; j < m * NC; j += nt) {       // NC columns of a row are neighbours in memory
        const int i = j >> sh, c = j & (NC - 1);
        smem[2 * c * BL + fpad(i)] = i < n ? C[(size_t)i * m + kx0 + c] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    float2* a = smem + 2 * threadIdx.y * BL;
    float2* r = fft_stockham(a, a + BL, m, tw, -1.f);
    float2* o = (r == a) ? a + BL : a;
    const int kx = kx0 + threadIdx.y;
    const float fx = (float)(kx <= m / 2 ? kx : kx - m) / (float)m;
    for (int ky = threadIdx.x; ky < m; ky += blockDim.x) {
        const float fy = (float)(ky <= m / 2 ? ky : ky - m) / (float)m;
        const float rho = sqrtf(fx * fx + fy * fy);
        float g = sqrtf(fmaxf(rho, f0));
        if (inverse_gain) g = 1.0f / g;
        const float2 v = r[fpad(ky)];
        r[fpad(ky)] = make_float2(v.x * g, v.y * g);
    }
    __syncthreads();
    r = fft_stockham(r, o, m, tw, 1.f);
    const int at = (int)(r - a);                   // the same buffer of every column
    for (int j = tid; j < n * NC; j += nt) {
        const int i = j >> sh, c = j & (NC - 1);
        C[(size_t)i * m + kx0 + c] = smem[2 * c * BL + at + fpad(i)];
    }
}

// inverse transform of row y: its first n values (times m^2) are the real parts
// of the returned buffer
__device__ __forceinline__ const float2* img_rows_inv_block(const float2* __restrict__ C, int m, int y,
                                                            const float2* __restrict__ tw, float2* smem) {
    float2* a = smem;
    float2* b = smem + fft_buf_len(m);
    for (int i = threadIdx.x; i < m; i += blockDim.x) a[fpad(i)] = C[(size_t)y * m + i];
    __syncthreads();
    return fft_stockham(a, b, m, tw, 1.f);
}

}  // namespace dgct
