// Shared-memory FFTs for the Radon preconditioner (Section 2.4, Eq. Aprecon).
//
//  * H on sinograms: one block per view, the real line of length P as a complex
//    one of length P/2 (even bins + i odd bins), split into the spectra of the
//    even and odd bins for the gain and put together again.
//  * V^-1 / V on images: a 2-D zero-padded FFT done as row FFTs, column FFTs
//    with the radial gain applied between the forward and inverse column
//    transforms, and inverse row FFTs.  It runs once per solve.
//
// The transform (fft_device.cuh) is a Stockham autosort FFT with radix-8
// stages, in shared memory.
#include <algorithm>

#include "fft_device.cuh"

namespace dgct {

// one thread per radix-8 butterfly, 32 to 512 threads
static int fft_threads(int P) { return P / 8 < 32 ? 32 : (P / 8 > 512 ? 512 : P / 8); }

// ------------------------------------------------------------ H on views --
// One view per block.  With z[j] = x[2j] + i x[2j + 1] and Z its DFT of length
// L = P / 2, the even and odd bins' DFTs are E = (Z[k] + conj Z[L-k]) / 2 and
// O = (Z[k] - conj Z[L-k]) / 2i, and x's own are E +- w^k O at k and k + L,
// w = exp(-2 pi i / P).  With these times the gains g[k] and g[k + L] = g[L-k] as
// A and C, E' = (A + C) / 2 and O' = w^-k (A - C) / 2, and Z' = E' + i O' (at L-k:
// conj E' + i conj O') transforms back to the filtered bins.  (Gathering E and O
// by (g[k] +- g[L-k]) instead saves an addition each, but lets the high
// frequencies' rounding into the low ones, which A^T then amplifies.)
//
// E - w^k O cancels at the low frequencies, where most of a sinogram lies, and the
// gain then raises what is left of the roundings; so E, O, w^k and the products
// keep their low parts up to that difference (filter_split).  Against 64 bits H is
// then as close as by two views in one complex line of length P (k_filter_pairs;
// 0.98-1.0 of its error over 24 geometries), where plain FP32 was 4-5% off it.
// The block's chain of stages and barriers bounds the kernel, not its arithmetic:
// 64 x 729 takes 5.8 us with or without the low parts, pairs of views 9.0;
// 90 x 1449 7.3 against 12.1.
struct TwoPart {
    float hi, lo;
};
__device__ __forceinline__ TwoPart two_sum(float a, float b) {      // Knuth: hi + lo = a + b exactly
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}

// E + d and E - d for d = c a + s b, c and s in two parts (w.x + w.z, w.y + w.w)
__device__ __forceinline__ void add_and_subtract(TwoPart E, TwoPart a, TwoPart b, float c, float s, float cl, float sl,
                                                 float& plus, float& minus) {
    const float p = __fmul_rn(c, a.hi), q = __fmul_rn(s, b.hi);
    const TwoPart d = two_sum(p, q);
    float lo = fmaf(c, a.hi, -p) + fmaf(s, b.hi, -q) + d.lo;
    lo = fmaf(c, a.lo, fmaf(s, b.lo, fmaf(cl, a.hi, fmaf(sl, b.hi, lo))));
    plus = __fadd_rn(__fadd_rn(E.hi, d.hi), E.lo + lo);
    minus = __fadd_rn(__fsub_rn(E.hi, d.hi), E.lo - lo);
}

// 2 (E + w^k O) and 2 (E - w^k O) from Z[k] and Z[L-k]; w = exp(2 pi i k / P) in two parts
__device__ __forceinline__ void filter_split(float2 z, float2 y, float4 w, float2& plus, float2& minus) {
    const TwoPart Ex = two_sum(z.x, y.x), Ey = two_sum(z.y, -y.y), Ox = two_sum(z.y, y.y), Oy = two_sum(y.x, -z.x);
    add_and_subtract(Ex, Ox, Oy, w.x, w.y, w.z, w.w, plus.x, minus.x);
    add_and_subtract(Ey, Oy, Ox, w.x, -w.y, w.z, -w.w, plus.y, minus.y);
}

template <typename T>
__global__ void __launch_bounds__(512)
k_filter_line(const T* in, T* out, int nd, int P, const float* __restrict__ gain, const float2* __restrict__ tw,
              const float4* __restrict__ wk) {
    extern __shared__ float2 smem[];
    const int L = P >> 1;
    float2* a = smem;
    float2* b = smem + fft_buf_len(L);
    const T* row = in + (size_t)blockIdx.x * nd;
    pdl_wait();
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        float2 v = make_float2(0.f, 0.f);
        if (2 * i < nd) v.x = ldf(row + 2 * i);
        if (2 * i + 1 < nd) v.y = ldf(row + 2 * i + 1);
        a[fpad(i)] = v;
    }
    __syncthreads();
    float2* r = fft_stockham(a, b, L, tw, -1.f);
    float2* o = (r == a) ? b : a;
    const float sc = 0.25f / (float)L;      // the two halvings above, and 1 / L of the inverse
    for (int k = threadIdx.x; k <= L / 2; k += blockDim.x) {
        const int kk = (L - k) & (L - 1);
        const float2 z = r[fpad(k)], y = r[fpad(kk)];
        const float ga = __ldg(gain + k) * sc, gb = __ldg(gain + L - k) * sc;
        const float4 w = wk[k];                                                                      // w^-k
        float2 A, C;
        filter_split(z, y, w, A, C);
        A = make_float2(ga * A.x, ga * A.y);
        C = make_float2(gb * C.x, gb * C.y);
        const float2 e = cadd(A, C), q = cmul(csub(A, C), make_float2(w.x, w.y));
        r[fpad(k)] = make_float2(e.x - q.y, e.y + q.x);
        if (kk != k) r[fpad(kk)] = make_float2(e.x + q.y, q.x - e.y);
    }
    __syncthreads();
    r = fft_stockham(r, o, L, tw, 1.f);
    T* w = out + (size_t)blockIdx.x * nd;
    for (int i = threadIdx.x; i < nd; i += blockDim.x) {
        const float2 v = r[fpad(i >> 1)];
        stf(w + i, (i & 1) ? v.y : v.x);
    }
}

// Two views per block as one complex line of length P, which the real and even
// gain filters both: the arithmetic of the fused sinogram kernel's FFT form, for
// Laplace solves that run it as a kernel of its own (filter_form).
template <typename T>
__global__ void __launch_bounds__(512)
k_filter_pairs(const T* in, T* out, int nv, int nd, int P,
               const float* __restrict__ gain, const float2* __restrict__ tw) {
    extern __shared__ float2 smem[];
    float2* a = smem;
    float2* b = smem + fft_buf_len(P);
    const int va = 2 * blockIdx.x, vb = va + 1;
    const bool hasb = vb < nv;
    const T* ra = in + (size_t)va * nd;
    const T* rb = in + (size_t)vb * nd;
    pdl_wait();
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        float2 v = make_float2(0.f, 0.f);
        if (i < nd) {
            v.x = ldf(ra + i);
            if (hasb) v.y = ldf(rb + i);
        }
        a[fpad(i)] = v;
    }
    __syncthreads();
    float2* r = fft_stockham(a, b, P, tw, -1.f);
    float2* o = (r == a) ? b : a;
    for (int i = threadIdx.x; i < P; i += blockDim.x) {
        const float g = __ldg(gain + i);
        const float2 v = r[fpad(i)];
        r[fpad(i)] = make_float2(v.x * g, v.y * g);
    }
    __syncthreads();
    r = fft_stockham(r, o, P, tw, 1.f);
    const float sc = 1.0f / (float)P;
    T* wa = out + (size_t)va * nd;
    T* wb = out + (size_t)vb * nd;
    for (int i = threadIdx.x; i < nd; i += blockDim.x) {
        const float2 v = r[fpad(i)];
        stf(wa + i, v.x * sc);
        if (hasb) stf(wb + i, v.y * sc);
    }
}

// ------------------------------------------------- H as a Toeplitz product --
// The same operator without an FFT: with zero padding to P >= 2 n_det there
// is no wrap-around, so (H z)[d] = sum_d' h[|d - d'|] z[d'] with
// h = IFFT_P(g) (real and even), computed in FP64 at plan time and stored as
// hx[m + n_det - 1] = h[|m|] for m in (-n_det, n_det).  Block = one view x
// 128 outputs; each lane keeps 4 consecutive outputs (a sliding window of
// hx in registers) and the 8 warps split the d' range, their partial sums
// added in a fixed order.
constexpr int kTzOut = 128, kTzWarps = 8;

template <typename T>
__global__ void __launch_bounds__(32 * kTzWarps)
k_filter_toeplitz(const T* in, T* out, int nd, const float* __restrict__ hx) {
    extern __shared__ float sm[];
    float* zs = sm;                       // [nd]
    float* hs = sm + nd;                  // [2 nd - 1]
    float* red = hs + 2 * nd - 1;         // [kTzWarps][kTzOut]
    const int v = blockIdx.y;
    const int d0 = blockIdx.x * kTzOut;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const T* row = in + (size_t)v * nd;
    for (int i = tid; i < 2 * nd - 1; i += blockDim.x) hs[i] = hx[i];      // plan constants: before the wait
    pdl_wait();
    for (int i = tid; i < nd; i += blockDim.x) zs[i] = ldf(row + i);
    __syncthreads();
    const int dl = d0 + 4 * lane;          // this lane's first output
    const int len = (nd + kTzWarps - 1) / kTzWarps;
    const int p0 = w * len, p1 = min(nd, p0 + len);
    float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
    if (dl < nd && p0 < p1) {
        // output dl + i at input d' uses hs[dl + i - d' + nd - 1]
        int base = dl - p0 + nd - 1;
        float h0 = hs[base], h1 = hs[min(base + 1, 2 * nd - 2)], h2 = hs[min(base + 2, 2 * nd - 2)],
              h3 = hs[min(base + 3, 2 * nd - 2)];
        for (int dp = p0; dp < p1; ++dp) {
            const float zv = zs[dp];
            a0 = fmaf(h0, zv, a0);
            a1 = fmaf(h1, zv, a1);
            a2 = fmaf(h2, zv, a2);
            a3 = fmaf(h3, zv, a3);
            // next d' shifts every index down by one
            h3 = h2;
            h2 = h1;
            h1 = h0;
            --base;
            h0 = base >= 0 ? hs[base] : 0.f;
        }
    }
    red[w * kTzOut + 4 * lane + 0] = a0;
    red[w * kTzOut + 4 * lane + 1] = a1;
    red[w * kTzOut + 4 * lane + 2] = a2;
    red[w * kTzOut + 4 * lane + 3] = a3;
    __syncthreads();
    for (int o = tid; o < kTzOut; o += blockDim.x) {
        const int d = d0 + o;
        if (d >= nd) continue;
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < kTzWarps; ++k) t += red[k * kTzOut + o];
        stf(out + (size_t)v * nd + d, t);
    }
}

static size_t toeplitz_smem(int nd) {
    return ((size_t)nd + 2 * nd - 1 + kTzWarps * kTzOut) * sizeof(float);
}

// H's form for launch_filter.  The single steps, and a solve with exact moments,
// take the plan's timed choice between the line per view and the Toeplitz product.
// A Laplace solve runs the three kernels only if told to (sino_fused = 0), beside
// the fused FFT form, and takes that form's arithmetic unless the tuning has set
// the Toeplitz product: the two then agree bit for bit, where another order of
// summation parts them by up to 1.6e-4 in tau_r over five iterations of a 16 x 16
// image (3 views of 24 bins).
enum FilterForm { kFilterLine, kFilterPairs, kFilterToeplitz };
static FilterForm filter_form(const dgamp_ct_plan_s* pl, int solve) {
    const bool laplace = solve && !pl->opt.output_moments;
    if (pl->filter_mode == 1 && (!laplace || pl->filter_set)) return kFilterToeplitz;
    return laplace ? kFilterPairs : kFilterLine;
}

template <typename T>
static int launch_filter_t(const dgamp_ct_plan_s* pl, FilterForm form, const T* in, T* out, cudaStream_t st) {
    const int P = pl->P;
    if (form == kFilterToeplitz) {
        // the block reads its whole input row first, so in == out needs a copy
        const T* src = in;
        if (in == out) {
            DGCT_CUDA(cudaMemcpyAsync(pl->ws.zraw2, in, (size_t)pl->M * sizeof(T), cudaMemcpyDeviceToDevice, st));
            src = (const T*)pl->ws.zraw2;
        }
        DGCT_CUDA(launch_pdl(k_filter_toeplitz<T>, dim3((pl->nd + kTzOut - 1) / kTzOut, pl->nv), dim3(32 * kTzWarps),
                             toeplitz_smem(pl->nd), st, src, out, pl->nd, pl->ws.hx));
        return DGAMP_CT_OK;
    }
    if (form == kFilterPairs) {
        DGCT_CUDA(launch_pdl(k_filter_pairs<T>, dim3((pl->nv + 1) / 2), dim3(fft_threads(P)),
                             (size_t)2 * fft_buf_len(P) * sizeof(float2), st, in, out, pl->nv, pl->nd, P, pl->ws.gain,
                             pl->ws.tw));
        return DGAMP_CT_OK;
    }
    DGCT_CUDA(launch_pdl(k_filter_line<T>, dim3(pl->nv), dim3(fft_threads(P / 2)),
                         (size_t)2 * fft_buf_len(P / 2) * sizeof(float2), st, in, out, pl->nd, P, pl->ws.gain,
                         pl->ws.twh, pl->ws.twk));
    return DGAMP_CT_OK;
}

// bf = 1: in and out hold BF16 (a solve with storage = 1); sums in FP32 either way
int launch_filter(const dgamp_ct_plan_s* pl, const float* in, float* out, cudaStream_t st, int bf, int solve) {
    const FilterForm form = filter_form(pl, solve);
    return bf ? launch_filter_t(pl, form, (const bf16s*)in, (bf16s*)out, st) : launch_filter_t(pl, form, in, out, st);
}

// Plan-time choice between the FFT and the Toeplitz form of H (same operator):
// time both on the plan's geometry and keep the faster.
int filter_autotune(dgamp_ct_plan_s* pl) {
    DGCT_CUDA(cudaMemset(pl->ws.zraw, 0, (size_t)pl->M * sizeof(float)));
    cudaEvent_t e0, e1;
    DGCT_CUDA(cudaEventCreate(&e0));
    DGCT_CUDA(cudaEventCreate(&e1));
    float best = 1e30f;
    int best_mode = 0, rc = DGAMP_CT_OK;
    for (int mode = 0; mode < 2 && rc == DGAMP_CT_OK; ++mode) {
        pl->filter_mode = mode;
        for (int rep = 0; rep < 6 && rc == DGAMP_CT_OK; ++rep) {
            if (rep == 1) cudaEventRecord(e0, 0);
            rc = launch_filter(pl, pl->ws.zraw, pl->ws.z, 0);
        }
        cudaEventRecord(e1, 0);
        const cudaError_t e = cudaEventSynchronize(e1);
        if (rc == DGAMP_CT_OK && e != cudaSuccess) rc = cuda_fail(e);
        float ms = 0.f;
        if (rc == DGAMP_CT_OK) cudaEventElapsedTime(&ms, e0, e1);
        if (rc == DGAMP_CT_OK && ms < best) {
            best = ms;
            best_mode = mode;
        }
    }
    pl->filter_mode = best_mode;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}

int toeplitz_set_smem_limit(int nd) {
    const size_t need = toeplitz_smem(nd);
    DGCT_TRY(raise_smem_limit((const void*)k_filter_toeplitz<float>, (int)need));
    DGCT_TRY(raise_smem_limit((const void*)k_filter_toeplitz<bf16s>, (int)need));
    return DGAMP_CT_OK;
}

// ------------------------------------------------------- V^-1 / V image --
// Image blockIdx.y of a batch (img and out [nimg][n][n], C [nimg][n][m]);
// a single image is the batch of one.  The passes are in fft_device.cuh.
__global__ void __launch_bounds__(512)
k_img_rows_fwd(const float* __restrict__ img, int n, int m, const float2* __restrict__ tw,
               float2* __restrict__ C) {
    extern __shared__ float2 smem[];
    pdl_wait();
    img_rows_fwd_block(img + (size_t)blockIdx.y * n * n, n, m, blockIdx.x, tw, C + (size_t)blockIdx.y * n * m, smem);
}

__global__ void __launch_bounds__(512)
k_img_cols(float2* __restrict__ C, int n, int m, const float2* __restrict__ tw, float f0,
           int inverse_gain) {
    extern __shared__ float2 smem[];
    pdl_wait();
    img_cols_block(C + (size_t)blockIdx.y * n * m, n, m, blockIdx.x, tw, f0, inverse_gain, smem);
}

// pass 3: inverse row FFTs, real part of the first n columns, scaled by 1/m^2.
__global__ void __launch_bounds__(512)
k_img_rows_inv(const float2* __restrict__ C, int n, int m, const float2* __restrict__ tw,
               float* __restrict__ out) {
    extern __shared__ float2 smem[];
    const int y = blockIdx.x;
    pdl_wait();
    const float2* r = img_rows_inv_block(C + (size_t)blockIdx.y * n * m, m, y, tw, smem);
    out += (size_t)blockIdx.y * n * n + (size_t)y * n;
    const float sc = 1.0f / ((float)m * (float)m);
    for (int i = threadIdx.x; i < n; i += blockDim.x) out[i] = r[fpad(i)].x * sc;
}

// pass 3 of V^-1 inside a fan-beam solve (Algorithm 1, Step 3 with
// Phi~^T = V^-1 A^T): r = x + tau_r Re(.) / m^2 with tau_r from the device
// scalars (the output step formed it), max |r| into S->rmax_bits (the output
// step reset it), and the consumed divergence flag cleared, as the
// parallel-beam back-projection does.
__global__ void __launch_bounds__(512)
k_img_rows_inv_update(const float2* __restrict__ C, int n, int m, const float2* __restrict__ tw,
                      const float* __restrict__ x, DevScalars* __restrict__ S, float* __restrict__ out) {
    extern __shared__ float2 smem[];
    __shared__ unsigned s_max;
    const int y = blockIdx.x;
    pdl_wait();
    if (threadIdx.x == 0) {
        s_max = 0u;
        if (y == 0) S->div_pending = 0u;
    }
    const float2* r = img_rows_inv_block(C, m, y, tw, smem);
    const float sc = (float)S->tau_r / ((float)m * (float)m);
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const size_t o = (size_t)y * n + i;
        const float rv = fmaf(sc, r[fpad(i)].x, x[o]);
        out[o] = rv;
        atomicMax(&s_max, __float_as_uint(fabsf(rv)));   // |r| >= 0: bit order is value order
    }
    __syncthreads();
    if (threadIdx.x == 0) atomicMax(&S->rmax_bits, s_max);
}

// The two first passes of nimg images.
static int launch_img_forward(const dgamp_ct_plan_s* pl, const float* in, float2* C, int nimg, int inverse_gain,
                              cudaStream_t st) {
    const int n = pl->n, m = pl->m2, thr = fft_threads(m), nc = img_cols_per_block(m);
    const size_t sm = (size_t)2 * fft_buf_len(m) * sizeof(float2);
    const float f0 = 1.0f / (2.0f * (float)pl->P);
    DGCT_CUDA(launch_pdl(k_img_rows_fwd, dim3(n, nimg), dim3(thr), sm, st, in, n, m, pl->ws.tw2, C));
    // V^-1 applies sqrt(max(rho, f0)); V applies its reciprocal
    DGCT_CUDA(launch_pdl(k_img_cols, dim3(m / nc, nimg), dim3(thr, nc), nc * sm, st, C, n, m, pl->ws.tw2,
                         f0, inverse_gain));
    return DGAMP_CT_OK;
}

int launch_precond_image_update(const dgamp_ct_plan_s* pl, const float* in, const float* x, float* out,
                                cudaStream_t st) {
    const int n = pl->n, m = pl->m2;
    const size_t sm = (size_t)2 * fft_buf_len(m) * sizeof(float2);
    DGCT_TRY(launch_img_forward(pl, in, pl->ws.fft2d, 1, 0, st));
    DGCT_CUDA(launch_pdl(k_img_rows_inv_update, dim3(n), dim3(fft_threads(m)), sm, st, pl->ws.fft2d, n, m,
                         pl->ws.tw2, x, pl->ws.S, out));
    return DGAMP_CT_OK;
}

int launch_precond_image(const dgamp_ct_plan_s* pl, const float* in, float* out, int inverse,
                         cudaStream_t st) {
    return launch_precond_images(pl, in, out, pl->ws.fft2d, 1, inverse, st);
}

// nimg images at once ([nimg][n][n] in and out) through the scratch C
// ([nimg][n][m2] complex, the caller's); the same kernels and arithmetic per
// image as launch_precond_image
int launch_precond_images(const dgamp_ct_plan_s* pl, const float* in, float* out, float2* C, int nimg, int inverse,
                          cudaStream_t st) {
    if (nimg < 1) return DGAMP_CT_ERR_INVALID_ARG;
    const int n = pl->n, m = pl->m2;
    const size_t sm = (size_t)2 * fft_buf_len(m) * sizeof(float2);
    DGCT_TRY(launch_img_forward(pl, in, C, nimg, inverse ? 0 : 1, st));
    DGCT_CUDA(launch_pdl(k_img_rows_inv, dim3(n, nimg), dim3(fft_threads(m)), sm, st, C, n, m, pl->ws.tw2, out));
    return DGAMP_CT_OK;
}

int fft_set_smem_limits(int bytes) {
    DGCT_TRY(raise_smem_limit((const void*)k_filter_line<float>, bytes));
    DGCT_TRY(raise_smem_limit((const void*)k_filter_line<bf16s>, bytes));
    DGCT_TRY(raise_smem_limit((const void*)k_filter_pairs<float>, bytes));
    DGCT_TRY(raise_smem_limit((const void*)k_filter_pairs<bf16s>, bytes));
    DGCT_TRY(raise_smem_limit((const void*)k_img_rows_fwd, bytes));
    // several columns a block up to m = 2048: 4 at 1024 and 2 at 2048 need the same 74 KB
    DGCT_TRY(raise_smem_limit((const void*)k_img_cols,
                              std::max(bytes, (int)(4 * 2 * fft_buf_len(1024) * sizeof(float2)))));
    DGCT_TRY(raise_smem_limit((const void*)k_img_rows_inv, bytes));
    DGCT_TRY(raise_smem_limit((const void*)k_img_rows_inv_update, bytes));
    return DGAMP_CT_OK;
}

}  // namespace dgct
