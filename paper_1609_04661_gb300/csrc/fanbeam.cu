// Flat-detector fan beam (Section 6; option of the plan, dgamp_ct_plan_fan):
// the Joseph projector A along each ray's own direction, its
// transpose, and ||Phi~||_F^2 for Phi~ = A V^-1 (Eq. precondAMP_op with the
// image-domain cone filter; the detector-axis form H A is a parallel-beam
// identity and does not apply).
//
// Geometry (pixel units, pixel centres as for parallel beam): at view angle
// theta the source sits at S = -dso e_c with e_c = (-sin, cos), the detector
// centre at ddo e_c, and bin d at the detector centre plus u_d e_u with
// e_u = (cos, sin), u_d = (d - (n_det-1)/2) du.  Ray d runs along
// v = T_d - S.  A ray with |v_x| >= |v_y| is marched by columns: in column s
// it sits at the fractional row a0 + s a_step, a_step = -v_y / v_x, and the
// linear interpolation between the two nearest rows is weighted by
// w = |v| / |v_x|; any other ray is marched by rows with the fractional
// column a0 + s a_step, a_step = -v_x / v_y, w = |v| / |v_y|.  Positions are
// 32.32 fixed point computed once per ray in FP64; the projector and the
// ray-driven and gather forms of the back-projector take bit-identical taps.
//
// A: one block = 32 adjacent rays of one view; 8 warps march disjoint parts
// of the step range and add their partial sums in a fixed order.  A ray
// marched by columns reads the staged transpose XC (line s = column s), one
// marched by rows the staged rows XR, as in joseph.cu; taps just outside the
// image read the zero guard cells.
//
// A^T, tiles pixel by pixel (bp_mode 1 where fan_gather_ok holds, as at a
// scanner's proportions): k_fan_backproject_gather below, whose weights come from
// the pixel's detector coordinate.
//
// A^T, ray-driven tiles (bp_mode 1 elsewhere, the default where a lane stride
// exists): one block = one 16 x 16 image tile, warp w takes views w, w + 8, ...
// The rays of a view that can put a tap in the tile are those whose bins lie between
// the bins of the corners of the tile grown by one pixel (the bin map is
// monotone along any segment in front of the source, so its extremes over
// the square are at the corners), widened by one bin each way.  A warp's 32
// lanes take rays S apart, S the plan's stride, and march them over the
// tile's 16 steps with the projector's own integer positions, adding
// (1 - f) s w at the left tap into one accumulator tile and f s w at the
// right tap into another -- rays marched by columns in one pass, rays
// marched by rows in another.  The two half-warps take the even and the odd
// bin offsets of a pass, each with its own pair of accumulator tiles, so a
// stride of 2 costs no second pass.  S is the smallest stride for which any two
// rays of a view marched the same way and S or more bins apart are at least
// one pixel apart on every march line through the image (checked at plan
// time from the integer positions), so no two lanes add to the same word of
// an accumulator in the same step.  The warps' tiles are summed in a fixed
// order.  Where no stride up to kFtMaxStride suffices (a source very close
// to the image with fine bins), the gather below is used.
//
// A^T, pixel-driven gather (bp_mode 0): one thread per pixel, views in order.  The rays
// of view k that can put a tap on pixel (X, Y) through column X are those
// crossing the segment (X, Y-1)-(X, Y+1); their bins lie between the
// projections of its end points through the source (bin(p) is monotone
// along a segment in front of the source), widened by one bin each way.
// Each candidate is then tested with the projector's own integer position,
// so the gather applies exactly the projector's taps.  Rays marched by rows
// are found through the segment (X-1, Y)-(X+1, Y) likewise.
//
// ||Phi~||_F^2 = sum over rays of ||V^-1 a_i||^2: plan-time, one ray at a
// time (its taps scattered into an image, V^-1 by the image filter of
// fft.cu, the sum of squares in FP64).
#include <algorithm>
#include <cmath>

#include <climits>

#include "internal.cuh"

namespace dgct {

constexpr int kFanSeg = 8;

// ------------------------------------------------------------ projector ----
template <typename T>
__global__ void __launch_bounds__(32 * kFanSeg)
k_fan_project(const T* __restrict__ XR, const T* __restrict__ XC, int ldp, int n, int nd,
              const FanRay* __restrict__ rays, float* __restrict__ sino) {
    __shared__ float red[kFanSeg][32];
    const int v = blockIdx.y;
    const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
    const int d = blockIdx.x * 32 + lane;
    float acc = 0.f, w = 0.f;
    FanRay R{};
    if (d < nd) R = rays[(size_t)v * nd + d];      // plan constants: before the wait
    pdl_wait();      // the staged image is the previous kernel's output
    if (d < nd) {
        w = R.w;
        const T* __restrict__ B = R.col ? XC : XR;
        int s0, s1;
        step_range(R.a0, R.a_step, n, s0, s1);
        const int len = (n + kFanSeg - 1) / kFanSeg;
        s0 = max(s0, seg * len);
        s1 = min(s1, seg * len + len - 1);
        if (s0 <= s1)
            acc = joseph_march<8>(B, R.P0 + (long long)s0 * R.PSTEP + ((long long)(s0 * ldp + kPad) << 32), R.PSTEP, ldp,
                               s1 - s0 + 1);
    }
    red[seg][lane] = acc;
    __syncthreads();
    if (seg == 0 && d < nd) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < kFanSeg; ++k) t += red[k][lane];
        sino[(size_t)v * nd + d] = t * w;
    }
}

// ------------------------------------------------------- back-projector ----
__device__ __forceinline__ float fan_bin(const FanView& V, float x, float y) {
    const float along = fmaf(x, V.ecx, fmaf(y, V.ecy, V.dso));   // > 0: in front of the source
    const float across = fmaf(x, V.eux, y * V.euy);
    return V.dsd * across / (along * V.du) + V.half;
}

__device__ __forceinline__ void fan_candidates(const FanView& V, float x1, float y1, float x2, float y2,
                                               int nd, int& lo, int& hi) {
    const float b1 = fan_bin(V, x1, y1), b2 = fan_bin(V, x2, y2);
    // both ends clamped to [-2, nd + 1] before the conversion to int
    const float bl = fminf(fmaxf(fminf(b1, b2), -2.f), (float)nd + 1.f);
    const float bh = fmaxf(fminf(fmaxf(b1, b2), (float)nd + 1.f), -2.f);
    lo = max(0, (int)floorf(bl) - 1);
    hi = min(nd - 1, (int)ceilf(bh) + 1);
}

__global__ void __launch_bounds__(256)
k_fan_backproject(const float* __restrict__ sino, const FanRay* __restrict__ rays,
                  const FanView* __restrict__ views, int n, int nv, int nd, float* __restrict__ img) {
    const int ix = blockIdx.x * 16 + (threadIdx.x & 15), iy = blockIdx.y * 16 + (threadIdx.x >> 4);
    if (ix >= n || iy >= n) return;
    const float c = 0.5f * (float)(n - 1);
    const float X = (float)ix - c, Y = c - (float)iy;
    float acc = 0.f;
    for (int k = 0; k < nv; ++k) {
        const FanView V = views[k];
        const FanRay* __restrict__ R = rays + (size_t)k * nd;
        const float* __restrict__ sk = sino + (size_t)k * nd;
        int lo, hi;
        // rays marched by columns that cross column X within one row of Y
        fan_candidates(V, X, Y - 1.f, X, Y + 1.f, nd, lo, hi);
        for (int d = lo; d <= hi; ++d) {
            const FanRay r = R[d];
            if (!r.col) continue;
            int i0;
            float f;
            joseph_tap(r.P0 + (long long)ix * r.PSTEP, i0, f);
            if (i0 == iy) acc = fmaf((1.f - f) * r.w, sk[d], acc);
            else if (i0 == iy - 1) acc = fmaf(f * r.w, sk[d], acc);
        }
        // rays marched by rows that cross row Y within one column of X
        fan_candidates(V, X - 1.f, Y, X + 1.f, Y, nd, lo, hi);
        for (int d = lo; d <= hi; ++d) {
            const FanRay r = R[d];
            if (r.col) continue;
            int i0;
            float f;
            joseph_tap(r.P0 + (long long)iy * r.PSTEP, i0, f);
            if (i0 == ix) acc = fmaf((1.f - f) * r.w, sk[d], acc);
            else if (i0 == ix - 1) acc = fmaf(f * r.w, sk[d], acc);
        }
    }
    img[(size_t)iy * n + ix] = acc;
}

constexpr int kFtS = 16, kFtLd = kFtS + 1, kFtWarps = 8, kFtMaxStride = 8;

// two accumulator pairs per warp: the two half-warps of a pass take rays of
// neighbouring bins, each half into its own pair
struct FtShared {
    float accL[kFtWarps][2][kFtS * kFtLd], accR[kFtWarps][2][kFtS * kFtLd];
};

// One pass of a warp over the tile: the lanes whose rays are marched by
// columns (COL = 1: step k = column tx0 + k, taps along rows) or by rows.
template <int COL>
__device__ __forceinline__ void fan_tile_pass(const FanRay& r, float sw, bool on, int tx0, int ty0, int ncol,
                                              int nrow, float* __restrict__ AL, float* __restrict__ AR) {
    constexpr int as = COL ? 1 : kFtLd, ac = COL ? kFtLd : 1;     // accumulator strides: step, tap
    if (!on) return;
    const int s0 = COL ? tx0 : ty0, c0 = COL ? ty0 : tx0;
    const int ns = COL ? ncol : nrow, nc = COL ? nrow : ncol;
    // position relative to the tile: the left tap's index in the tile is the high word
    long long pos = r.P0 + (long long)s0 * r.PSTEP - ((long long)c0 << 32);
    auto step = [&](int k) {
        const int rel = (int)(pos >> 32);
        const float f = __uint_as_float(0x3F800000u | ((unsigned)pos >> 9)) - 1.0f;
        const int at = k * as + rel * ac;
        if ((unsigned)rel < (unsigned)nc) AL[at] += (1.f - f) * sw;
        if ((unsigned)(rel + 1) < (unsigned)nc) AR[at + ac] += f * sw;
        pos += r.PSTEP;
    };
    if (ns == kFtS) {
#pragma unroll
        for (int k = 0; k < kFtS; ++k) step(k);
    } else {
        for (int k = 0; k < ns; ++k) step(k);
    }
}

__global__ void __launch_bounds__(kFtWarps * 32, 4)
k_fan_backproject_tile(const float* __restrict__ sino, const FanRay* __restrict__ rays,
                       const FanView* __restrict__ views, int n, int nv, int nd, int stride,
                       float* __restrict__ img) {
    __shared__ FtShared sh;
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
    const int tx0 = blockIdx.x * kFtS, ty0 = blockIdx.y * kFtS;
    const int ncol = min(kFtS, n - tx0), nrow = min(kFtS, n - ty0);
    const int half = lane >> 4, hl = lane & 15;
    float* AL = sh.accL[wp][half];
    float* AR = sh.accR[wp][half];
    for (int i = hl; i < kFtS * kFtLd; i += 16) AL[i] = AR[i] = 0.f;
    __syncwarp();
    // lane stride rounded up to even: pass p gives bin offset 2p + half to each
    // half-warp, whose 16 lanes then take rays `st` bins apart
    const int st = stride + (stride & 1);
    // the tile grown by one pixel each way, centred coordinates (x right, y up)
    const float c = 0.5f * (float)(n - 1);
    const float xa = (float)(tx0 - 1) - c, xb = (float)(tx0 + ncol) - c;
    const float ya = c - (float)(ty0 - 1), yb = c - (float)(ty0 + nrow);
    for (int v = wp; v < nv; v += kFtWarps) {
        const FanView V = views[v];
        const float b0 = fan_bin(V, xa, ya), b1 = fan_bin(V, xa, yb), b2 = fan_bin(V, xb, ya), b3 = fan_bin(V, xb, yb);
        const float bl = fminf(fmaxf(fminf(fminf(b0, b1), fminf(b2, b3)), -2.f), (float)nd + 1.f);
        const float bh = fmaxf(fminf(fmaxf(fmaxf(b0, b1), fmaxf(b2, b3)), (float)nd + 1.f), -2.f);
        const int lo = max(0, (int)floorf(bl) - 1), hi = min(nd - 1, (int)ceilf(bh) + 1);
        const FanRay* __restrict__ R = rays + (size_t)v * nd;
        const float* __restrict__ sk = sino + (size_t)v * nd;
        for (int base = lo; base <= hi; base += 16 * st) {
            for (int p = 0; 2 * p < st; ++p) {
                const int d = base + 2 * p + half + st * hl;
                const bool valid = d <= hi;
                FanRay r{};
                float sw = 0.f;
                if (valid) {
                    r = R[d];
                    sw = sk[d] * r.w;
                }
                const bool by_col = valid && r.col, by_row = valid && !r.col;
                if (__any_sync(0xffffffffu, by_col)) fan_tile_pass<1>(r, sw, by_col, tx0, ty0, ncol, nrow, AL, AR);
                __syncwarp();
                if (__any_sync(0xffffffffu, by_row)) fan_tile_pass<0>(r, sw, by_row, tx0, ty0, ncol, nrow, AL, AR);
                __syncwarp();
            }
        }
    }
    __syncthreads();
    for (int p = tid; p < kFtS * kFtS; p += blockDim.x) {
        const int ly = p / kFtS, lx = p % kFtS;
        if (lx >= ncol || ly >= nrow) continue;
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < kFtWarps; ++w)
#pragma unroll
            for (int h = 0; h < 2; ++h) t += sh.accL[w][h][ly * kFtLd + lx] + sh.accR[w][h][ly * kFtLd + lx];
        img[(size_t)(ty0 + ly) * n + tx0 + lx] = t;
    }
}

// Pixel form of the tiles (fan_gather_ok), as the parallel beam's (joseph.cu).
// At depth s = p . e_c + dso the rays of a view are du s / dsd apart along e_u,
// so with q the pixel's detector coordinate ray d lies |q - d| du s / dsd from it
// along e_u, and |q - d| A_d, A_d = s du / max(|v_x|, |v_y|), along the ray's
// own interpolated axis: its Joseph weight is max(0, 1 - |q - d| A_d) w_d.  Where
// no A_d falls below 1/2 inside the image, only rays floor(q) - 1 .. floor(q) + 2
// can reach a pixel: four shared-memory reads of (A_d / s, w_d v_d) and four
// weights, where marching the rays through accumulator tiles took 131 warp
// instructions per pixel and view (110 M at 512^2/102/736).
//
// q is a projective function of the pixel.  In a tile it is q0 + rel / (1 + sig)
// with rel and sig linear in the pixel; q0 + rel is 6.26 fixed point from
// FP64 constants, and only the correction -rel sig / (1 + sig), about one bin
// at most at a scanner's proportions, is FP32.  A^T + A with both filters at
// 512^2/102/736: 210 -> 144 us (with the tile corners in FP64 too: 150).
constexpr int kFgS = 16, kFgThreads = 128;
constexpr int kFgViews = 32;      // views staged at a time (16 KB)
constexpr int kFgSlots = 64;      // rays a view can need (checked by fan_gather_ok)
constexpr int kFgUnroll = 8, kFgBatch = 4;
constexpr int kFgFrac = 26;
constexpr double kFgMaxStep = 3.0;   // widest ray spacing in pixels (fan_gather_ok)

struct FgShared {
    float2 seg[kFgViews][kFgSlots];       // A_d / s, w_d v_d
    int4 fix[kFgViews];                   // position of pixel (8, 8), its steps along x and y; first staged ray
    float4 lin[kFgViews];                 // rel and sig per pixel along x and y
    float s0[kFgViews];                   // depth of pixel (8, 8)
};

__device__ __forceinline__ void fg_view_setup(const FanView* __restrict__ views, int v0, int cnt, int n, int tx0, int ty0,
                                              FgShared& sh) {
    for (int i = threadIdx.x; i < kFgViews; i += kFgThreads) {
        if (i >= cnt) {                   // pads the last kFgUnroll views: no rays, all values 0
            sh.fix[i] = make_int4(1 << kFgFrac, 0, 0, INT_MIN / 2);
            sh.lin[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            sh.s0[i] = 0.f;
            continue;
        }
        const FanView& V = views[v0 + i];
        const double c = 0.5 * (n - 1), X = tx0 + kFgS / 2 - c, Y = c - (ty0 + kFgS / 2);
        const double t0 = X * V.deux + Y * V.deuy, s0 = X * V.decx + Y * V.decy + V.ddso;
        const double is0 = 1.0 / s0, k = V.dscale * is0 * is0;
        const double kx = k * (V.deux * s0 - t0 * V.decx), ky = -k * (V.deuy * s0 - t0 * V.decy);
        const double gx = V.decx * is0, gy = -V.decy * is0;
        const double q0 = V.dhalf + V.dscale * t0 * is0;
        // lowest q - q0 over the tile's pixels of the image (grown by one; sig > -1 in front of the
        // source), in FP32: only the first staged ray depends on it, and it leaves a margin
        const float fkx = (float)kx, fky = (float)ky, fgx = (float)gx, fgy = (float)gy;
        const float xe = (float)min(kFgS / 2, n - tx0 - kFgS / 2), ye = (float)min(kFgS / 2, n - ty0 - kFgS / 2);
        float ql = -8.f * (fabsf(fkx) + fabsf(fky));      // the linear part may fall below q itself
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            const float x = (h & 1) ? xe : -8.f, y = (h & 2) ? ye : -8.f;
            ql = fminf(ql, (fkx * x + fky * y) / (1.f + fgx * x + fgy * y));
        }
        const double lo = floor(q0 + ql) - 2.0;           // room for ray floor(q) - 1
        const double unit = (double)(1 << kFgFrac);
        sh.fix[i] = make_int4((int)(unsigned)((q0 - lo) * unit + 0.5), (int)rint(kx * unit), (int)rint(ky * unit), (int)lo);
        sh.lin[i] = make_float4(fkx, fky, fgx, fgy);
        sh.s0[i] = (float)s0;
    }
}

// Staged rays of the views; true if a value is not finite.
__device__ __forceinline__ bool fg_stage(const float* __restrict__ sino, const float2* __restrict__ gw, int v0, int cnt,
                                         int nd, FgShared& sh) {
    const int pad = (cnt + kFgUnroll - 1) / kFgUnroll * kFgUnroll;
    const int tot = pad * kFgSlots;
    bool bad = false;
    for (int j0 = threadIdx.x; j0 < tot; j0 += kFgThreads * kFgBatch) {
        float2 g[kFgBatch];
        float v[kFgBatch];
#pragma unroll
        for (int b = 0; b < kFgBatch; ++b) {
            const int j = min(j0 + b * kFgThreads, tot - 1), i = j / kFgSlots;
            const int d = sh.fix[i].w + (j & (kFgSlots - 1));
            g[b] = make_float2(0.f, 0.f);
            v[b] = 0.f;
            if ((unsigned)d < (unsigned)nd) {
                const size_t o = (size_t)(v0 + i) * nd + d;
                g[b] = gw[o];
                v[b] = sino[o] * g[b].y;
            }
        }
#pragma unroll
        for (int b = 0; b < kFgBatch; ++b) {
            const int j = j0 + b * kFgThreads;
            if (j >= tot) break;
            bad |= !(fabsf(v[b]) <= 3.402823466e38f);
            sh.seg[j / kFgSlots][j & (kFgSlots - 1)] = make_float2(g[b].x, v[b]);
        }
    }
    return bad;
}

template <bool SAFE>
__device__ __forceinline__ void fg_pixel(const float2* __restrict__ seg, unsigned q, float rel, float sig, float s0,
                                         float& acc) {
    const float corr = -__fdividef(rel * sig, 1.f + sig);
    const float f = __uint2float_rn(q & ((1u << kFgFrac) - 1u));
    const float g = fmaf(f, 1.f / (float)(1 << kFgFrac), corr), r = (g - 0.5f) + 12582912.f;     // floor(g), up to a tie
    const int base = min(max((int)(q >> kFgFrac) + (__float_as_int(r) - 0x4B400000), 1), kFgSlots - 3);
    const float u = g - (r - 12582912.f), s = fmaf(s0, sig, s0);
#pragma unroll
    for (int j = -1; j < 3; ++j) {
        const float2 t = seg[base + j];
        const float w = __saturatef(fmaf(-fabsf(u - (float)j), s * t.x, 1.f));
        if (!SAFE || w > 0.f) acc = fmaf(w, t.y, acc);
    }
}

template <bool SAFE>
__device__ __forceinline__ void fg_views(const FgShared& sh, int cnt, int lx, int ly, float& acc0, float& acc1) {
    const float fx = (float)lx, fy = (float)ly;
    float g0 = 0.f, g1 = 0.f;      // a chunk's views apart from the pixel's sum: shorter chains of additions
    for (int i0 = 0; i0 < cnt; i0 += kFgUnroll) {
        float t0 = 0.f, t1 = 0.f;
#pragma unroll
        for (int k = 0; k < kFgUnroll; ++k) {
            const int i = i0 + k;
            const int4 c = sh.fix[i];
            const float4 l = sh.lin[i];
            const float s0 = sh.s0[i];
            const unsigned q = (unsigned)c.x + (unsigned)(lx * c.y) + (unsigned)(ly * c.z);
            const float rel = fmaf(l.x, fx, l.y * fy), sig = fmaf(l.z, fx, l.w * fy);
            fg_pixel<SAFE>(sh.seg[i], q, rel, sig, s0, t0);
            fg_pixel<SAFE>(sh.seg[i], q + 8u * (unsigned)c.z, fmaf(8.f, l.y, rel), fmaf(8.f, l.w, sig), s0, t1);
        }
        g0 += t0;
        g1 += t1;
    }
    acc0 += g0;
    acc1 += g1;
}

__global__ void __launch_bounds__(kFgThreads, 8)
k_fan_backproject_gather(const float* __restrict__ sino, const float2* __restrict__ gw,
                         const FanView* __restrict__ views, int n, int nv, int nd, float* __restrict__ img) {
    __shared__ FgShared sh;
    const int tid = threadIdx.x;
    const int tx0 = blockIdx.x * kFgS, ty0 = blockIdx.y * kFgS;
    const int lx = (tid & 15) - kFgS / 2, ly = (tid >> 4) - kFgS / 2;      // relative to pixel (8, 8)
    float acc0 = 0.f, acc1 = 0.f;
    for (int v0 = 0; v0 < nv; v0 += kFgViews) {
        const int cnt = min(kFgViews, nv - v0);
        if (v0 > 0) __syncthreads();                                       // the previous views are done with
        fg_view_setup(views, v0, cnt, n, tx0, ty0, sh);
        if (v0 == 0) pdl_wait();      // the views are plan constants, the sinogram is not
        __syncthreads();
        const bool bad = fg_stage(sino, gw, v0, cnt, nd, sh);
        if (__syncthreads_or(bad))
            fg_views<true>(sh, cnt, lx, ly, acc0, acc1);
        else
            fg_views<false>(sh, cnt, lx, ly, acc0, acc1);
    }
    const int ix = tx0 + (tid & 15), iy = ty0 + (tid >> 4);
    if (ix < n && iy < n) img[(size_t)iy * n + ix] = acc0;
    if (ix < n && iy + 8 < n) img[(size_t)(iy + 8) * n + ix] = acc1;
}

// Whether the pixel form applies: inside the image's circumscribed circle rays
// are between 1/2 and kFgMaxStep pixels apart along any ray's axis, and a tile's
// rays fit the staged slots.  A position's rounding, a fixed share of a bin, grows
// with the spacing in pixels: against 64 bits A^T s was off by 0.85 times as much
// as from the ray-driven tiles at spacings up to 2.7, 0.91 at 3.2, but 1.04-1.2 at
// 4.2, 2 at 8.5 and 17 at 68 (2.4e-6), so wider rays keep those.  q's gradient is
// (dsd / du) sqrt(s^2 + t^2) / s^2 (t = p . e_u); its largest value is taken over the
// circle grown to hold the centre pixel of a tile that the image's edge cuts.
static bool fan_gather_ok(int n, double dso, double ddo, double du, int nd) {
    const double dsd = dso + ddo, u = 0.5 * (nd - 1) * du, R = n / std::sqrt(2.0) + 1.0, Rc = R + 12.0;
    if (!(dso - Rc >= 1.0) || !(du * (dso - R) / std::hypot(dsd, u) >= 0.5)) return false;
    // max(|v_x|, |v_y|) >= |v| / sqrt 2 >= dsd / sqrt 2
    if (!(du * (dso + R) * std::sqrt(2.0) / dsd <= kFgMaxStep)) return false;
    double grad = 0.0;
    for (int k = 0; k <= 1024; ++k) {
        const double a = 3.14159265358979 * k / 1024, s = dso - Rc * std::cos(a), t = Rc * std::sin(a);
        grad = std::max(grad, dsd / du * std::hypot(s, t) / (s * s));
    }
    return 16.0 * std::sqrt(2.0) * 1.02 * grad + 8.0 <= kFgSlots;
}

// ------------------------------------------------------- ||Phi~||_F^2 ----
// Ray ray0 + b's taps scattered into zeroed image b of a batch ([nimg][n][n],
// one block per image; a ray puts at most one tap on a pixel, so the writes
// do not collide).  Rays past the last (nrays) leave their image zero.
__global__ void __launch_bounds__(1024)
k_fan_ray_image(const FanRay* __restrict__ rays, long long ray0, long long nrays, int n, float* __restrict__ img) {
    const size_t N = (size_t)n * n;
    img += (size_t)blockIdx.x * N;
    for (size_t i = threadIdx.x; i < N; i += blockDim.x) img[i] = 0.f;
    __syncthreads();
    const long long ray = ray0 + blockIdx.x;
    if (ray >= nrays) return;
    const FanRay R = rays[ray];
    for (int s = threadIdx.x; s < n; s += blockDim.x) {
        int i0;
        float f;
        joseph_tap(R.P0 + (long long)s * R.PSTEP, i0, f);
        const float t[2] = {(1.f - f) * R.w, f * R.w};
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int q = i0 + j;
            if (q < 0 || q >= n) continue;
            const size_t o = R.col ? (size_t)q * n + s : (size_t)s * n + q;
            img[o] = t[j];
        }
    }
}

// out[slot0 + b] = sum of squares of image b (FP64, one block per image,
// fixed order), for the images of rays before nrays.
__global__ void __launch_bounds__(1024)
k_sum_squares(const float* __restrict__ img, long long N, double* __restrict__ out, long long slot0,
              long long nrays) {
    __shared__ double red[32];
    if (slot0 + blockIdx.x >= nrays) return;
    img += (size_t)blockIdx.x * N;
    double acc = 0.0;
    for (long long i = threadIdx.x; i < N; i += blockDim.x) {
        const double v = img[i];
        acc += v * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) out[slot0 + blockIdx.x] = t;
    }
}

// ----------------------------------------------------------------- host ----
static void fan_constants(int n, int nd, const std::vector<double>& ang, double dso, double ddo, double du,
                          std::vector<FanRay>& rays, std::vector<FanView>& views, std::vector<float2>* gw = nullptr) {
    const double c = 0.5 * (n - 1), half = 0.5 * (nd - 1), q = 4294967296.0;
    rays.resize(ang.size() * (size_t)nd);
    views.resize(ang.size());
    if (gw) gw->resize(rays.size());
    for (size_t k = 0; k < ang.size(); ++k) {
        const double st = std::sin(ang[k]), ct = std::cos(ang[k]);
        const double sx = dso * st, sy = -dso * ct;
        views[k] = FanView{(float)ct, (float)st, (float)-st, (float)ct, (float)dso, (float)(dso + ddo),
                           (float)du, (float)half, ct, st, -st, ct, dso, (dso + ddo) / du, half};
        for (int d = 0; d < nd; ++d) {
            const double u = (d - half) * du;
            const double vx = -ddo * st + u * ct - sx, vy = ddo * ct + u * st - sy;
            const double L = std::hypot(vx, vy);
            FanRay R{};
            double a0, as, w;
            if (std::fabs(vx) >= std::fabs(vy)) {       // by columns: row c - (S_y + (X - S_x) v_y / v_x)
                const double t = vy / vx;
                a0 = c - sy + (sx + c) * t;
                as = -t;
                w = L / std::fabs(vx);
                R.col = 1;
            } else {                                     // by rows: column S_x + (Y - S_y) v_x / v_y + c
                const double t = vx / vy;
                a0 = sx + c + (c - sy) * t;
                as = -t;
                w = L / std::fabs(vy);
                R.col = 0;
            }
            R.P0 = std::llround(a0 * q);
            R.PSTEP = std::llround(as * q);
            R.a0 = (float)a0;
            R.a_step = (float)as;
            R.w = (float)w;
            rays[k * (size_t)nd + d] = R;
            if (gw) (*gw)[k * (size_t)nd + d] = make_float2((float)(du / std::max(std::fabs(vx), std::fabs(vy))), R.w);
        }
    }
}

int launch_fan_project(const dgamp_ct_plan_s* pl, float* sino, cudaStream_t st) {
    const dim3 grd((unsigned)((pl->nd + 31) / 32), (unsigned)pl->nv);
    DGCT_CUDA(launch_pdl(k_fan_project<float>, grd, dim3(32 * kFanSeg), 0, st, pl->ws.XR, pl->ws.XC, pl->ldp, pl->n,
                         pl->nd, pl->ws.fan_rays, sino));
    return DGAMP_CT_OK;
}

int launch_fan_backproject(const dgamp_ct_plan_s* pl, const float* sino, float* img, cudaStream_t st) {
    const dim3 grd((unsigned)((pl->n + 15) / 16), (unsigned)((pl->n + 15) / 16));
    if (pl->bp_mode == 1 && pl->fan_stride > 0 && pl->ws.fan_gw)
        DGCT_CUDA(launch_pdl(k_fan_backproject_gather, grd, dim3(kFgThreads), 0, st, sino, pl->ws.fan_gw,
                             pl->ws.fan_views, pl->n, pl->nv, pl->nd, img));
    else if (pl->bp_mode == 1 && pl->fan_stride > 0)
        k_fan_backproject_tile<<<grd, kFtWarps * 32, 0, st>>>(sino, pl->ws.fan_rays, pl->ws.fan_views, pl->n, pl->nv,
                                                              pl->nd, pl->fan_stride, img);
    else
        k_fan_backproject<<<grd, 256, 0, st>>>(sino, pl->ws.fan_rays, pl->ws.fan_views, pl->n, pl->nv, pl->nd, img);
    DGCT_LAUNCH_CHECK();
    return DGAMP_CT_OK;
}

// Smallest lane stride S of the tile back-projection: for every view and
// every bin d, the next ray d + kS (k >= 1) marched the same way is at least
// one pixel away from ray d at both ends of the march (s = 0 and s = n - 1,
// the same side at both, so everywhere between: the gap is linear in s).
// Positions along a march line are monotone in the bin, so rays further
// apart are further apart still.  0 when no S <= kFtMaxStride works.
static int fan_tile_stride(const std::vector<FanRay>& rays, int nv, int nd, int n) {
    const double one = 4294967296.0;
    for (int S = 1; S <= kFtMaxStride; ++S) {
        bool ok = true;
        for (int v = 0; v < nv && ok; ++v) {
            const FanRay* R = rays.data() + (size_t)v * nd;
            for (int d = 0; d < nd && ok; ++d) {
                int e = d + S;
                while (e < nd && R[e].col != R[d].col) e += S;
                if (e >= nd) continue;
                const double g0 = (double)(R[e].P0 - R[d].P0);
                const double g1 = g0 + (double)(n - 1) * (double)(R[e].PSTEP - R[d].PSTEP);
                if (!(g0 * g1 > 0.0) || std::fabs(g0) < one || std::fabs(g1) < one) ok = false;
            }
        }
        if (ok) return S;
    }
    return 0;
}

int fan_setup(dgamp_ct_plan_s* pl, const std::vector<double>& ang, double src_dist, double det_dist,
              double det_spacing) {
    std::vector<FanRay> rays;
    std::vector<FanView> views;
    std::vector<float2> gw;
    const bool gather = fan_gather_ok(pl->n, src_dist, det_dist, det_spacing, pl->nd);
    fan_constants(pl->n, pl->nd, ang, src_dist, det_dist, det_spacing, rays, views, gather ? &gw : nullptr);
    if (cudaMalloc((void**)&pl->ws.fan_rays, rays.size() * sizeof(FanRay)) != cudaSuccess ||
        cudaMalloc((void**)&pl->ws.fan_views, views.size() * sizeof(FanView)) != cudaSuccess ||
        (gather && cudaMalloc((void**)&pl->ws.fan_gw, gw.size() * sizeof(float2)) != cudaSuccess)) {
        cudaGetLastError();
        return DGAMP_CT_ERR_OOM;
    }
    DGCT_CUDA(cudaMemcpy(pl->ws.fan_rays, rays.data(), rays.size() * sizeof(FanRay), cudaMemcpyHostToDevice));
    DGCT_CUDA(cudaMemcpy(pl->ws.fan_views, views.data(), views.size() * sizeof(FanView), cudaMemcpyHostToDevice));
    if (gather)
        DGCT_CUDA(cudaMemcpy(pl->ws.fan_gw, gw.data(), gw.size() * sizeof(float2), cudaMemcpyHostToDevice));
    pl->fan = 1;
    pl->fan_stride = fan_tile_stride(rays, pl->nv, pl->nd, pl->n);
    pl->bp_mode = pl->fan_stride > 0 ? 1 : 0;
    // ||Phi~||_F^2: batches of B rays -- their tap images, V^-1 of them (the
    // image filter, batched), one FP64 sum of squares per ray into `sums` --
    // added on the host in ray order.  Each ray's arithmetic is that of the
    // single-image filter.  B keeps the scratch near 512 MB.
    const int64_t M = pl->M, N = pl->N;
    const size_t per_img = (size_t)N * 2 * sizeof(float) + (size_t)pl->n * pl->m2 * sizeof(float2);
    const int B = (int)std::max<size_t>(1, std::min<size_t>(64, ((size_t)512 << 20) / per_img));
    double* sums = nullptr;
    float* imgs = nullptr;
    float2* C = nullptr;
    if (cudaMalloc((void**)&sums, (size_t)M * sizeof(double)) != cudaSuccess ||
        cudaMalloc((void**)&imgs, (size_t)B * N * 2 * sizeof(float)) != cudaSuccess ||
        cudaMalloc((void**)&C, (size_t)B * pl->n * pl->m2 * sizeof(float2)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(sums);
        cudaFree(imgs);
        cudaFree(C);
        return DGAMP_CT_ERR_OOM;
    }
    int rc = DGAMP_CT_OK;
    for (int64_t i = 0; i < M && rc == DGAMP_CT_OK; i += B) {
        k_fan_ray_image<<<B, 1024>>>(pl->ws.fan_rays, i, M, pl->n, imgs);
        rc = launch_precond_images(pl, imgs, imgs + (size_t)B * N, C, B, 1, 0);
        if (rc == DGAMP_CT_OK) k_sum_squares<<<B, 1024>>>(imgs + (size_t)B * N, N, sums, i, M);
        const cudaError_t e = cudaGetLastError();
        if (rc == DGAMP_CT_OK && e != cudaSuccess) rc = cuda_fail(e);
    }
    cudaFree(imgs);
    cudaFree(C);
    std::vector<double> h((size_t)M);
    if (rc == DGAMP_CT_OK) {
        const cudaError_t e = cudaMemcpy(h.data(), sums, (size_t)M * sizeof(double), cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) rc = cuda_fail(e);
    }
    cudaFree(sums);
    if (rc != DGAMP_CT_OK) return rc;
    double tot = 0.0;
    for (double v : h) tot += v;
    pl->frob2 = tot;
    DGCT_CUDA(cudaMemcpy(&pl->ws.S->frob2, &tot, sizeof(double), cudaMemcpyHostToDevice));
    return DGAMP_CT_OK;
}

}  // namespace dgct

using namespace dgct;

extern "C" int dgamp_ct_fan_ray_constants(const dgamp_ct_fan_geometry* g, int64_t* p0, int64_t* pstep, float* w,
                                          int32_t* col) {
    if (!g || !p0 || !pstep || !w || !col) return DGAMP_CT_ERR_INVALID_ARG;
    const dgamp_ct_geometry& b = g->base;
    if (b.n < 2 || b.n_views < 1 || b.n_det < 2 || !(g->det_spacing > 0) || !std::isfinite(g->src_dist) ||
        !std::isfinite(g->det_dist))
        return DGAMP_CT_ERR_INVALID_ARG;
    std::vector<double> ang(b.n_views);
    for (int k = 0; k < b.n_views; ++k)
        ang[k] = b.angles ? b.angles[k] : (double)k * (2.0 * 3.14159265358979323846 / b.n_views);
    std::vector<FanRay> rays;
    std::vector<FanView> views;
    fan_constants(b.n, b.n_det, ang, g->src_dist, g->det_dist, g->det_spacing, rays, views);
    for (size_t i = 0; i < rays.size(); ++i) {
        p0[i] = rays[i].P0;
        pstep[i] = rays[i].PSTEP;
        w[i] = rays[i].w;
        col[i] = rays[i].col;
    }
    return DGAMP_CT_OK;
}
