// gs_loss.cu -- loss terms of the mapping / refinement objectives and the Adam step.
//
// L1 (Eq. 4's photometric and depth terms): one pass per pixel producing the loss and its
// gradient.  SSIM (Eq. 23's structural term): two tiled passes with an 11-tap separable Gaussian
// (sigma 1.5, zero padding) in shared memory:
//   pass 1 blurs x, y, x^2, y^2, xy, sums the SSIM map and |x - y|, and writes the per-pixel derivatives of the SSIM map with
//          respect to mu_x, E[x^2] and E[xy];
//   pass 2 blurs those three maps (the adjoint of a zero-padded symmetric blur is the same blur)
//          and combines dSSIM/dx = blur(dS/dmu_x) + 2 x blur(dS/dE[x^2]) + y blur(dS/dE[xy]),
//          fused with the L1 gradient.
// Adam: one pass over the 14 scalars of every Gaussian, bias-corrected, opacity through its logit.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "gs_kernels.cuh"

namespace gs {

__device__ __forceinline__ float sgnf(float d) { return d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f); }

__device__ __forceinline__ void block_add_double(double v, double *out) {
    __shared__ double s_part[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double w = lane < (int)(blockDim.x >> 5) ? s_part[lane] : 0.0;
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if (lane == 0 && w != 0.0) atomicAdd(out, w);
    }
}

// grid (blocks, V): view v = blockIdx.y; pixels of the view strided over the x-blocks, four at a
// time (16-byte loads and stores) when the plane size and the pointers allow it.
template <bool kVec>
__global__ void k_l1(long long HWn, const float *rgb, const float *rgb_t, const float *depth, const float *depth_t,
                     float sc_rgb, float sc_d, float *d_rgb, float *d_depth, double *loss) {
    float acc_rgb = 0.f, acc_d = 0.f;      // per-thread sums of |d| (a few dozen terms each)
    const long long v = blockIdx.y;
    const long long stride = (long long)gridDim.x * blockDim.x;
    if (kVec) {
        const long long n4 = HWn >> 2;
        for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += stride) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const long long off = (3 * v + c) * n4 + q;
                const float4 x = reinterpret_cast<const float4 *>(rgb)[off];
                const float4 y = reinterpret_cast<const float4 *>(rgb_t)[off];
                const float4 d = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
                acc_rgb += (fabsf(d.x) + fabsf(d.y)) + (fabsf(d.z) + fabsf(d.w));
                reinterpret_cast<float4 *>(d_rgb)[off] =
                    make_float4(sgnf(d.x) * sc_rgb, sgnf(d.y) * sc_rgb, sgnf(d.z) * sc_rgb, sgnf(d.w) * sc_rgb);
            }
            if (depth) {
                const long long off = v * n4 + q;
                const float4 x = reinterpret_cast<const float4 *>(depth)[off];
                const float4 y = reinterpret_cast<const float4 *>(depth_t)[off];
                const float4 d = make_float4(x.x - y.x, x.y - y.y, x.z - y.z, x.w - y.w);
                acc_d += (fabsf(d.x) + fabsf(d.y)) + (fabsf(d.z) + fabsf(d.w));
                reinterpret_cast<float4 *>(d_depth)[off] =
                    make_float4(sgnf(d.x) * sc_d, sgnf(d.y) * sc_d, sgnf(d.z) * sc_d, sgnf(d.w) * sc_d);
            }
        }
    } else {
        for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < HWn; p += stride) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const long long idx = (3 * v + c) * HWn + p;
                const float d = rgb[idx] - rgb_t[idx];
                acc_rgb += fabsf(d);
                d_rgb[idx] = sgnf(d) * sc_rgb;
            }
            if (depth) {
                const long long idx = v * HWn + p;
                const float d = depth[idx] - depth_t[idx];
                acc_d += fabsf(d);
                d_depth[idx] = sgnf(d) * sc_d;
            }
        }
    }
    block_add_double((double)acc_rgb * sc_rgb + (double)acc_d * sc_d, loss);
}

static bool aligned16(const void *p) { return p == nullptr || ((uintptr_t)p & 15u) == 0; }

int launch_loss_l1(int V, int W, int H, const float *rgb, const float *rgb_t, const float *depth,
                   const float *depth_t, float w_rgb, float w_depth, float *d_rgb, float *d_depth, double *loss,
                   cudaStream_t s) {
    const long long HWn = (long long)W * H;
    const float sc_rgb = (float)((double)w_rgb / (3.0 * V * HWn));
    const float sc_d = (float)((double)w_depth / ((double)V * HWn));
    const bool use_d = depth && depth_t && d_depth && w_depth != 0.f;
    const bool vec = (HWn % 4 == 0) && aligned16(rgb) && aligned16(rgb_t) && aligned16(d_rgb) &&
                     (!use_d || (aligned16(depth) && aligned16(depth_t) && aligned16(d_depth)));
    const long long units = vec ? HWn / 4 : HWn;
    // about four resident blocks of 256 threads per SM in total, spread over the views
    const long long want = std::max<long long>(1, ((long long)device_sm_count() * 4 + V - 1) / V);
    const int gx = (int)std::max<long long>(1, std::min<long long>((units + 255) / 256, want));
    if (cudaMemsetAsync(loss, 0, sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    const dim3 grid(gx, V);
    if (vec)
        k_l1<true><<<grid, 256, 0, s>>>(HWn, rgb, rgb_t, use_d ? depth : nullptr, depth_t, sc_rgb, sc_d, d_rgb,
                                        use_d ? d_depth : nullptr, loss);
    else
        k_l1<false><<<grid, 256, 0, s>>>(HWn, rgb, rgb_t, use_d ? depth : nullptr, depth_t, sc_rgb, sc_d, d_rgb,
                                         use_d ? d_depth : nullptr, loss);
    count_launches(1);
    return check_launch();
}

// ------------------------------------------------------------------------------------------
// SSIM
// ------------------------------------------------------------------------------------------
constexpr int kSB = 32;            // output tile
constexpr int kR = 5;              // window radius
constexpr int kSI = kSB + 2 * kR;  // input tile with halo
constexpr float kC1 = 0.0001f, kC2 = 0.0009f;

struct SsimTaps {
    float w[11];
};

static SsimTaps make_taps() {
    SsimTaps t;
    double g[11], sum = 0.0;
    for (int k = 0; k < 11; ++k) {
        const double d = k - 5;
        g[k] = exp(-d * d / (2.0 * 1.5 * 1.5));
        sum += g[k];
    }
    for (int k = 0; k < 11; ++k) t.w[k] = (float)(g[k] / sum);
    return t;
}

// Both passes: 256 threads walk a strip of 32 columns down `seg` rows, 32 rows a step.  The inputs of a step are
// fetched 16 bytes at a time where the planes allow it: 48 columns, from 8 left of the strip, so that every group
// of four is in or out as a whole.  The horizontal filter gives a thread four adjacent columns of one row, so it
// loads 16 inputs for four outputs; the vertical filter four rows of one column.  The last ten filtered rows of a
// step are the first of the next, and the sums are reduced once per strip.  Values that take the same taps are
// the two components of packed FP32x2 arithmetic: pass 1 filters (x, y) and (x^2, y^2) packed and x y alone, pass
// 2 (dS/dmu_x, dS/dE[x^2]) packed and dS/dE[xy] alone.  (The SSIM map's mean enters an FP64 loss and its bias
// comes from the rounding of these sums, so their operations are part of the result: taps in ascending order,
// w x rounded before it is added or meets its second factor; used twice, it is not joined with the sum.)  The pitches below and the order of the lanes in
// the horizontal filter (hlane) keep every 16-byte shared access of eight lanes on 32 different banks.
// 8 views of 1200 x 680 (19.6 M samples): pass 1 187 us (68 % of the issue slots; 392 MB take 58 us), pass 2 142 us
// (62 %; 470 MB, 69 us); tiles of 32 x 32 on their own 213 and 173 us; with one sample per load and scalar
// arithmetic 318 and 279 us, plus 47 us for a pass of its own for |x - y|.
constexpr int kSVR = 4;            // rows per thread in the vertical filter, columns in the horizontal one
constexpr int kSC = 48;            // input columns, the strip's own from kSL
constexpr int kSL = 8;
constexpr int kHalo = 2 * kR;      // filtered rows that two steps share

struct __align__(16) Ssim1Smem {
    float2 xy[kSB][kSC + 2];
    float4 h[kSI][kSB + 4];        // filtered x, y, x^2, y^2 of column c at c ^ (c >> 2)
    float hxy[kSI][kSB + 8];       // filtered x y, likewise
};
struct __align__(16) Ssim2Smem {
    float2 a[kSB][kSC + 2];        // dS/dmu_x, dS/dE[x^2]
    float b[kSB][kSC];             // dS/dE[xy]
    float2 ha[kSI][kSB + 2];
    float hb[kSI][kSB + 16];
};

// item i of the horizontal filter: four lanes along a row, the next four on the row below it
__device__ __forceinline__ int hlane_row(int i) { return (i >> 5) * 4 + ((i >> 2) & 1) + ((i >> 3) & 2); }
__device__ __forceinline__ int hlane_group(int i) { return (i & 3) + ((i >> 1) & 4); }

// p[0..3] of a row whose columns gx..gx+3 may lie outside [0, W) (all or none of them with VEC)
template <bool VEC>
__device__ __forceinline__ float4 load4(const float *row, int gx, int W) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) {
        if (gx >= 0 && gx < W) v = *reinterpret_cast<const float4 *>(row + gx);
    } else {
        if (gx >= 0 && gx < W) v.x = row[gx];
        if (gx + 1 >= 0 && gx + 1 < W) v.y = row[gx + 1];
        if (gx + 2 >= 0 && gx + 2 < W) v.z = row[gx + 2];
        if (gx + 3 >= 0 && gx + 3 < W) v.w = row[gx + 3];
    }
    return v;
}

// (a, b) summed over the CTA (256 threads) and added to *pa, *pb: as float pairs within a warp, in FP64
// across warps
__device__ __forceinline__ void block_add2(float2 a, float2 b, double *pa, double *pb) {
    __shared__ double2 s_part[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float ax = __shfl_xor_sync(0xffffffffu, a.x, o), ay = __shfl_xor_sync(0xffffffffu, a.y, o);
        const float bx = __shfl_xor_sync(0xffffffffu, b.x, o), by = __shfl_xor_sync(0xffffffffu, b.y, o);
        a.y = fp::add(a.y, ay);
        b.y = fp::add(b.y, by);
        add_to_pair(a, ax);
        add_to_pair(b, bx);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) s_part[warp] = make_double2(pair_value(a), pair_value(b));
    __syncthreads();
    if (threadIdx.x < 2) {
        double v = 0.0;
        for (int w = 0; w < 8; ++w) v += threadIdx.x ? s_part[w].y : s_part[w].x;
        if (v != 0.0) atomicAdd(threadIdx.x ? pb : pa, v);
    }
}

// One row's four columns t of the horizontal filters, from row r of the inputs into row d of the filtered rows
__device__ __forceinline__ void ssim1_hfilter(Ssim1Smem &sm, const SsimTaps &tp, int r, int t, int d) {
    float2 m[kSVR], q[kSVR];
    float p[kSVR];
#pragma unroll
    for (int j = 0; j < kSVR; ++j) {
        m[j] = q[j] = make_float2(0.f, 0.f);
        p[j] = 0.f;
    }
    // output column 4 t + j takes inputs 4 t + j + kSL - kR + (0 .. 2 kR)
    const float4 *src = reinterpret_cast<const float4 *>(&sm.xy[r][4 * t]);
    constexpr int kFirst = kSL - kR;
#pragma unroll
    for (int u = kFirst / 2; u <= (kFirst + kSVR - 1 + 2 * kR) / 2; ++u) {
        const float4 f = src[u];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int k = 2 * u + e - kFirst;
            const float2 v = e ? make_float2(f.z, f.w) : make_float2(f.x, f.y);
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (k - j >= 0 && k - j <= 2 * kR) {
                    const float2 wv = fp2::mul(fp2::splat(tp.w[k - j]), v);
                    m[j] = fp2::add(wv, m[j]);
                    q[j] = fp2::fma(wv, v, q[j]);
                    p[j] = fmaf(wv.x, v.y, p[j]);
                }
            }
        }
    }
#pragma unroll
    for (int j = 0; j < kSVR; ++j) {
        const int c = (4 * t + j) ^ t;
        sm.h[d][c] = make_float4(m[j].x, m[j].y, q[j].x, q[j].y);
        sm.hxy[d][c] = p[j];
    }
}

__device__ __forceinline__ void ssim2_hfilter(Ssim2Smem &sm, const SsimTaps &tp, int r, int t, int d) {
    float2 a[kSVR];
    float b[kSVR];
#pragma unroll
    for (int j = 0; j < kSVR; ++j) {
        a[j] = make_float2(0.f, 0.f);
        b[j] = 0.f;
    }
    const float4 *sa = reinterpret_cast<const float4 *>(&sm.a[r][4 * t]);
    const float4 *sb = reinterpret_cast<const float4 *>(&sm.b[r][4 * t]);
    constexpr int kFirst = kSL - kR;
#pragma unroll
    for (int u = 0; u <= (kFirst + kSVR - 1 + 2 * kR) / 4; ++u) {
        const float4 f0 = sa[2 * u], f1 = sa[2 * u + 1], fb = sb[u];
        const float2 va[4] = {make_float2(f0.x, f0.y), make_float2(f0.z, f0.w), make_float2(f1.x, f1.y),
                              make_float2(f1.z, f1.w)};
        const float vb[4] = {fb.x, fb.y, fb.z, fb.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = 4 * u + e - kFirst;
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (k - j >= 0 && k - j <= 2 * kR) {
                    a[j] = fp2::fma(fp2::splat(tp.w[k - j]), va[e], a[j]);
                    b[j] = fmaf(tp.w[k - j], vb[e], b[j]);
                }
            }
        }
    }
    float4 *da = reinterpret_cast<float4 *>(&sm.ha[d][4 * t]);
    da[0] = make_float4(a[0].x, a[0].y, a[1].x, a[1].y);
    da[1] = make_float4(a[2].x, a[2].y, a[3].x, a[3].y);
    *reinterpret_cast<float4 *>(&sm.hb[d][4 * t]) = make_float4(b[0], b[1], b[2], b[3]);
}

// Pass 1 of a strip of one plane, rows [y_begin, y_end): x, y (x optionally as fl(fl(ea x) + eb)), zero padding;
// the blurred moments, the SSIM map and |x - y| summed over the thread's share, and the three per-pixel
// derivatives dS/dmu_x, dS/dE[x^2], dS/dE[xy] (scaled by inv_n) written for pass 2.
template <bool EXPO, bool VEC>
__device__ __forceinline__ void ssim_pass1_strip(Ssim1Smem &sm, int W, int H, const float *xp, const float *yp, float ea,
                                                 float eb, const SsimTaps &tp, float inv_n, float *dmu, float *dexx,
                                                 float *dexy, int y_begin, int y_end, float2 &s_ssim, float2 &s_l1) {
    const int x0 = blockIdx.x * kSB - kSL;
    const int hr = hlane_row(threadIdx.x), ht = hlane_group(threadIdx.x);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, tc = tx ^ (tx >> 2);
    const int gx = blockIdx.x * kSB + tx;
    s_ssim = s_l1 = make_float2(0.f, 0.f);
    for (int y0 = y_begin - kSB; y0 < y_end; y0 += kSB) {   // the first step only makes the ten rows above the strip
        const bool lead = y0 < y_begin;
        const int rows = lead ? kHalo : kSB, first = lead ? y_begin - kR : y0 + kR;
        float4 xv[2], yv[2];
#pragma unroll
        for (int part = 0; part < 2; ++part) {   // every load before the first store
            const int i = threadIdx.x + 256 * part, r = i / (kSC / 4), c = (i - r * (kSC / 4)) * 4;
            const int lx = x0 + c, ly = first + r;
            xv[part] = yv[part] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < rows && ly >= 0 && ly < H) {
                xv[part] = load4<VEC>(xp + (long long)ly * W, lx, W);
                yv[part] = load4<VEC>(yp + (long long)ly * W, lx, W);
                if (EXPO) {   // the padding stays zero
                    float4 &x = xv[part];
                    if (lx >= 0 && lx < W) x.x = fp::add(fp::mul(ea, x.x), eb);
                    if (VEC ? lx >= 0 && lx < W : lx + 1 >= 0 && lx + 1 < W) x.y = fp::add(fp::mul(ea, x.y), eb);
                    if (VEC ? lx >= 0 && lx < W : lx + 2 >= 0 && lx + 2 < W) x.z = fp::add(fp::mul(ea, x.z), eb);
                    if (VEC ? lx >= 0 && lx < W : lx + 3 >= 0 && lx + 3 < W) x.w = fp::add(fp::mul(ea, x.w), eb);
                }
                if (c >= kSL && c < kSL + kSB && ly >= y_begin && ly < y_end) {   // the strip's own (zeros beyond W)
                    add_to_pair(s_l1, fabsf(xv[part].x - yv[part].x));
                    add_to_pair(s_l1, fabsf(xv[part].y - yv[part].y));
                    add_to_pair(s_l1, fabsf(xv[part].z - yv[part].z));
                    add_to_pair(s_l1, fabsf(xv[part].w - yv[part].w));
                }
            }
        }
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const int i = threadIdx.x + 256 * part, r = i / (kSC / 4), c = (i - r * (kSC / 4)) * 4;
            if (r >= rows) break;
            float4 *d = reinterpret_cast<float4 *>(&sm.xy[r][c]);
            d[0] = make_float4(xv[part].x, yv[part].x, xv[part].y, yv[part].y);
            d[1] = make_float4(xv[part].z, yv[part].z, xv[part].w, yv[part].w);
        }
        __syncthreads();   // inputs stored; the last step's vertical filter is done
        if (lead) {
            if (hr < kHalo) ssim1_hfilter(sm, tp, hr, ht, hr);
            __syncthreads();
            continue;
        }
        if (y0 > y_begin) {
            for (int i = threadIdx.x; i < kHalo * kSB; i += 256) {
                const int r = i / kSB, c = i % kSB;
                sm.h[r][c] = sm.h[kSB + r][c];
                sm.hxy[r][c] = sm.hxy[kSB + r][c];
            }
            __syncthreads();
        }
        ssim1_hfilter(sm, tp, hr, ht, kHalo + hr);
        __syncthreads();
        float2 m[kSVR], q[kSVR];
        float p[kSVR];
#pragma unroll
        for (int j = 0; j < kSVR; ++j) {
            m[j] = q[j] = make_float2(0.f, 0.f);
            p[j] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kSVR + 2 * kR; ++k) {
            const float4 v = sm.h[ty * kSVR + k][tc];
            const float vp = sm.hxy[ty * kSVR + k][tc];
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (k - j >= 0 && k - j <= 2 * kR) {
                    const float2 w = fp2::splat(tp.w[k - j]);
                    m[j] = fp2::fma(w, make_float2(v.x, v.y), m[j]);
                    q[j] = fp2::fma(w, make_float2(v.z, v.w), q[j]);
                    p[j] = fmaf(tp.w[k - j], vp, p[j]);
                }
            }
        }
        const int gy0 = y0 + ty * kSVR;
#pragma unroll
        for (int j = 0; j < kSVR; ++j) {
            if (gx >= W || gy0 + j >= y_end) break;
            const float mx = m[j].x, my = m[j].y, exx = q[j].x, eyy = q[j].y, exy = p[j];
            const float vx = exx - mx * mx, vy = eyy - my * my, cxy = exy - mx * my;
            const float A1 = 2.f * mx * my + kC1, A2 = 2.f * cxy + kC2;
            const float B1 = mx * mx + my * my + kC1, B2 = vx + vy + kC2;
            const float iB = 1.f / (B1 * B2), iB1 = iB * B2, iB2 = iB * B1;
            const float S = A1 * A2 * iB;
            add_to_pair(s_ssim, S);
            const long long o = (long long)(gy0 + j) * W + gx;
            dmu[o] = inv_n * ((2.f * my * A2 - 2.f * my * A1) * iB - S * (2.f * mx * iB1 - 2.f * mx * iB2));
            dexx[o] = inv_n * (-S * iB2);
            dexy[o] = inv_n * (2.f * A1 * iB);
        }
    }
}

// Pass 2 of a strip: the three derivative maps blurred (the adjoint of a zero-padded symmetric blur is the same
// blur).  Per step, before(y) is called ahead of the loads and after(y, ga, gb) with
// ga = (blur(dS/dmu_x), blur(dS/dE[x^2])) and gb = blur(dS/dE[xy]) of the thread's kSVR outputs, rows y ...
template <bool VEC, typename Before, typename After>
__device__ __forceinline__ void ssim_pass2_strip(Ssim2Smem &sm, int W, int H, const float *dmu, const float *dexx,
                                                 const float *dexy, const SsimTaps &tp, int y_begin, int y_end,
                                                 Before before, After after) {
    const int x0 = blockIdx.x * kSB - kSL;
    const int hr = hlane_row(threadIdx.x), ht = hlane_group(threadIdx.x);
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int y0 = y_begin - kSB; y0 < y_end; y0 += kSB) {
        const bool lead = y0 < y_begin;
        const int rows = lead ? kHalo : kSB, first = lead ? y_begin - kR : y0 + kR;
        if (!lead) before(y0 + ty * kSVR);
        float4 v0[2], v1[2], v2[2];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const int i = threadIdx.x + 256 * part, r = i / (kSC / 4), c = (i - r * (kSC / 4)) * 4;
            const int lx = x0 + c, ly = first + r;
            v0[part] = v1[part] = v2[part] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (r < rows && ly >= 0 && ly < H) {
                const long long o = (long long)ly * W;
                v0[part] = load4<VEC>(dmu + o, lx, W);
                v1[part] = load4<VEC>(dexx + o, lx, W);
                v2[part] = load4<VEC>(dexy + o, lx, W);
            }
        }
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            const int i = threadIdx.x + 256 * part, r = i / (kSC / 4), c = (i - r * (kSC / 4)) * 4;
            if (r >= rows) break;
            float4 *d = reinterpret_cast<float4 *>(&sm.a[r][c]);
            d[0] = make_float4(v0[part].x, v1[part].x, v0[part].y, v1[part].y);
            d[1] = make_float4(v0[part].z, v1[part].z, v0[part].w, v1[part].w);
            *reinterpret_cast<float4 *>(&sm.b[r][c]) = v2[part];
        }
        __syncthreads();
        if (lead) {
            if (hr < kHalo) ssim2_hfilter(sm, tp, hr, ht, hr);
            __syncthreads();
            continue;
        }
        if (y0 > y_begin) {
            for (int i = threadIdx.x; i < kHalo * kSB; i += 256) {
                const int r = i / kSB, c = i % kSB;
                sm.ha[r][c] = sm.ha[kSB + r][c];
                sm.hb[r][c] = sm.hb[kSB + r][c];
            }
            __syncthreads();
        }
        ssim2_hfilter(sm, tp, hr, ht, kHalo + hr);
        __syncthreads();
        float2 ga[kSVR];
        float gb[kSVR];
#pragma unroll
        for (int j = 0; j < kSVR; ++j) {
            ga[j] = make_float2(0.f, 0.f);
            gb[j] = 0.f;
        }
#pragma unroll
        for (int k = 0; k < kSVR + 2 * kR; ++k) {
            const float2 va = sm.ha[ty * kSVR + k][tx];
            const float vb = sm.hb[ty * kSVR + k][tx];
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (k - j >= 0 && k - j <= 2 * kR) {
                    ga[j] = fp2::fma(fp2::splat(tp.w[k - j]), va, ga[j]);
                    gb[j] = fmaf(tp.w[k - j], vb, gb[j]);
                }
            }
        }
        after(y0 + ty * kSVR, ga, gb);
    }
}

// the images at a thread's outputs, asked for before pass 2 waits for its inputs (on tiles, 8 views of 1200 x 680:
// 235 us with these loads after the filter, 173 us before it)
__device__ __forceinline__ void load_outputs(const float *x, const float *y, int W, int H, int gx, int gy0,
                                             float (&px)[kSVR], float (&py)[kSVR]) {
#pragma unroll
    for (int j = 0; j < kSVR; ++j) {
        const bool in = gx < W && gy0 + j < H;
        const long long o = (long long)(gy0 + j) * W + gx;
        px[j] = in ? x[o] : 0.f;
        py[j] = in ? y[o] : 0.f;
    }
}

// pass 1: per image plane (view * 3 + channel) = blockIdx.z, strip blockIdx.x, rows from blockIdx.y seg;
// sums[0] += |x - y|, sums[1] += SSIM
template <bool VEC>
__global__ void __launch_bounds__(256, 4) k_ssim1(int W, int H, int seg, const float *x, const float *y, SsimTaps tp,
                                                  float inv_n, float *dmu, float *dexx, float *dexy, double *sums) {
    __shared__ Ssim1Smem sm;
    const long long off = (long long)blockIdx.z * W * H;
    const int y_begin = blockIdx.y * seg;
    float2 s, l;
    ssim_pass1_strip<false, VEC>(sm, W, H, x + off, y + off, 1.f, 0.f, tp, inv_n, dmu + off, dexx + off, dexy + off,
                                 y_begin, min(H, y_begin + seg), s, l);
    block_add2(l, s, sums, sums + 1);
}

// pass 2: blur the three derivative maps and combine with the L1 gradient
template <bool VEC>
__global__ void __launch_bounds__(256, 4) k_ssim2(int W, int H, int seg, const float *x, const float *y, SsimTaps tp,
                                                  const float *dmu, const float *dexx, const float *dexy, float l1_scale,
                                                  float w_ssim, float *d_rgb) {
    __shared__ Ssim2Smem sm;
    const long long off = (long long)blockIdx.z * W * H;
    const int gx = blockIdx.x * kSB + (threadIdx.x & 31), y_begin = blockIdx.y * seg, y_end = min(H, y_begin + seg);
    float px[kSVR], py[kSVR];
    ssim_pass2_strip<VEC>(
        sm, W, H, dmu + off, dexx + off, dexy + off, tp, y_begin, y_end,
        [&](int gy0) { load_outputs(x + off, y + off, W, H, gx, gy0, px, py); },
        [&](int gy0, const float2(&ga)[kSVR], const float(&gb)[kSVR]) {
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (gx >= W || gy0 + j >= y_end) break;
                const float gs = ga[j].x + 2.f * px[j] * ga[j].y + py[j] * gb[j];
                d_rgb[off + (long long)(gy0 + j) * W + gx] = l1_scale * sgnf(px[j] - py[j]) - w_ssim * gs;
            }
        });
}

// Rows of a strip's segment, in steps of kSB: a CTA costs its steps and about half of one more (the ten rows above,
// the reduction), and the last of the waves of four CTAs per SM is half empty on average; the product is least at
// 11 of 22 steps for 24 planes of 1200 x 680 (pass 1 and pass 2 together 329 us; 5 steps 347, 4 steps 355, 2 steps
// 388), at one step for a single plane.
static int ssim_segment(int W, int H, long long planes) {
    const int steps = (H + kSB - 1) / kSB;
    const double strips = (double)((W + kSB - 1) / kSB) * planes, slots = 4.0 * device_sm_count();
    int best = 1;
    double least = 0.0;
    for (int n = 1; n <= steps; ++n) {
        const double waves = (steps + n - 1) / n * strips / slots + 0.5, cost = std::max(1.0, waves) * (n + 0.5);
        if (n == 1 || cost < least) {
            least = cost;
            best = n;
        }
    }
    return best * kSB;
}

__global__ void k_ssim_finish(double *scratch_sums, float w_l1, float w_ssim, double inv_n, double *loss) {
    // scratch_sums[0] = sum |x - y|, scratch_sums[1] = sum of the SSIM map
    *loss = w_l1 * scratch_sums[0] * inv_n + w_ssim * (1.0 - scratch_sums[1] * inv_n);
}

// 16-byte accesses: every row of every plane starts on such a boundary
static bool ssim_vec(int W, const float *x, const float *y, const float *maps) {
    return W % 4 == 0 && aligned16(x) && aligned16(y) && aligned16(maps);
}

size_t ssim_scratch_bytes(int V, int W, int H) {
    return 256 + 3 * sizeof(float) * (size_t)V * 3 * W * H;
}

// both passes over grid.z planes
static void launch_ssim(dim3 grid, int seg, int W, int H, const float *x, const float *y, const SsimTaps &taps, float inv_n,
                        float *dmu, float *dexx, float *dexy, double *sums, float l1_scale, float w_ssim, float *d_rgb,
                        cudaStream_t s) {
    if (ssim_vec(W, x, y, dmu)) {
        k_ssim1<true><<<grid, 256, 0, s>>>(W, H, seg, x, y, taps, inv_n, dmu, dexx, dexy, sums);
        k_ssim2<true><<<grid, 256, 0, s>>>(W, H, seg, x, y, taps, dmu, dexx, dexy, l1_scale, w_ssim, d_rgb);
    } else {
        k_ssim1<false><<<grid, 256, 0, s>>>(W, H, seg, x, y, taps, inv_n, dmu, dexx, dexy, sums);
        k_ssim2<false><<<grid, 256, 0, s>>>(W, H, seg, x, y, taps, dmu, dexx, dexy, l1_scale, w_ssim, d_rgb);
    }
}

int launch_loss_l1_ssim(int V, int W, int H, const float *rgb, const float *rgb_t, float w_l1, float w_ssim,
                        float *d_rgb, double *loss, void *scratch, cudaStream_t s) {
    static const SsimTaps taps = make_taps();
    const long long plane = (long long)W * H, n = 3LL * V * plane;
    double *sums = reinterpret_cast<double *>(scratch);
    float *dmu = reinterpret_cast<float *>(static_cast<char *>(scratch) + 256);
    float *dexx = dmu + n, *dexy = dexx + n;
    if (cudaMemsetAsync(sums, 0, 2 * sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    const int seg = ssim_segment(W, H, 3LL * V);
    dim3 grid((W + kSB - 1) / kSB, (H + seg - 1) / seg, 3 * V);
    const float inv_n = (float)(1.0 / (double)n);
    launch_ssim(grid, seg, W, H, rgb, rgb_t, taps, inv_n, dmu, dexx, dexy, sums, w_l1 * inv_n, w_ssim, d_rgb, s);
    k_ssim_finish<<<1, 1, 0, s>>>(sums, w_l1, w_ssim, 1.0 / (double)n, loss);
    count_launches(3);
    return check_launch();
}

// ------------------------------------------------------------------------------------------
// The loss above without a caller-provided scratch buffer (for callers that cannot allocate).
// Its scratch is this file's static device array: two running sums (256 bytes) followed by the
// three derivative maps of ONE image plane; planes are processed one after another on the
// caller's stream, each reusing the maps.
// ------------------------------------------------------------------------------------------
constexpr long long kNoallocMaxPlane = GS_SSIM_NOALLOC_MAX_PLANE;
constexpr size_t kNoallocBytes = 256 + 3 * sizeof(float) * (size_t)kNoallocMaxPlane;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoallocBytes];

static std::mutex g_noalloc_mu;
static void *g_noalloc_addr[64];

// Device address of g_noalloc_scratch on the current device.  (On the host the symbol names a
// host-side stand-in, never the device memory itself.)  Outside stream capture every call looks
// the address up again, which is cheap and stays right after a device reset has reloaded the
// module; while `s` is being captured the address cached by the last call outside capture is
// used, and without one the lookup is attempted once more.
static int noalloc_scratch(cudaStream_t s, void **out) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return GS_ERR_CUDA;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) != cudaSuccess) return GS_ERR_CUDA;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (cs == cudaStreamCaptureStatusNone || !g_noalloc_addr[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || p == nullptr) return GS_ERR_CUDA;
        g_noalloc_addr[dev] = p;
    }
    *out = g_noalloc_addr[dev];
    return GS_OK;
}

int launch_loss_l1_ssim_noalloc(int V, int W, int H, const float *rgb, const float *rgb_t, float w_l1,
                                float w_ssim, float *d_rgb, double *loss, cudaStream_t s) {
    const long long plane = (long long)W * H, n = 3LL * V * plane;
    if (plane > kNoallocMaxPlane) return GS_ERR_TOO_LARGE;
    static const SsimTaps taps = make_taps();
    void *base = nullptr;
    int rc = noalloc_scratch(s, &base);
    if (rc) return rc;
    double *sums = reinterpret_cast<double *>(base);
    float *dmu = reinterpret_cast<float *>(static_cast<char *>(base) + 256);
    float *dexx = dmu + plane, *dexy = dexx + plane;
    if (cudaMemsetAsync(sums, 0, 2 * sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    const float inv_n = (float)(1.0 / (double)n);
    const int seg = ssim_segment(W, H, 1);
    dim3 grid((W + kSB - 1) / kSB, (H + seg - 1) / seg, 1);
    for (long long p = 0; p < 3LL * V; ++p) {
        const long long off = p * plane;
        launch_ssim(grid, seg, W, H, rgb + off, rgb_t + off, taps, inv_n, dmu, dexx, dexy, sums, w_l1 * inv_n, w_ssim,
                    d_rgb + off, s);
    }
    k_ssim_finish<<<1, 1, 0, s>>>(sums, w_l1, w_ssim, 1.0 / (double)n, loss);
    count_launches((int)(1 + 6LL * V));
    return check_launch();
}

// ------------------------------------------------------------------------------------------
// Adam
// ------------------------------------------------------------------------------------------
struct AdamArgs {
    long long n;
    float *p[5];            // means, log_scales, quats, opacity_logits, colors
    float *opac;            // activated opacity (rewritten)
    float *g[5];            // grads: means, log_scales, quats, opacities (w.r.t. o), colors
    float *m, *v;
    const int32_t *step;
    float lr[5];
    int zero;
    float iso_weight;       // lambda_s of the isotropy regulariser (0: none)
    double *iso_loss;       // optional: receives lambda_s L_iso (overwritten)
};

// Gradient of the isotropy regulariser (Eq. 4), lambda_s sum_axes |s - mean(s)| with s = exp(log-scale), of one
// Gaussian: with respect to log-scale b it is lambda_s (sg_b - mean(sg)) s_b, sg = sign(s - mean).  Returns the
// sum over the axes.
__device__ __forceinline__ float iso_grad(const float *ls, float weight, float (&giso)[3]) {
    float sc[3], sg[3], lsum = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) sc[k] = expf(ls[k]);
    const float sbar = (sc[0] + sc[1] + sc[2]) * (1.f / 3.f);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float d = sc[k] - sbar;
        sg[k] = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
        lsum += fabsf(d);
    }
    const float sgm = (sg[0] + sg[1] + sg[2]) * (1.f / 3.f);
#pragma unroll
    for (int k = 0; k < 3; ++k) giso[k] = weight * (sg[k] - sgm) * sc[k];
    return lsum;
}

template <int VEC>
__device__ __forceinline__ void load_vec(const float *p, float (&v)[VEC]) {
    if constexpr (VEC == 4) {
        const float4 t = *reinterpret_cast<const float4 *>(p);
        v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else {
        v[0] = *p;
    }
}
template <int VEC>
__device__ __forceinline__ void store_vec(float *p, const float (&v)[VEC]) {
    if constexpr (VEC == 4)
        *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
    else
        *p = v[0];
}

// VEC scalars of one group: parameter pv, gradient gv and moments mv, vv, the learning rate lr and the bias
// corrections c1, c2
template <int VEC>
__device__ __forceinline__ void adam_step(float (&pv)[VEC], const float (&gv)[VEC], float (&mv)[VEC], float (&vv)[VEC],
                                          float lr, float c1, float c2) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-15f;
#pragma unroll
    for (int d = 0; d < VEC; ++d) {
        const float gr = gv[d];
        mv[d] = b1 * mv[d] + (1.f - b1) * gr;
        vv[d] = b2 * vv[d] + (1.f - b2) * gr * gr;
        pv[d] = pv[d] - lr * (mv[d] / c1) / (sqrtf(vv[d] / c2) + eps);
    }
}

// Moments are stored group-major, in the same layout as the parameters ([N,3] means | [N,3] log-scales |
// [N,4] quats | [N] logits | [N,3] colours), so the step is one pass over 14 N scalars, VEC at a time: 4 where
// every group of every array starts on a 16-byte boundary (N a multiple of 4), else 1.  With the isotropy
// regulariser the log-scales go first, 32 VEC Gaussians to a warp: the warp reads all their log-scales before it
// writes any, and each lane takes the regulariser of VEC whole Gaussians through shared memory.
// Bound by memory: 1 M Gaussians move 392 MB in 68 us (58 us at the copy rate); a thread per Gaussian, whose
// stores are 4 bytes 12 or 16 apart, took 103 us.  One resident wave of CTAs: the two powers of the bias
// correction cost a thread more than a step of the loop (a CTA per 256 units: 77 to 90 us).
template <int VEC>
__global__ void __launch_bounds__(256, 4) k_adam(AdamArgs a) {
    __shared__ __align__(16) float s_ls[8][96 * VEC];
    const int t = *a.step + 1;
    const float c1 = 1.f - powf(0.9f, (float)t), c2 = 1.f - powf(0.999f, (float)t);
    const int lane = threadIdx.x & 31;
    const bool iso = a.iso_weight != 0.f;
    if (iso) {
        float *ls = s_ls[threadIdx.x >> 5];
        const long long n3 = 3 * a.n, stride = (long long)gridDim.x * (blockDim.x >> 5) * (96 * VEC);
        double liso = 0.0;
        for (long long c = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (96 * VEC); c < n3; c += stride) {
            float pv[3][VEC];
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int o = (q * 32 + lane) * VEC;
                if (c + o < n3) {
                    load_vec(a.p[1] + c + o, pv[q]);
                    store_vec(ls + o, pv[q]);
                }
            }
            __syncwarp();
#pragma unroll
            for (int d = 0; d < VEC; ++d) {
                const int o = 3 * (d * 32 + lane);
                if (c + o < n3) {
                    float gi[3];
                    liso += (double)(a.iso_weight * iso_grad(ls + o, a.iso_weight, gi));
#pragma unroll
                    for (int k = 0; k < 3; ++k) ls[o + k] = gi[k];
                }
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int o = (q * 32 + lane) * VEC;
                if (c + o >= n3) break;
                const long long e = n3 + c + o;
                float gv[VEC], gi[VEC], mv[VEC], vv[VEC];
                load_vec(a.g[1] + c + o, gv);
                load_vec(a.m + e, mv);
                load_vec(a.v + e, vv);
                load_vec(ls + o, gi);
#pragma unroll
                for (int d = 0; d < VEC; ++d) gv[d] += gi[d];
                adam_step(pv[q], gv, mv, vv, a.lr[1], c1, c2);
                store_vec(a.m + e, mv);
                store_vec(a.v + e, vv);
                store_vec(a.p[1] + c + o, pv[q]);
                if (a.zero) {
#pragma unroll
                    for (int d = 0; d < VEC; ++d) gv[d] = 0.f;
                    store_vec(a.g[1] + c + o, gv);
                }
            }
            __syncwarp();
        }
        if (a.iso_loss) {   // one double atomic per warp
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) liso += __shfl_xor_sync(0xffffffffu, liso, o);
            if (lane == 0 && liso != 0.0) atomicAdd(a.iso_loss, liso);
        }
    }
    const long long done = iso ? 3 * a.n : 0, total = 14 * a.n - done, stride = (long long)gridDim.x * blockDim.x * VEC;
    for (long long f = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * VEC; f < total; f += stride) {
        const long long e = f < 3 * a.n ? f : f + done;
        const int grp = e < 3 * a.n ? 0 : e < 6 * a.n ? 1 : e < 10 * a.n ? 2 : e < 11 * a.n ? 3 : 4;
        const long long i = e - (grp == 0 ? 0 : grp == 1 ? 3 * a.n : grp == 2 ? 6 * a.n : grp == 3 ? 10 * a.n : 11 * a.n);
        float *pp = (grp == 0 ? a.p[0] : grp == 1 ? a.p[1] : grp == 2 ? a.p[2] : grp == 3 ? a.p[3] : a.p[4]) + i;
        float *gp = (grp == 0 ? a.g[0] : grp == 1 ? a.g[1] : grp == 2 ? a.g[2] : grp == 3 ? a.g[3] : a.g[4]) + i;
        const float lr = grp == 0 ? a.lr[0] : grp == 1 ? a.lr[1] : grp == 2 ? a.lr[2] : grp == 3 ? a.lr[3] : a.lr[4];
        float pv[VEC], gv[VEC], mv[VEC], vv[VEC], ov[VEC];
        load_vec(gp, gv);
        load_vec(a.m + e, mv);
        load_vec(a.v + e, vv);
        load_vec(pp, pv);
        if (grp == 3) {
            load_vec(a.opac + i, ov);
#pragma unroll
            for (int d = 0; d < VEC; ++d) gv[d] *= ov[d] * (1.f - ov[d]);
        }
        adam_step(pv, gv, mv, vv, lr, c1, c2);
        store_vec(a.m + e, mv);
        store_vec(a.v + e, vv);
        store_vec(pp, pv);
        if (grp == 3) {
#pragma unroll
            for (int d = 0; d < VEC; ++d) ov[d] = 1.f / (1.f + __expf(-pv[d]));
            store_vec(a.opac + i, ov);
        }
        if (a.zero) {
#pragma unroll
            for (int d = 0; d < VEC; ++d) gv[d] = 0.f;
            store_vec(gp, gv);
        }
    }
}

__global__ void k_step_inc(int32_t *step) { *step += 1; }

int launch_adam(long long n, const gs_adam_state &st, const gs_grads &g, const float lr[5], int zero_grads,
                cudaStream_t s, float iso_weight, double *iso_loss) {
    AdamArgs a;
    a.iso_weight = iso_weight;
    a.iso_loss = iso_loss;
    if (iso_loss && cudaMemsetAsync(iso_loss, 0, sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    a.n = n;
    a.p[0] = st.means; a.p[1] = st.log_scales; a.p[2] = st.quats; a.p[3] = st.opacity_logits; a.p[4] = st.colors;
    a.opac = st.opacities;
    a.g[0] = g.means; a.g[1] = g.log_scales; a.g[2] = g.quats; a.g[3] = g.opacities; a.g[4] = g.colors;
    a.m = st.m;
    a.v = st.v;
    a.step = st.step;
    for (int k = 0; k < 5; ++k) a.lr[k] = lr[k];
    a.zero = zero_grads;
    if (n > 0) {
        bool vec = n % 4 == 0 && aligned16(a.opac) && aligned16(a.m) && aligned16(a.v);
        for (int k = 0; k < 5; ++k) vec = vec && aligned16(a.p[k]) && aligned16(a.g[k]);
        const long long threads = vec ? 14 * n / 4 : 14 * n;
        const int grid = (int)std::min<long long>((threads + 255) / 256, (long long)device_sm_count() * 4);
        if (vec)
            k_adam<4><<<grid, 256, 0, s>>>(a);
        else
            k_adam<1><<<grid, 256, 0, s>>>(a);
        count_launches(1);
    }
    k_step_inc<<<1, 1, 0, s>>>(st.step);
    count_launches(1);
    return check_launch();
}

}  // namespace gs

namespace gs {

// ------------------------------------------------------------------------------------------
// Joint refinement (Sec. III-C, Eq. 23): loss on the exposure-compensated render
// I~_v = exp(a_v) I^_v + b_v, its gradients with respect to I^, D^ and (a_v, b_v); pruning of
// Gaussians with opacity below a threshold; Adam on per-view pose deltas and exposures.
// ------------------------------------------------------------------------------------------
// I~ is formed as fl(fl(e^a I^) + b) with the decision-chain exponential, so the sign of the L1 term
// (an FP32 decision) is reproducible by any implementation that follows the same two roundings.
struct RefineArgs {
    int V, W, H;
    const float *rgb, *rgb_t, *depth, *depth_t, *expo;
    float w_l1, w_ssim, w_depth;
    float *d_rgb, *d_depth, *d_expo;
    double *loss;
    double *sums;          // [0] sum |I~ - I|, [1] sum SSIM map, [2] sum |D^ - D-|, then g_a[V], g_b[V]
    float *dmu, *dexx, *dexy;
};

// the depth term, 16 bytes at a time where the maps allow it (8 views of 1200 x 680, 78 MB: 15 us, 23 us with
// 4-byte accesses)
template <int VEC>
__global__ void __launch_bounds__(256) k_refine_depth(RefineArgs a) {
    const long long total = (long long)a.V * a.W * a.H;
    const long long stride = (long long)gridDim.x * blockDim.x * VEC;
    float2 acc = make_float2(0.f, 0.f);
    const float sc_d = (float)((double)a.w_depth / (double)total);
    for (long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * VEC; i < total; i += stride) {
        float x[VEC], y[VEC], g[VEC];
        load_vec(a.depth + i, x);
        load_vec(a.depth_t + i, y);
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
            const float d = x[k] - y[k];
            add_to_pair(acc, fabsf(d));
            g[k] = sgnf(d) * sc_d;
        }
        store_vec(a.d_depth + i, g);
    }
    block_add_double(pair_value(acc), a.sums + 2);
}

template <bool VEC>
__global__ void __launch_bounds__(256, 4) k_refine_ssim1(RefineArgs a, int seg, SsimTaps tp, float inv_n) {
    __shared__ Ssim1Smem sm;
    const long long plane = blockIdx.z;
    const int v = (int)(plane / 3);
    const float ea = spec_expf(a.expo[2 * v]), eb = a.expo[2 * v + 1];
    const long long off = plane * (long long)a.W * a.H;
    float2 s, l;
    const int y_begin = blockIdx.y * seg;
    ssim_pass1_strip<true, VEC>(sm, a.W, a.H, a.rgb + off, a.rgb_t + off, ea, eb, tp, inv_n, a.dmu + off, a.dexx + off,
                                a.dexy + off, y_begin, min(a.H, y_begin + seg), s, l);
    block_add2(l, s, a.sums, a.sums + 1);
}

template <bool VEC>
__global__ void __launch_bounds__(256, 4) k_refine_ssim2(RefineArgs a, int seg, SsimTaps tp, float l1_scale) {
    __shared__ Ssim2Smem sm;
    const int W = a.W, H = a.H;
    const long long plane = blockIdx.z;
    const int v = (int)(plane / 3);
    const float ea = spec_expf(a.expo[2 * v]), eb = a.expo[2 * v + 1];
    const long long off = plane * (long long)W * H;
    const int gx = blockIdx.x * kSB + (threadIdx.x & 31), y_begin = blockIdx.y * seg, y_end = min(H, y_begin + seg);
    float px[kSVR], py[kSVR];
    float2 sa = make_float2(0.f, 0.f), sb = sa;
    ssim_pass2_strip<VEC>(
        sm, W, H, a.dmu + off, a.dexx + off, a.dexy + off, tp, y_begin, y_end,
        [&](int gy0) { load_outputs(a.rgb + off, a.rgb_t + off, W, H, gx, gy0, px, py); },
        [&](int gy0, const float2(&ba)[kSVR], const float(&bb)[kSVR]) {
            float ga = 0.f, gb = 0.f;
#pragma unroll
            for (int j = 0; j < kSVR; ++j) {
                if (gx >= W || gy0 + j >= y_end) break;
                const float xv = px[j], yv = py[j];
                const float xt = fp::add(fp::mul(ea, xv), eb);   // I~ exactly as the FP32 L1 sign decision takes it
                const float g = l1_scale * sgnf(xt - yv) - a.w_ssim * (ba[j].x + 2.f * xt * ba[j].y + yv * bb[j]);
                a.d_rgb[off + (long long)(gy0 + j) * W + gx] = ea * g;   // dL/dI^ = e^a dL/dI~
                ga += g * ea * xv;
                gb += g;
            }
            add_to_pair(sa, ga);
            add_to_pair(sb, gb);
        });
    block_add2(sa, sb, a.sums + 3 + v, a.sums + 3 + a.V + v);
}

__global__ void k_refine_finish(RefineArgs a, double inv_n) {
    const int v = threadIdx.x;
    if (v == 0) {
        const double npx = (double)a.V * a.W * a.H;
        *a.loss = a.w_l1 * a.sums[0] * inv_n + a.w_ssim * (1.0 - a.sums[1] * inv_n) + a.w_depth * a.sums[2] / npx;
    }
    if (v < a.V && a.d_expo) {
        a.d_expo[2 * v] = (float)a.sums[3 + v];
        a.d_expo[2 * v + 1] = (float)a.sums[3 + a.V + v];
    }
}

size_t refine_scratch_bytes(int V, int W, int H) {
    const size_t head = ((size_t)(3 + 2 * V) * sizeof(double) + 255) & ~(size_t)255;
    return head + 3 * sizeof(float) * (size_t)V * 3 * W * H;
}

int launch_loss_refine(int V, int W, int H, const float *rgb, const float *rgb_t, const float *depth,
                       const float *depth_t, const float *expo, float w_l1, float w_ssim, float w_depth, float *d_rgb,
                       float *d_depth, float *d_expo, double *loss, void *scratch, cudaStream_t s) {
    static const SsimTaps taps = make_taps();
    const long long plane = (long long)W * H, n = 3LL * V * plane;
    const size_t head = ((size_t)(3 + 2 * V) * sizeof(double) + 255) & ~(size_t)255;
    RefineArgs a;
    a.V = V; a.W = W; a.H = H;
    a.rgb = rgb; a.rgb_t = rgb_t; a.depth = depth; a.depth_t = depth_t; a.expo = expo;
    a.w_l1 = w_l1; a.w_ssim = w_ssim; a.w_depth = (depth && depth_t && d_depth) ? w_depth : 0.f;
    a.d_rgb = d_rgb; a.d_depth = (depth && depth_t) ? d_depth : nullptr; a.d_expo = d_expo;
    a.loss = loss;
    a.sums = reinterpret_cast<double *>(scratch);
    a.dmu = reinterpret_cast<float *>(static_cast<char *>(scratch) + head);
    a.dexx = a.dmu + n;
    a.dexy = a.dexx + n;
    if (cudaMemsetAsync(a.sums, 0, (size_t)(3 + 2 * V) * sizeof(double), s) != cudaSuccess) return GS_ERR_CUDA;
    const float inv_n = (float)(1.0 / (double)n);
    const long long total = (long long)V * plane;
    const int g1 = (int)std::max<long long>(1, std::min<long long>((total + 255) / 256, (long long)device_sm_count() * 8));
    const bool use_depth = a.depth && a.d_depth;
    const bool vec_d = total % 4 == 0 && aligned16(a.depth) && aligned16(a.depth_t) && aligned16(a.d_depth);
    if (use_depth && vec_d) k_refine_depth<4><<<g1, 256, 0, s>>>(a);
    if (use_depth && !vec_d) k_refine_depth<1><<<g1, 256, 0, s>>>(a);
    const int seg = ssim_segment(W, H, 3LL * V);
    dim3 grid((W + kSB - 1) / kSB, (H + seg - 1) / seg, 3 * V);
    if (ssim_vec(W, rgb, rgb_t, a.dmu)) {
        k_refine_ssim1<true><<<grid, 256, 0, s>>>(a, seg, taps, inv_n);
        k_refine_ssim2<true><<<grid, 256, 0, s>>>(a, seg, taps, w_l1 * inv_n);
    } else {
        k_refine_ssim1<false><<<grid, 256, 0, s>>>(a, seg, taps, inv_n);
        k_refine_ssim2<false><<<grid, 256, 0, s>>>(a, seg, taps, w_l1 * inv_n);
    }
    k_refine_finish<<<1, ((V + 31) / 32) * 32, 0, s>>>(a, 1.0 / (double)n);
    count_launches(3 + use_depth);
    return check_launch();
}

// ---- pruning: order-preserving compaction of the Gaussians with opacity >= threshold ----
__global__ void k_prune_flags(long long n, const float *op, float thr, uint32_t *flags) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        flags[i] = op[i] >= thr ? 1u : 0u;
}

__global__ void k_prune_scatter(long long n, gs_gaussians in, gs_gaussian_arrays out, const uint32_t *incl,
                                long long *kept) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const uint32_t hi = incl[i], lo = i > 0 ? incl[i - 1] : 0u;
        if (i == n - 1) *kept = (long long)hi;
        if (hi == lo) continue;
        const long long j = hi - 1;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            out.means[3 * j + k] = in.means[3 * i + k];
            out.log_scales[3 * j + k] = in.log_scales[3 * i + k];
            out.colors[3 * j + k] = in.colors[3 * i + k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) out.quats[4 * j + k] = in.quats[4 * i + k];
        out.opacities[j] = in.opacities[i];
    }
}

size_t prune_scratch_bytes(long long n) {
    const long long parts = (n + kScanTile - 1) / kScanTile;
    return 256 + (((size_t)n * 4 + 255) & ~(size_t)255) + (size_t)parts * 8;
}

int launch_prune(long long n, const gs_gaussians &in, float thr, const gs_gaussian_arrays &out, long long *kept,
                 void *scratch, cudaStream_t s) {
    BinArgs b;
    std::memset(&b, 0, sizeof(b));
    b.st = reinterpret_cast<DevStatus *>(scratch);
    b.touched = reinterpret_cast<uint32_t *>(static_cast<char *>(scratch) + 256);
    b.scan_state = reinterpret_cast<unsigned long long *>(static_cast<char *>(scratch) + 256 +
                                                          (((size_t)n * 4 + 255) & ~(size_t)255));
    b.P = n;
    b.cap = (1LL << 30) - 1;
    b.fault_scan_part = -1;
    b.spin_limit = kSpinLimit;
    if (cudaMemsetAsync(b.st, 0, sizeof(DevStatus), s) != cudaSuccess) return GS_ERR_CUDA;
    const int grid = (int)std::max<long long>(1, std::min<long long>((n + 255) / 256, (long long)device_sm_count() * 8));
    k_prune_flags<<<grid, 256, 0, s>>>(n, in.opacities, thr, b.touched);
    count_launches(1);
    int rc = run_scan_only(b, s);
    if (rc) return rc;
    k_prune_scatter<<<grid, 256, 0, s>>>(n, in, out, b.touched, kept);
    count_launches(1);
    return check_launch();
}

// ---- per-view Adam on the pose delta (applied as T <- Exp(delta) T) and the exposure ----
__global__ void k_view_adam(int V, gs_camera *cams, float *expo, float *m, float *vv, const int32_t *step,
                            const float *pose_grad, const float *expo_grad, float lr_pose, float lr_expo) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    const int t = *step + 1;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-15f;
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    float d[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float g = k < 6 ? pose_grad[6 * v + k] : expo_grad[2 * v + (k - 6)];
        const float mm = b1 * m[8 * v + k] + (1.f - b1) * g;
        const float vk = b2 * vv[8 * v + k] + (1.f - b2) * g * g;
        m[8 * v + k] = mm;
        vv[8 * v + k] = vk;
        d[k] = -(k < 6 ? lr_pose : lr_expo) * (mm / c1) / (sqrtf(vk / c2) + eps);
    }
    expo[2 * v] += d[6];
    expo[2 * v + 1] += d[7];
    // Exp of the twist (rho = d[0..2], phi = d[3..5]): Rodrigues rotation and left Jacobian
    const float px = d[3], py = d[4], pz = d[5];
    const float th2 = px * px + py * py + pz * pz, th = sqrtf(th2);
    float A, B, Cc;   // Exp(phi) = I + A K + B K^2 ; Jl = I + B K + Cc K^2
    if (th < 1e-4f) {
        A = 1.f - th2 / 6.f;
        B = 0.5f - th2 / 24.f;
        Cc = 1.f / 6.f - th2 / 120.f;
    } else {
        A = sinf(th) / th;
        B = (1.f - cosf(th)) / th2;
        Cc = (th - sinf(th)) / (th2 * th);
    }
    const float K[9] = {0.f, -pz, py, pz, 0.f, -px, -py, px, 0.f};
    float K2[9], Rx[9], Jl[9];
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) K2[3 * i + j] = K[3 * i] * K[j] + K[3 * i + 1] * K[3 + j] + K[3 * i + 2] * K[6 + j];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float I = (i % 4 == 0) ? 1.f : 0.f;
        Rx[i] = I + A * K[i] + B * K2[i];
        Jl[i] = I + B * K[i] + Cc * K2[i];
    }
    gs_camera c = cams[v];
    float R[9], tt[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) R[3 * i + j] = Rx[3 * i] * c.R[j] + Rx[3 * i + 1] * c.R[3 + j] + Rx[3 * i + 2] * c.R[6 + j];
        tt[i] = Rx[3 * i] * c.t[0] + Rx[3 * i + 1] * c.t[1] + Rx[3 * i + 2] * c.t[2] + Jl[3 * i] * d[0] +
                Jl[3 * i + 1] * d[1] + Jl[3 * i + 2] * d[2];
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) c.R[i] = R[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) c.t[i] = tt[i];
    cams[v] = c;
}

int launch_view_adam(int V, const gs_view_adam_state &st, const float *pose_grad, const float *expo_grad, float lr_pose,
                     float lr_expo, cudaStream_t s) {
    k_view_adam<<<(V + 127) / 128, 128, 0, s>>>(V, st.cameras, st.expo, st.m, st.v, st.step, pose_grad, expo_grad,
                                                 lr_pose, lr_expo);
    k_step_inc<<<1, 1, 0, s>>>(st.step);
    count_launches(2);
    return check_launch();
}

// ------------------------------------------------------------------------------------------
// zeroing of the five gradient arrays in one launch
// ------------------------------------------------------------------------------------------
struct ZeroArgs {
    float *p[5];
    long long len[5];     // floats per array
};

// grid (blocks, 5): row y clears array y, 16 bytes per store where the pointer allows it.
__global__ void k_zero_grads(ZeroArgs a) {
    float *p = a.p[blockIdx.y];
    const long long n = a.len[blockIdx.y];
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long head = 0;
    if (((uintptr_t)p & 15u) == 0) {
        const long long n4 = n >> 2;
        float4 *q = reinterpret_cast<float4 *>(p);
        for (long long i = t0; i < n4; i += stride) q[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        head = n4 << 2;
    }
    for (long long i = head + t0; i < n; i += stride) p[i] = 0.f;
}

int launch_grads_zero(long long n, const gs_grads &g, cudaStream_t s) {
    ZeroArgs a;
    float *ptr[5] = {g.means, g.log_scales, g.quats, g.opacities, g.colors};
    const long long per[5] = {3, 3, 4, 1, 3};
    for (int k = 0; k < 5; ++k) {
        a.p[k] = ptr[k];
        a.len[k] = per[k] * n;
    }
    const long long blocks = std::max<long long>(1, std::min<long long>((4 * n + 1023) / 1024,
                                                                        (long long)device_sm_count() * 2));
    k_zero_grads<<<dim3((unsigned)blocks, 5), 256, 0, s>>>(a);
    count_launches(1);
    return check_launch();
}

}  // namespace gs
