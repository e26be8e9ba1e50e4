// Dense supporting layers of the MobileNet-v1 chain: depthwise 3x3, the thin-input first 3x3
// convolution and the global average pool.  All are bandwidth-bound: every kernel reads and
// writes NHWC rows with float4 accesses that are contiguous across a warp.
#include "common.h"
#include "pipeline.cuh"

namespace sbnn {
namespace {

// ---- depthwise 3x3 --------------------------------------------------------------------------
// One thread: 4 channels x TW consecutive output columns of one output row.  The 3 x (S*(TW-1)+3)
// input window is read once into registers and slides across the TW outputs.
// WIDE: 92 registers instead of 66 (96, 78 at stride 2), for more loads in flight, where two CTAs an SM take the whole launch (1 x 13 x
// 13 x 40 3.6 -> 3.2 us, 2 x 28 x 28 x 256 at stride 2 4.0 -> 3.4); with more it loses (9 x 28 x 28 x 256, 441 CTAs, 5.1 -> 6.6).
template <int S, int TW, bool WIDE>
__global__ void __launch_bounds__(256, WIDE ? 1 : 0)
dwconv3x3_kernel(const float* __restrict__ w, const float* __restrict__ b, const float* __restrict__ x,
                 float* __restrict__ y, int N, int H, int W, int C, int Ho, int Wo, int relu) {
    const int C4 = C >> 2;
    const int strips = (Wo + TW - 1) / TW;
    const int64_t total = (int64_t)N * Ho * strips * C4;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int c4 = (int)(t % C4);
    int64_t r = t / C4;
    const int sx = (int)(r % strips); r /= strips;
    const int oy = (int)(r % Ho);
    const int n = (int)(r / Ho);
    const int ox0 = sx * TW;
    constexpr int IW = S * (TW - 1) + 3;

    const float4* w4 = reinterpret_cast<const float4*>(w);
    float4 wk[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) wk[i] = __ldg(w4 + i * C4 + c4);
    const float4 bias = b ? __ldg(reinterpret_cast<const float4*>(b) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 acc[TW];
#pragma unroll
    for (int i = 0; i < TW; ++i) acc[i] = bias;

    const int ix0 = ox0 * S - 1;
#pragma unroll
    for (int kh = 0; kh < 3; ++kh) {
        const int iy = oy * S + kh - 1;
        if (iy < 0 || iy >= H) continue;
        const float4* row = reinterpret_cast<const float4*>(x + ((size_t)n * H + iy) * W * C) + c4;
        float4 in[IW];
#pragma unroll
        for (int j = 0; j < IW; ++j) {
            const int ix = ix0 + j;
            in[j] = (ix >= 0 && ix < W) ? __ldg(row + (size_t)ix * C4) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < TW; ++i)
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) {
                const float4 v = in[i * S + kw], k = wk[kh * 3 + kw];
                acc[i].x = fmaf(v.x, k.x, acc[i].x);
                acc[i].y = fmaf(v.y, k.y, acc[i].y);
                acc[i].z = fmaf(v.z, k.z, acc[i].z);
                acc[i].w = fmaf(v.w, k.w, acc[i].w);
            }
    }
    float4* out = reinterpret_cast<float4*>(y + (((size_t)n * Ho + oy) * Wo) * C) + c4;
#pragma unroll
    for (int i = 0; i < TW; ++i) {
        const int ox = ox0 + i;
        if (ox >= Wo) break;
        float4 v = acc[i];
        if (relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
        out[(size_t)ox * C4] = v;
    }
}

// A thread's outputs next to the border once more without the taps above and below the image, for weights that are not finite:
// the sliding kernel multiplies the zeros there, which then is not nothing.
template <int S>
__device__ __forceinline__ void dw_rows_inside(const float* w, const float* b, const float* x, float* y, int H, int W, int C, int Ho, int Wo, int relu,
                                               int TW, int R) {
    const unsigned C4 = (unsigned)C >> 2, strips = (Wo + TW - 1) / TW, segs = (Ho + R - 1) / R;
    const unsigned t = blockIdx.x * 256u + threadIdx.x;
    const int c = (int)(t % C4) * 4, ox0 = (int)(t / C4 % strips) * TW, oy0 = (int)(t / C4 / strips % segs) * R;
    const size_t n = t / C4 / strips / segs;
    if constexpr (S == 1) {       // outputs that bad activations alone have spoiled stay as they are (at stride 2 this look costs registers)
        float probe = 0.0f;
#pragma unroll 1
        for (int k = 0; k < 9; ++k) {
            const float4 g = *reinterpret_cast<const float4*>(w + (size_t)k * C + c);
            probe = fmaf(g.x, 0.f, fmaf(g.y, 0.f, fmaf(g.z, 0.f, fmaf(g.w, 0.f, probe))));
        }
        if (probe == 0.0f) return;
    }
#pragma unroll 1
    for (int oy = oy0; oy < min(oy0 + R, Ho); ++oy) {
        if (oy > 0 && oy * S + 2 <= H) continue;
#pragma unroll 1
        for (int ox = ox0; ox < min(ox0 + TW, Wo); ++ox) {
            float4 acc = b ? *reinterpret_cast<const float4*>(b + c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
            for (int k = 0; k < 9; ++k) {
                const int iy = oy * S + k / 3 - 1, ix = ox * S + k % 3 - 1;
                if (iy < 0 || iy >= H) continue;
                const float4 g = *reinterpret_cast<const float4*>(w + (size_t)k * C + c);
                float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                if (ix >= 0 && ix < W) v = *reinterpret_cast<const float4*>(x + ((n * H + iy) * W + ix) * C + c);
                acc.x = fmaf(v.x, g.x, acc.x); acc.y = fmaf(v.y, g.y, acc.y); acc.z = fmaf(v.z, g.z, acc.z); acc.w = fmaf(v.w, g.w, acc.w);
            }
            if (relu) acc = make_float4(fmaxf(acc.x, 0.f), fmaxf(acc.y, 0.f), fmaxf(acc.z, 0.f), fmaxf(acc.w, 0.f));
            *reinterpret_cast<float4*>(y + ((n * Ho + oy) * Wo + ox) * C + c) = acc;
        }
    }
}

// The same for launches with enough work: one thread slides down R output rows of TW columns, 4 channels wide.  Every input
// row is loaded once (a row ahead of its use) and added to the up to three output rows it belongs to, so an output costs
// (TW + 2) / TW loads instead of 3 (TW + 2) / TW, and the FMAs are packed pairs.  Bound by HBM (and by the 5 or 6 row
// loads in flight a thread; wider strips spill).  64 x 56 x 56 x 128: 55.9 -> 42.1 us (4.9 TB/s), 64 x 112 x 112 x 64 at
// stride 2: 57.7 -> 44.8 us.
template <int S, int TW, int R>
__global__ void __launch_bounds__(256, 2)
dwconv3x3_slide_kernel(const float* __restrict__ w, const float* __restrict__ b, const float* __restrict__ x, float* __restrict__ y, int N,
                       int H, int W, int C, int Ho, int Wo, int relu) {
    constexpr int IW = S * (TW - 1) + 3, ROWS = S * (R - 1) + 3;
    const unsigned C4 = (unsigned)C >> 2, strips = (Wo + TW - 1) / TW, segs = (Ho + R - 1) / R;
    unsigned t = blockIdx.x * 256u + threadIdx.x;
    const unsigned c4 = t % C4;
    t /= C4;
    const int ox0 = (int)(t % strips) * TW;
    t /= strips;
    const int oy0 = (int)(t % segs) * R, n = (int)(t / segs);
    if (n >= N) return;

    const ulonglong2* w4 = reinterpret_cast<const ulonglong2*>(w) + c4;
    ulonglong2 wk[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) wk[i] = __ldg(w4 + (size_t)i * C4);
    ulonglong2 bias = make_ulonglong2(0, 0);
    if (b) bias = __ldg(reinterpret_cast<const ulonglong2*>(b) + c4);

    const int ix0 = ox0 * S - 1, iy0 = oy0 * S - 1;
    const ulonglong2* src = reinterpret_cast<const ulonglong2*>(x) + (((long long)n * H + iy0) * W + ix0) * C4 + c4;
    auto load = [&](int r, ulonglong2 (&in)[IW]) {
        const bool row = (unsigned)(iy0 + r) < (unsigned)H;
#pragma unroll
        for (int j = 0; j < IW; ++j) {
            in[j] = make_ulonglong2(0, 0);
            if (row && (unsigned)(ix0 + j) < (unsigned)W) in[j] = __ldg(src + ((long long)r * W + j) * C4);
        }
    };
    ulonglong2 in[2][IW], acc[3][TW];
    bool again = false;       // an output next to the upper or lower border is not finite
    load(0, in[0]);
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        if (r + 1 < ROWS) load(r + 1, in[(r + 1) & 1]);
#pragma unroll
        for (int kh = 0; kh < 3; ++kh) {
            if ((r - kh) % S != 0 || r < kh || (r - kh) / S >= R) continue;
            const int o = (r - kh) / S;
#pragma unroll
            for (int i = 0; i < TW; ++i) {
                ulonglong2& a = acc[o % 3][i];
                if (kh == 0) a = bias;
#pragma unroll
                for (int kw = 0; kw < 3; ++kw) {
                    fma2(a.x, in[r & 1][i * S + kw].x, wk[kh * 3 + kw].x);
                    fma2(a.y, in[r & 1][i * S + kw].y, wk[kh * 3 + kw].y);
                }
            }
        }
        if (r >= 2 && (r - 2) % S == 0) {
            const int o = (r - 2) / S, oy = oy0 + o;
            float4* out = reinterpret_cast<float4*>(y + (((size_t)n * Ho + oy) * Wo + ox0) * C) + c4;
            if (S == 1 && (oy == 0 || oy * S + 2 > H)) {
                f32x2 probe = 0;
                float lo, hi;
#pragma unroll
                for (int i = 0; i < TW; ++i) {
                    fma2(probe, acc[o % 3][i].x, 0);
                    fma2(probe, acc[o % 3][i].y, 0);
                }
                unpack2(probe, lo, hi);
                again |= !(lo + hi == 0.f);
            }
#pragma unroll
            for (int i = 0; i < TW; ++i) {
                float4 v;
                unpack2(acc[o % 3][i].x, v.x, v.y);
                unpack2(acc[o % 3][i].y, v.z, v.w);
                if (S == 2 && (oy == 0 || oy * S + 2 > H)) again |= !(fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, v.w * 0.f))) == 0.f);
                if (relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
                if (oy < Ho && ox0 + i < Wo) out[(size_t)i * C4] = v;
            }
        }
    }
    // (The kernel is short of registers.  Of the ways to see such outputs these cost least: 64 x 56 x 56 x 128 stays at 43.2 us,
    // 64 x 112 x 112 x 64 at stride 2 goes from 47.0 to 48.0; conditions on the FMAs 46.9 and 50.9, branches around them 55.)
    if (again) dw_rows_inside<S>(w, b, x, y, H, W, C, Ho, Wo, relu, TW, R);
}

template <int S, int TW, int R>
long long slide_blocks(int N, int C, int Ho, int Wo) {
    return ((long long)N * ((Ho + R - 1) / R) * ((Wo + TW - 1) / TW) * (C / 4) + 255) / 256;
}

// ---- first layer: dense 3x3 on a thin input ---------------------------------------------------
// One thread: 4 consecutive output columns x 8 output channels.  Weights sit in shared memory as
// [tap][cin][Cout] so the 8 channels of a thread are two broadcast float4 reads.
template <int S>
__global__ void __launch_bounds__(256)
conv3x3_thin_kernel(const float* __restrict__ w, const float* __restrict__ b, const float* __restrict__ x,
                    float* __restrict__ y, int N, int H, int W, int Cin, int Cout, int Ho, int Wo, int relu) {
    extern __shared__ __align__(16) float ws[];  // [9][Cin][Cout]
    for (int i = threadIdx.x; i < 9 * Cin * Cout; i += blockDim.x) {
        const int o = i % Cout, tc = i / Cout;  // tc = tap*Cin + c
        ws[i] = w[(size_t)o * 9 * Cin + tc];
    }
    __syncthreads();
    constexpr int TW = 4, IW = S * (TW - 1) + 3;
    const int CG = Cout >> 3;
    const int strips = (Wo + TW - 1) / TW;
    const int64_t total = (int64_t)N * Ho * strips * CG;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const int cg = (int)(t % CG);
    int64_t r = t / CG;
    const int sx = (int)(r % strips); r /= strips;
    const int oy = (int)(r % Ho);
    const int n = (int)(r / Ho);
    const int ox0 = sx * TW, ix0 = ox0 * S - 1;

    float acc[TW][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const float bv = b ? __ldg(b + cg * 8 + j) : 0.f;
#pragma unroll
        for (int i = 0; i < TW; ++i) acc[i][j] = bv;
    }
#pragma unroll
    for (int kh = 0; kh < 3; ++kh) {
        const int iy = oy * S + kh - 1;
        if (iy < 0 || iy >= H) continue;
        const float* row = x + ((size_t)n * H + iy) * W * Cin;
        for (int c = 0; c < Cin; ++c) {
            float in[IW];
#pragma unroll
            for (int j = 0; j < IW; ++j) {
                const int ix = ix0 + j;
                in[j] = (ix >= 0 && ix < W) ? __ldg(row + (size_t)ix * Cin + c) : 0.f;
            }
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) {
                const float4* wp = reinterpret_cast<const float4*>(ws + ((kh * 3 + kw) * Cin + c) * Cout + cg * 8);
                const float4 w0 = wp[0], w1 = wp[1];
                const float wv[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
#pragma unroll
                for (int i = 0; i < TW; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(in[i * S + kw], wv[j], acc[i][j]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < TW; ++i) {
        const int ox = ox0 + i;
        if (ox >= Wo) break;
        float4* out = reinterpret_cast<float4*>(y + (((size_t)n * Ho + oy) * Wo + ox) * Cout + cg * 8);
        float v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = relu ? fmaxf(acc[i][j], 0.f) : acc[i][j];
        out[0] = make_float4(v[0], v[1], v[2], v[3]);
        out[1] = make_float4(v[4], v[5], v[6], v[7]);
    }
}

// ---- global average pool ------------------------------------------------------------------
__global__ void __launch_bounds__(256)
avgpool_kernel(const float* __restrict__ x, float* __restrict__ y, int N, int HW, int C) {
    const int C4 = C >> 2;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= N * C4) return;
    const int c4 = t % C4, n = t / C4;
    const float4* p = reinterpret_cast<const float4*>(x + (size_t)n * HW * C) + c4;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int i = 0; i < HW; ++i) {
        const float4 v = __ldg(p + (size_t)i * C4);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    const float inv = 1.0f / (float)HW;
    reinterpret_cast<float4*>(y + (size_t)n * C)[c4] = make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv);
}

}  // namespace
}  // namespace sbnn

using namespace sbnn;

extern "C" sbnn_status sbnn_dwconv3x3(const float* w_dev, const float* b_dev, const float* x_dev, float* y_dev, int N,
                                      int H, int W, int C, int stride, int flags, void* cuda_stream) {
    clear_error();
    if (!w_dev || !x_dev || !y_dev) return fail(SBNN_ERR_NULL, "w_dev, x_dev and y_dev must not be NULL");
    if (N < 0 || H < 0 || W < 0 || C <= 0) return fail(SBNN_ERR_SHAPE, "bad shape N=%d H=%d W=%d C=%d", N, H, W, C);
    if (stride != 1 && stride != 2) return fail(SBNN_ERR_SHAPE, "stride %d: only 1 and 2", stride);
    if (flags & ~SBNN_RELU) return fail(SBNN_ERR_UNSUPPORTED, "unknown flag bits 0x%x", flags);
    if (C % 4) return fail(SBNN_ERR_UNSUPPORTED, "C=%d is not a multiple of 4", C);
    if (!aligned16(w_dev) || !aligned16(x_dev) || !aligned16(y_dev) || (b_dev && !aligned16(b_dev)))
        return fail(SBNN_ERR_ALIGN, "device pointers must be 16-byte aligned");
    if ((int64_t)N * H * W == 0) return SBNN_OK;
    sbnn_status st = check_device();
    if (st != SBNN_OK) return st;
    const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
    constexpr int TW = 4;
    const int64_t total = (int64_t)N * Ho * ((Wo + TW - 1) / TW) * (C / 4);
    const int64_t blocks = (total + 255) / 256;
    if (blocks > 0x7fffffff) return fail(SBNN_ERR_SHAPE, "tensor too large");
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const int relu = flags & SBNN_RELU;
    // Four output rows a thread wherever that still makes two CTAs an SM (9 x 28 x 28 x 256 has half of that and stays at
    // 5.1 us with the kernel that gives every row a thread).
    constexpr int SR1 = 4, SR2 = 4;
    const long long b1 = slide_blocks<1, 3, SR1>(N, C, Ho, Wo), b2 = slide_blocks<2, 2, SR2>(N, C, Ho, Wo);
    if (stride == 1 && b1 >= 2 * device_sms() && b1 <= 0xffffff)
        dwconv3x3_slide_kernel<1, 3, SR1><<<(unsigned)b1, 256, 0, s>>>(w_dev, b_dev, x_dev, y_dev, N, H, W, C, Ho, Wo, relu);
    else if (stride == 2 && b2 >= 2 * device_sms() && b2 <= 0xffffff)
        dwconv3x3_slide_kernel<2, 2, SR2><<<(unsigned)b2, 256, 0, s>>>(w_dev, b_dev, x_dev, y_dev, N, H, W, C, Ho, Wo, relu);
    else {
        const bool wide = blocks <= 2 * device_sms();
        auto* const kernel = stride == 1 ? (wide ? dwconv3x3_kernel<1, TW, true> : dwconv3x3_kernel<1, TW, false>)
                                         : (wide ? dwconv3x3_kernel<2, TW, true> : dwconv3x3_kernel<2, TW, false>);
        kernel<<<(unsigned)blocks, 256, 0, s>>>(w_dev, b_dev, x_dev, y_dev, N, H, W, C, Ho, Wo, relu);
    }
    SBNN_CUDA_TRY(cudaGetLastError());
    return SBNN_OK;
}

extern "C" sbnn_status sbnn_conv3x3_dense(const float* w_dev, const float* b_dev, const float* x_dev, float* y_dev,
                                          int N, int H, int W, int Cin, int Cout, int stride, int flags,
                                          void* cuda_stream) {
    clear_error();
    if (!w_dev || !x_dev || !y_dev) return fail(SBNN_ERR_NULL, "w_dev, x_dev and y_dev must not be NULL");
    if (N < 0 || H < 0 || W < 0 || Cin <= 0 || Cout <= 0) return fail(SBNN_ERR_SHAPE, "bad shape");
    if (stride != 1 && stride != 2) return fail(SBNN_ERR_SHAPE, "stride %d: only 1 and 2", stride);
    if (flags & ~SBNN_RELU) return fail(SBNN_ERR_UNSUPPORTED, "unknown flag bits 0x%x", flags);
    if (Cin > 4 || Cout % 8 || Cout > 64)
        return fail(SBNN_ERR_UNSUPPORTED, "thin-input conv needs Cin <= 4, Cout %% 8 == 0, Cout <= 64 (got %d, %d)", Cin, Cout);
    if (!aligned16(y_dev)) return fail(SBNN_ERR_ALIGN, "y_dev must be 16-byte aligned");
    if ((int64_t)N * H * W == 0) return SBNN_OK;
    sbnn_status st = check_device();
    if (st != SBNN_OK) return st;
    const int Ho = (H - 1) / stride + 1, Wo = (W - 1) / stride + 1;
    const int64_t total = (int64_t)N * Ho * ((Wo + 3) / 4) * (Cout / 8);
    const int64_t blocks = (total + 255) / 256;
    if (blocks > 0x7fffffff) return fail(SBNN_ERR_SHAPE, "tensor too large");
    const size_t smem = sizeof(float) * 9 * Cin * Cout;
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    const int relu = flags & SBNN_RELU;
    if (stride == 1)
        conv3x3_thin_kernel<1><<<(unsigned)blocks, 256, smem, s>>>(w_dev, b_dev, x_dev, y_dev, N, H, W, Cin, Cout, Ho, Wo, relu);
    else
        conv3x3_thin_kernel<2><<<(unsigned)blocks, 256, smem, s>>>(w_dev, b_dev, x_dev, y_dev, N, H, W, Cin, Cout, Ho, Wo, relu);
    SBNN_CUDA_TRY(cudaGetLastError());
    return SBNN_OK;
}

extern "C" sbnn_status sbnn_avgpool(const float* x_dev, float* y_dev, int N, int HW, int C, void* cuda_stream) {
    clear_error();
    if (!x_dev || !y_dev) return fail(SBNN_ERR_NULL, "x_dev and y_dev must not be NULL");
    if (N < 0 || HW <= 0 || C <= 0) return fail(SBNN_ERR_SHAPE, "bad shape N=%d HW=%d C=%d", N, HW, C);
    if (C % 4) return fail(SBNN_ERR_UNSUPPORTED, "C=%d is not a multiple of 4", C);
    if (!aligned16(x_dev) || !aligned16(y_dev)) return fail(SBNN_ERR_ALIGN, "device pointers must be 16-byte aligned");
    if (N == 0) return SBNN_OK;
    sbnn_status st = check_device();
    if (st != SBNN_OK) return st;
    const int total = N * (C / 4);
    avgpool_kernel<<<(total + 255) / 256, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(x_dev, y_dev, N, HW, C);
    SBNN_CUDA_TRY(cudaGetLastError());
    return SBNN_OK;
}
