// Group-sparse 1x1 convolution for launches with few pixels (Algorithm 1 with the loop nest turned round).
//
// The pipelined kernel of conv1x1_cm.cu deals tiles of 256 pixels x 16-24 groups to the SMs; a layer with a
// few hundred pixels (the classifier, every layer of a batch-1 forward) gives it a handful of tiles, and each
// of them walks all of Cin alone.  Here the work is cut the other way: a CTA owns 32 pixels of ONE group, its
// 1-8 warps (more for longer lists) split the group's kept-unit list and add their partial sums through shared memory.
// Lanes are pixels, so an activation row X[c][m0 .. m0+31] is one coalesced 128-byte read straight from the
// channel-major tensor (it stays in L1/L2 for the other groups' CTAs), and the unit's index and its G weights
// are the same address for the whole warp.  No private weight layout: the canonical packed arrays are read.
#include <algorithm>

#include "common.h"
#include "pipeline.cuh"

namespace sbnn {
namespace {


// Index and weights of unit `u` for lane-parallel fetching: lane l of a warp fetches unit u0 + l (two coalesced
// requests for 32 units) and puts them into shared memory, from where the whole warp reads them, so the only per-unit
// access to global memory left is the activation row itself and 16 of those are independent.
// (Handing them round by shuffle, 1 + G for a unit, bound the launch: one pixel, 1024 -> 1000 dense, 10.1 -> 6.8 us; one
// 14 x 14 image, 512 -> 512 at 50 %, G = 4 13 -> 7.5 us, 3 x 2 x 2 pixels, G = 8 4.0 -> 2.8.)
template <int G>
struct UnitRegs {
    int c;
    float w[G];
};

template <int G>
__device__ __forceinline__ void fetch_unit(const int32_t* __restrict__ idx, const float* __restrict__ val, int u, int uend,
                                           UnitRegs<G>& r) {
    const bool ok = u < uend;
    r.c = ok ? ld_early(idx + u) : 0;
    const float* p = val + (size_t)(ok ? u : 0) * G;
    if constexpr (G % 4 == 0) {
#pragma unroll
        for (int q = 0; q < G / 4; ++q) {
            const float4 t = ld_early(reinterpret_cast<const float4*>(p) + q);
            r.w[4 * q] = t.x; r.w[4 * q + 1] = t.y; r.w[4 * q + 2] = t.z; r.w[4 * q + 3] = t.w;
        }
    } else if constexpr (G == 2) {
        const float2 t = ld_early(reinterpret_cast<const float2*>(p));
        r.w[0] = t.x; r.w[1] = t.y;
    } else {
        r.w[0] = ld_early(p);
    }
    if (!ok) {
#pragma unroll
        for (int q = 0; q < G; ++q) r.w[q] = 0.0f;                 // units past the end multiply pixel row 0 by zero
    }
}

// KSPLIT = warps per CTA; each takes that fraction of the group's kept units.  PX = pixels per lane (the CTA covers
// 32 * PX pixels): with two, a unit's index and weights, once read from shared memory, serve twice the FMAs.
// WIDE (eight warps): one CTA an SM is stated to be enough; the compiler then takes more registers (G = 4: 96 instead of 64, with two
// pixels 104 instead of 79) and has more of a round's loads in flight, but fewer CTAs are resident, see wide_limit.  With four warps it
// costs more than it gains at any size (14 x 14, 256 -> 512 at 50 %: 4.6 -> 5.1 us).  Sixteen warps are no faster than eight (1 pixel,
// 1024 -> 1000: 6.9 and 6.6).
template <int G, int KSPLIT, bool OUT_CM, int PX, bool WIDE>
__global__ void __launch_bounds__(32 * KSPLIT, WIDE ? 1 : 0)
conv1x1_small_kernel(const float* __restrict__ X, int ldx, float* __restrict__ Y, int ldy, const int32_t* __restrict__ group_ptr,
                     const int32_t* __restrict__ idx, const float* __restrict__ val, const float* __restrict__ bias, int M,
                     int relu) {
    __shared__ float red[KSPLIT][G][32 * PX];
    __shared__ __align__(16) float wsm[KSPLIT][32 * G];
    __shared__ __align__(16) int csm[KSPLIT][32];
    const int lane = threadIdx.x & 31, kq = threadIdx.x >> 5;
    const int g = blockIdx.y;
    int m[PX];
    const float* xp[PX];
#pragma unroll
    for (int j = 0; j < PX; ++j) {
        m[j] = (blockIdx.x * PX + j) * 32 + lane;
        xp[j] = X + (m[j] < M ? m[j] : M - 1);                     // lanes past the end read a valid pixel, store nothing
    }
    const int beg = ld_early(group_ptr + g), n = ld_early(group_ptr + g + 1) - beg;
    const int per = (n + KSPLIT - 1) / KSPLIT;
    const int u0 = beg + min(n, kq * per), uend = beg + min(n, (kq + 1) * per);
    float acc[PX][G];
#pragma unroll
    for (int j = 0; j < PX; ++j)
#pragma unroll
        for (int r = 0; r < G; ++r) acc[j][r] = 0.0f;
    UnitRegs<G> cur, nxt;
    fetch_unit<G>(idx, val, u0 + lane, uend, cur);
    grid_dependency_wait();      // X comes from the previous kernel of the stream; the weights above do not
    grid_dependency_release();
    for (int ub = u0; ub < uend; ub += 32) {
        csm[kq][lane] = cur.c;
#pragma unroll
        for (int r = 0; r < G; ++r) wsm[kq][lane * G + r] = cur.w[r];
        __syncwarp();
        fetch_unit<G>(idx, val, ub + 32 + lane, uend, nxt);        // the next 32 units, while these are consumed
        const int cnt = min(32, uend - ub);                        // warp-uniform
#pragma unroll
        for (int h = 0; h < 2; ++h) {                              // 16 * PX activation loads in flight per lane
            if (h * 16 >= cnt) break;
            float xv[PX][16];
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) {
                const int4 c4 = reinterpret_cast<const int4*>(csm[kq])[h * 4 + k4];
                const int c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                for (int e = 0; e < 4; ++e)
#pragma unroll
                    for (int j = 0; j < PX; ++j) xv[j][k4 * 4 + e] = (h * 16 + k4 * 4 + e < cnt) ? __ldg(xp[j] + (size_t)c[e] * ldx) : 0.0f;
            }
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                float w[G];
                const float* wp = wsm[kq] + (h * 16 + k) * G;
                if constexpr (G % 4 == 0) {
#pragma unroll
                    for (int q = 0; q < G / 4; ++q) {
                        const float4 t = reinterpret_cast<const float4*>(wp)[q];
                        w[4 * q] = t.x; w[4 * q + 1] = t.y; w[4 * q + 2] = t.z; w[4 * q + 3] = t.w;
                    }
                } else {
#pragma unroll
                    for (int r = 0; r < G; ++r) w[r] = wp[r];
                }
#pragma unroll
                for (int r = 0; r < G; ++r)
#pragma unroll
                    for (int j = 0; j < PX; ++j) acc[j][r] = fmaf(xv[j][k], w[r], acc[j][r]);
            }
        }
        __syncwarp();                                              // before the next units take their place
        cur = nxt;
    }
#pragma unroll
    for (int j = 0; j < PX; ++j)
#pragma unroll
        for (int r = 0; r < G; ++r) red[kq][r][j * 32 + lane] = acc[j][r];
    __syncthreads();
    if (kq != 0) return;
#pragma unroll
    for (int j = 0; j < PX; ++j) {
        if (m[j] >= M) continue;
        float v[G];
#pragma unroll
        for (int r = 0; r < G; ++r) {
            float s = red[0][r][j * 32 + lane];
#pragma unroll
            for (int q = 1; q < KSPLIT; ++q) s += red[q][r][j * 32 + lane];
            s += __ldg(bias + g * G + r);
            v[r] = relu ? fmaxf(s, 0.0f) : s;
        }
        if constexpr (OUT_CM) {
#pragma unroll
            for (int r = 0; r < G; ++r) Y[(size_t)(g * G + r) * ldy + m[j]] = v[r];
        } else {
            float* yp = Y + (size_t)m[j] * ldy + g * G;
            if constexpr (G >= 4) {
#pragma unroll
                for (int q = 0; q < G / 4; ++q)
                    reinterpret_cast<float4*>(yp)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            } else if constexpr (G == 2) {
                *reinterpret_cast<float2*>(yp) = make_float2(v[0], v[1]);
            } else {
                yp[0] = v[0];
            }
        }
    }
}

// CTAs an SM up to which a launch of eight warps takes the WIDE instance.  Measured without and with it, us: G = 4, two pixels a lane,
// 1024 -> 1024 at 50 %: 256 CTAs 8.4 and 5.9, 512 11.4 and 11.0, 1792 31.7 and 32.1; 512 -> 512 at 50 %: 256 CTAs 4.9 and 3.8, 1280 13.5
// and 14.3; one pixel: 128 CTAs 2.2 and 2.1, 256 4.0 and 4.1, 512 (1024 -> 2048) 6.5 and 7.4 (but the network, whose classifier is a
// launch of 250 behind another, takes 120.6 us on one image at 30 % without and 117.7 with it).  G = 2, 1024 -> 256 at 50 %: one pixel,
// 128 CTAs 3.2 and 2.8; two pixels, 256 CTAs 7.0 and 5.3, 896 14.5 and 15.7; 512 -> 512, one pixel, 256 CTAs 3.4 and 4.2.  G = 1, 512 ->
// 512 at 50 %: one pixel, 512 CTAs 3.7 and 3.3, two pixels, 5.2 and 5.8, 1024 CTAs 8.6 and 10.1.  G = 8 gains 1 to 4 % up to 832 CTAs
// (1024 -> 2048, one pixel: 7.0 and 5.7) and loses up to 6 % above; G = 16 gains 0 to 10 % everywhere.
template <int G, int PX>
constexpr long long wide_limit() {
    if (G == 8) return 6;
    if (PX == 2) return G == 4 ? 4 : 2;
    return G == 1 ? 4 : (G == 4 ? 2 : 1);
}

template <int G, int KS, int PX, bool WIDE>
sbnn_status launch_small_as(const sbnn_packed* p, dim3 grid, const float* x, int ldx, float* y, int ldy, int M, int relu, bool out_cm,
                            cudaStream_t st) {
    ChainedLaunchScope early;   // before its wait the kernel reads the layer's own arrays only
    auto* const kernel = out_cm ? conv1x1_small_kernel<G, KS, true, PX, WIDE> : conv1x1_small_kernel<G, KS, false, PX, WIDE>;
    SBNN_CUDA_TRY(launch_kernel(kernel, grid, 32 * KS, 0, st, x, ldx, y, ldy, p->d_group_ptr, p->d_idx, p->d_val, p->d_bias, M, relu));
    return SBNN_OK;
}
template <int G, int KS, int PX>
sbnn_status launch_small_ks(const sbnn_packed* p, const float* x, int ldx, float* y, int ldy, int M, int relu, bool out_cm,
                            cudaStream_t st) {
    const dim3 grid((unsigned)((M + 32 * PX - 1) / (32 * PX)), (unsigned)p->ngroups);
    if constexpr (KS == 8 && G == 16) {
        return launch_small_as<G, KS, PX, true>(p, grid, x, ldx, y, ldy, M, relu, out_cm, st);
    } else {
        if constexpr (KS == 8) {
            if ((long long)grid.x * grid.y <= wide_limit<G, PX>() * device_sms())
                return launch_small_as<G, KS, PX, true>(p, grid, x, ldx, y, ldy, M, relu, out_cm, st);
        }
        return launch_small_as<G, KS, PX, false>(p, grid, x, ldx, y, ldy, M, relu, out_cm, st);
    }
}

// Warps of a CTA and pixels of a lane.  Long lists are split over more warps (shorter dependent chains); short ones are not worth the
// reduction.  Long lists and more than one 32-pixel block: two pixels per lane halve the reads of weights per FMA (classifier at batch 64
// when the weights still came by shuffle: 18.3 -> 14.9 us inside the step); groups of 16 channels would need 32 more accumulators
// and stay with one.
struct SmallShape {
    int warps, px;
};
SmallShape small_shape(const sbnn_packed* p, long long M) {
    const long long avg = p->ngroups ? p->nnz / p->ngroups : 0;
    if (avg >= 256) return {8, M > 32 && p->G <= 8 ? 2 : 1};
    return {avg >= 96 ? 4 : (avg >= 40 ? 2 : 1), 1};
}

template <int G>
sbnn_status launch_small(const sbnn_packed* p, const float* x, int ldx, float* y, int ldy, int M, int relu, bool out_cm,
                         cudaStream_t st) {
    const SmallShape s = small_shape(p, M);
    if constexpr (G <= 8)
        if (s.px == 2) return launch_small_ks<G, 8, 2>(p, x, ldx, y, ldy, M, relu, out_cm, st);
    if (s.warps == 8) return launch_small_ks<G, 8, 1>(p, x, ldx, y, ldy, M, relu, out_cm, st);
    if (s.warps == 4) return launch_small_ks<G, 4, 1>(p, x, ldx, y, ldy, M, relu, out_cm, st);
    if (s.warps == 2) return launch_small_ks<G, 2, 1>(p, x, ldx, y, ldy, M, relu, out_cm, st);
    return launch_small_ks<G, 1, 1>(p, x, ldx, y, ldy, M, relu, out_cm, st);
}

}  // namespace

sbnn_status conv1x1_small(const sbnn_packed* p, const float* x, int ldx, float* y, int ldy, int M, int relu, bool out_cm,
                          cudaStream_t st) {
    if (p->ngroups > 65535) return fail(SBNN_ERR_SHAPE, "too many groups for the few-pixel kernel");
    if (prepare_only()) return SBNN_OK;   // reads the canonical arrays: nothing to build
    switch (p->G) {
        case 1: return launch_small<1>(p, x, ldx, y, ldy, M, relu, out_cm, st);
        case 2: return launch_small<2>(p, x, ldx, y, ldy, M, relu, out_cm, st);
        case 4: return launch_small<4>(p, x, ldx, y, ldy, M, relu, out_cm, st);
        case 8: return launch_small<8>(p, x, ldx, y, ldy, M, relu, out_cm, st);
        default: return launch_small<16>(p, x, ldx, y, ldy, M, relu, out_cm, st);
    }
}

// Microseconds a call takes: a fixed part, a warp's chain of kept units, and for every round of CTAs over the SMs, how many of them
// an SM works through, their units and their warps.  Fitted to 2472 calls of random sizes (1 to 3200 pixels, 32 to 2048 channels in, 16
// to 1536 out, all group sizes, dense to 90 % pruned): 90 % of them are within 17 % below and 15 % above what was measured.  With more
// than 64 pixels a call takes no less than 0.19 us (0.138 in groups of 8 and 16) for a million multiply-adds of whole blocks of 32
// pixels: without that limit ten calls of 4924 left the tensor cores, eight of which are 17 % slower here on average.
double conv1x1_small_us(const sbnn_packed* p, long long M) {
    static constexpr double cost[5][3][4] = {   // G = 1, 2, 4, 8, 16; fewer than eight warps, eight, eight with two pixels a lane
        {{1.19, 0.016, 0.017, 0.076}, {0.66, 0.018, 0.035, 0.045}, {1.48, 0.007, 0.086, 0.043}},
        {{1.16, 0.015, 0.011, 0.090}, {1.24, 0.010, 0.057, 0.017}, {1.44, 0.009, 0.101, 0.039}},
        {{1.15, 0.019, 0.038, 0.080}, {0.89, 0.014, 0.054, 0.060}, {1.14, 0.010, 0.117, 0.071}},
        {{1.45, 0.021, 0.073, 0.102}, {0.97, 0.019, 0.067, 0.108}, {1.46, 0.010, 0.169, 0.111}},
        {{1.76, 0.047, 0.079, 0.123}, {0.79, 0.034, 0.115, 0.174}, {0.79, 0.034, 0.115, 0.174}}};
    const SmallShape s = small_shape(p, M);
    const double* const c = cost[p->G == 1 ? 0 : p->G == 2 ? 1 : p->G == 4 ? 2 : p->G == 8 ? 3 : 4][s.px == 2 ? 2 : s.warps == 8];
    const long long ctas = (M + 32 * s.px - 1) / (32 * s.px) * p->ngroups, sms = std::max(1, device_sms());
    const double units = p->ngroups ? (double)p->nnz / p->ngroups : 0.0, rounds = (double)((ctas + sms - 1) / sms);
    const double us = c[0] + c[1] * units / s.warps + rounds * (c[2] * units / 32 + c[3] * s.warps);
    const double macs = 1e-6 * (double)((M + 31) / 32 * 32) * p->nnz * p->G;
    return M > 64 ? std::max(us, 1.7 + macs * (p->G >= 8 ? 0.138 : 0.19)) : us;
}

}  // namespace sbnn
