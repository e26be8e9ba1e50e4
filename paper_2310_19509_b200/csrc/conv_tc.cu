// Group-sparse convolutions in fp32 on the 5th-generation tensor cores (tcgen05), 1x1 and 3x3.
//
//   Y[m][o] = act( bias[o] + sum_{t,c} W~[o][t][c] * X[pixel(m) + tap t][c] ),   W~ = W (.) M  (Section 3.1)
//
// Precision: fp32 operands, fp32 result.  Every fp32 number is the exact sum of three bf16 numbers (8 + 8 + 8
// significand bits), x = xh + xm + xl, w = wh + wm + wl, and the product of two bf16 numbers is exact in fp32.  The
// kernel adds the six products xl*wh, xh*wl, xm*wm, xm*wh, xh*wm, xh*wh; the three that are left out (m*l, l*m, l*l) are
// together below 2^-25 |x*w|, because every image is rounded to nearest (|m| <= 2^-9, |l| <= 2^-18 of the number).
// The tensor core truncates when it adds to its accumulator, so no long sum is left to it: a 64-channel step is summed in
// a fresh accumulator, the five small products first, and added to the running sum in registers, rounded to nearest.
// What the truncations of one step take from the magnitude of its sum on average, 5.4e-8 of it (measured for 64 to
// 1024 channels, dense to 90 % pruned, 1x1 and 3x3, alone and in a network: 3.6e-8 to 5.9e-8), is put back in the weights,
// which are scaled by kTruncation before they are split; without it the layers of a network lose the same fraction one
// after the other.  What remains is -0.6e-8 to 1.0e-8 for 64 to 1024 channels and up to 1.6e-8 for 4 to 48, whose steps are
// half as long, against 3e-8 to 9e-8 of rounding.
// Small operands: bf16 ends at 2^-133, so the third image of a number below 2^-109 loses bits, and a number below 2^-133 is
// lost: an output is then off by up to 2^-133 times the other operands (the FMA kernels: 2^-149).
//
// The contraction runs dense over the masked weights (pruned entries are zeros): a group shares its kept channels over
// only G = 4..8 outputs, far too few for a 128-row MMA to gather for.  Six products per dense MAC still beat the FMA
// pipe on kept MACs alone until most of the layer is pruned; the rule is decide() below.
//
// Structure, one CTA per SM, persistent over tiles of 128 pixels x BN output channels, 20 warps in 5 warpgroups:
//   warpgroups 0, 1  drain: tcgen05.ld of a finished step, added to the fp32 sums in registers, which start at the bias;
//                    after the last step ReLU and stores;
//   warpgroups 2, 3  split: a thread owns one pixel and 16 of the 32 channels of a staged fp32 tile, splits them and
//                    writes the three bf16 images into tensor memory, where the MMAs read them as the A operand
//                    (so either activation layout is read with conflict-free loads and nothing is transposed);
//   warp 16          copies activations (tiled or im2col tensor-map copies of 32 channels x 128 pixels);
//   warp 17          copies weights (one linear copy per step and 128 output channels: the three bf16 images,
//                    stored in the swizzled order the MMA reads);
//   warps 18, 19     issue the MMAs, each into an accumulator of its own: while one waits for its operands the other's MMAs run.
// (With one issuing warp the waits between its batches of 24 MMAs, 740 cycles, came on top of the 1900 cycles a batch
// takes; with one split warpgroup a step took 1300 cycles to split, as long as its MMAs.)
// Every wait is bounded, as in the other pipelined kernels.
//
// The bf16 mode (SBNN_BF16_TC: activations and weights rounded to bf16 once, fp32 sums) is the same kernel with one image
// of each operand (IMAGES = 1): one product, summed over all steps of a tile in the accumulator and drained once.
//
// A launch can do the depthwise 3x3 layer in front of a 1x1 layer as well (SRC_DW, see DwShape), whose output then never reaches
// memory: the split warps compute it from the staged input, in fp32, and split it.
//
// Launches with too few tiles for the SMs (small batches, small maps) run with 64 output channels a tile and the steps of a
// tile dealt to the CTAs of a cluster (SPLIT): each sums its share, then every CTA adds up a part of the channels, which
// the others have written into its shared memory, in rank order, and stores it.
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <new>
#include <type_traits>

#include <cuda.h>   // CUtensorMap (type only)

#include "common.h"
#include "pipeline.cuh"
#include "tcgen05.cuh"

namespace sbnn {
namespace {

constexpr double kTruncation = 1.0 + 5.4e-8;

// SRC_CM3: 3x3 on channel-major activations.  A tap shifts the 128 pixels of a tile by dy * W + dx, so a copy of 136 pixels
// (from a multiple of 4) serves the three taps of a kernel row; the split warps blank what lies outside the image.
// SRC_DW: 1x1 on the result of a depthwise 3x3 (stride 1 or 2, bias, ReLU) of channel-major square images, which the split
// warps compute on the way (see DwShape).
enum Source { SRC_NHWC, SRC_CM, SRC_IM2COL, SRC_CM3, SRC_DW };

// Element strides of the activations and the arrays of the packed layer, for the outputs of pixels that hold a
// non-finite value (see sum_kept_units).
struct ExactArgs {
    const float* x;
    long long pixel_stride, channel_stride;
    const int32_t* group_ptr;
    const int32_t* idx;
    const float* val;
    const uint16_t* taps;  // of the kept units, where the FMA kernels leave pruned taps out; else NULL
    int G;
};

struct TcArgs {
    const uint4* wts;      // [output tile of NUC][step][image][NUC rows][64] bf16, swizzled
    const float* bias;
    float* y;
    int ldy;
    int M, Cin, Cout;
    int steps;             // 64-channel steps x taps (taps inner)
    int ntiles_m, ntiles_n;
    int dm, dn;            // a CTA's next tile: dm pixel tiles and dn channel tiles further (grid size divided by ntiles_n)
    int W, H;              // image size (3x3 only)
    int relu;
    int split;             // CTAs of a cluster that share a tile's steps
    int sa, sb;            // stages of activations and of weights
    // Not shared: whether every tile uses the same weights and all of them have a stage, so that they are loaded once.  Shared: a CTA's part
    // of a drain thread's chunks of outputs, in units of 2^-16 and rounded up (see store_shared_tile).  (One word for both: with eight
    // bytes more of arguments a launch takes the host 0.4 us longer, 4.5 -> 4.9.)
    int resident_or_share;
    int* status;
    ExactArgs ex;
};
static_assert(sizeof(TcArgs) == 160, "arguments of a launch");
struct DwArgs : TcArgs {
    CUtensorMap wmap;      // the depthwise weights [9][Cin]
    const float* dw_w;
    const float* dw_b;
};

// What a stage holds for the depthwise layer in front of a 1x1 layer (SRC_DW), for images of WI x WI input pixels, 112 to 28: of
// SUB channels every input pixel that the 128 output pixels of a tile need, as BOXES tiled copies of PB consecutive pixels each
// (box-major, then channel, then pixel), behind them the nine rows of weights and the bias of these channels.
// Stride 1: the 128 pixels and a row and a pixel more on both sides are one run, except for 112 pixels a row, where a box
// holds the run of one kernel row (three of 140 pixels; one run, in two boxes, would be 360).
// Stride 2: the input rows of the output rows that the tile touches, BR rows to a box.
// A box has LEAD pixels in front of the tile's, so that it starts at a multiple of 4 pixels and four pixels of a row at one; PB / 4
// is odd, so that 16-byte loads of 8 channels fall into different banks.
constexpr int kMaxDwChannels = 1024;
template <int WI_, int S_>
struct DwShape {
    static constexpr int WI = WI_, S = S_, WO = WI / S, SUB = S == 1 ? 16 : 8;
    static constexpr bool ROWS3 = S == 1 && WI == 112;
    static constexpr int BR = WI == 112 ? 1 : 2;         // (stride 2)
    static constexpr int LEAD = S == 2 ? 0 : (ROWS3 ? 4 : WI + 4);
    static constexpr int RUN = S == 2 ? BR * WI : (ROWS3 ? 133 : 128 + WI + 1 + LEAD);
    static constexpr int PB = (RUN + 3) / 4 * 4 + ((RUN + 3) / 4 % 2 ? 0 : 4);
    static constexpr int BOXES = S == 2 ? (2 * ((126 + WO) / WO) + 3 + BR - 1) / BR : (ROWS3 ? 3 : 1);
    static constexpr int BOX = SUB * PB;                 // floats
    static constexpr int X_BYTES = BOXES * BOX * 4, COPIED = X_BYTES + 10 * SUB * 4, STAGE = (COPIED + 127) / 128 * 128;
    // The depthwise output of a stage on its way from lanes that own channels to lanes that own pixels, of each split warpgroup.
    static constexpr int PITCH = 132, OUTPUT = 2 * SUB * PITCH * 4;
    static constexpr int ZEROS = 16;                     // what is read outside the image
    static_assert(WI % 4 == 0 && WO % 4 == 0 && PB <= 256 && PB / 4 % 2 == 1 && BOX * 4 % 128 == 0, "boxes");
};
template <>
struct DwShape<0, 1> {
    static constexpr int SUB = 32, COPIED = 0, STAGE = 0, OUTPUT = 0, ZEROS = 0, S = 1;
};

template <int BN_, int SRC_, bool OUT_CM_, bool SPLIT_ = false, int IMAGES_ = 3, int WI_ = 0, int STRIDE_ = 1>
struct TC {
    static constexpr int BM = 128, BN = BN_, BK = 64, SRC = SRC_;
    static constexpr bool FUSED = SRC == SRC_DW;
    using DW = DwShape<WI_, STRIDE_>;
    using Args = std::conditional_t<FUSED, DwArgs, TcArgs>;
    static constexpr bool OUT_CM = OUT_CM_, SPLIT = SPLIT_;
    static constexpr int IMAGES = IMAGES_;
    static constexpr int TAPS = SRC == SRC_IM2COL || SRC == SRC_CM3 ? 9 : 1;
    static constexpr int RUN = SRC == SRC_CM3 ? 3 : 1;   // steps that read the same activation stages
    static constexpr int PIX = SRC == SRC_CM3 ? 136 : 128;   // pixels of a stage
    static constexpr int NUC = BN < 128 ? BN : 128;      // columns of one MMA
    static constexpr int NU = BN / NUC;                  // MMA column blocks per tile
    static constexpr int SUB = DW::SUB;                  // channels of one activation stage
    static constexpr int A_COPIED = FUSED ? DW::COPIED : SUB * PIX * 4, A_BYTES = FUSED ? DW::STAGE : A_COPIED;
    static constexpr int B_BYTES = IMAGES * NUC * BK * 2;
    static constexpr int OUT_TILES = DW::S == 2 ? 1 : 2;      // staging tiles of 32 pixels x 16 channels for each drain warp
    static constexpr int OUT_BYTES = 8 * OUT_TILES * 2048;
    static constexpr int CTRL = 512;                     // mbarriers, tensor-memory base, abort flag; zeros for SRC_DW
    // Stages share what is left of 227 KB: weights that fit as a whole and serve every tile stay (see launch_tc), else
    // SB stages of them; the rest goes to activations, up to SA_MAX stages.
    static constexpr int SB = IMAGES == 1 ? 6 : (BN < 128 ? (WI_ == 112 ? 2 : 4) : (WI_ == 112 ? 1 : (SRC == SRC_CM3 || FUSED ? 2 : 3))), SA_MAX = 12, SB_MAX = 6;
    static constexpr int ROOM = 227 * 1024 - 1024 - CTRL - OUT_BYTES - DW::OUTPUT;
    static constexpr int SA_MIN = SRC == SRC_CM3 || FUSED ? 4 : 3;
    static_assert((2 * SA_MAX + 3 * SB_MAX + 12) * 8 + 8 + 16 + DW::ZEROS <= CTRL && SB * B_BYTES + SA_MIN * A_BYTES <= ROOM, "shared memory");
    static constexpr int NT = 640;
    // registers a thread of the drain, split and remaining warps: 2 x + 2 y + z = 5 x 96, what the launch reserves
    static constexpr int LAUNCH_REGS = 96, DRAIN_REGS = BN == 256 ? 160 : 128, SPLIT_REGS = BN == 256 ? 56 : 80, AUX_REGS = BN == 256 ? 48 : 64;
    static_assert(2 * DRAIN_REGS + 2 * SPLIT_REGS + AUX_REGS == 5 * LAUNCH_REGS, "register shares");
    static constexpr int COLS = BN / 2;                  // output channels a drain thread sums
    static constexpr int DEMPTY = NU == 2 ? 4 : 8;       // warps that drain one accumulator
    // tensor-memory columns: two accumulators, behind them NA stages of A images
    static constexpr int D_COLS = NUC, A_COL0 = 2 * D_COLS, A_COLS = 32 * IMAGES, NA = BN == 64 || IMAGES == 1 ? 4 : 2;
    static_assert(A_COL0 + NA * A_COLS <= 512, "tensor memory");
    static_assert(BN == 64 || BN == 128 || BN == 256, "tile width");
    // (shared by 7, the most for an exchange: 7 senders of up to 2 of a thread's 8 chunks)
    static_assert(!SPLIT || (BN == 64 && SB * B_BYTES + SA_MIN * A_BYTES >= 7 * 2 * 256 * 16), "the cluster's exchange");
    static_assert(IMAGES == 3 || (IMAGES == 1 && SRC == SRC_NHWC), "bf16 mode");
    // Pixels that are summed again: the sums of 32 of them fit the staging tiles, or the stages hold all of their channels at once (see
    // sum_kept_units).
    static_assert(BN * 32 * 4 <= OUT_BYTES || (FUSED && SB * B_BYTES + SA_MIN * A_BYTES >= kMaxDwChannels * 32 * 4 + 6144), "sums of bad pixels");
};

__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t join2(uint32_t lo, uint32_t hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
    return r;
}
// (first, second) -> two bf16, rounded to nearest even, the first in the lower half.
__device__ __forceinline__ uint32_t bf16x2(float first, float second) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(second), "f"(first));
    return r;
}

// Splits two fp32 values into bf16 images packed as (first, second): x = h + m + l exactly, down to 2^-109 (see above).
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint32_t bf16_of(uint64_t x) {
    float first, second;
    unpack2(x, first, second);
    return bf16x2(first, second);
}
__device__ __forceinline__ uint64_t widen(uint32_t b) { return join2(b << 16, b & 0xffff0000u); }
__device__ __forceinline__ void split2(uint64_t x, uint32_t& h, uint32_t& m, uint32_t& l) {
    h = bf16_of(x);
    const uint64_t r = sub2(x, widen(h));
    m = bf16_of(r);
    l = bf16_of(sub2(r, widen(m)));
}
__device__ __forceinline__ void load_shared(uint32_t addr, uint64_t& a, uint64_t& b) {
    asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr) : "memory");
}

// Position in a ring of `n` stages: the stage, and the parity of its current use.
struct Ring {
    int n, stage = 0, uses = 0;
    uint32_t parity = 0;
    __device__ explicit Ring(int stages) : n(stages) {}
    __device__ bool reused() const { return uses > 0; }
    __device__ void next() {
        if (++stage == n) {
            stage = 0;
            parity ^= 1;
            ++uses;
        }
    }
    // The weight stages have two "full" barriers each, used in turn.  With an odd number of stages the two MMA warps take
    // turns at a stage; a barrier for every second use is one that only the same warp waits for, once in each of its
    // phases (the parity of a barrier that others complete in between would not tell its phases apart).
    __device__ int turn() const { return stage + (uses & 1 ? n : 0); }
    __device__ uint32_t turn_parity() const { return uses >> 1 & 1; }
    // A producer that gives up at `stage` lets the copies it has issued land before the shared memory is released.
    __device__ void settle(uint64_t* full, bool turns) const {
        for (int s = 0; s < (uses ? n : stage); ++s) {
            const int use = s < stage ? uses : uses - 1;
            bool landed = false;
            for (uint32_t i = 0; i < kWaitLimit && !landed; ++i)
                landed = mbar_try_wait(full + s + (turns && (use & 1) ? n : 0), (turns ? use >> 1 : use) & 1);
        }
    }
};

// The tiles of a CTA: every gridDim.x-th, channel tiles innermost (a cluster that shares a tile has just that one).
struct Tiles {
    const TcArgs& a;
    int m, n;
    __device__ explicit Tiles(const TcArgs& args) : a(args), m(blockIdx.x / args.split / args.ntiles_n), n(blockIdx.x / args.split % args.ntiles_n) {}
    __device__ bool left() const { return m < a.ntiles_m; }
    __device__ void next() {
        m += a.dm;
        n += a.dn;
        if (n >= a.ntiles_n) {
            n -= a.ntiles_n;
            ++m;
        }
    }
};

// All threads of the cluster: what any of them wrote before, to whose shared memory ever, is visible to all after.
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Stores 16 bytes at the address that `addr` has in the shared memory of CTA `rank` of the cluster.
__device__ __forceinline__ void store_remote(uint32_t addr, uint32_t rank, float4 v) {
    asm volatile(
        "{\n\t.reg .b32 r;\n\t"
        "mapa.shared::cluster.u32 r, %0, %1;\n\t"
        "st.shared::cluster.v4.f32 [r], {%2, %3, %4, %5};\n\t}"
        ::"r"(addr), "r"(rank), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
        : "memory");
}

template <int REGS>
__device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS)); }
template <int REGS>
__device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS)); }

// Box of 128 consecutive output positions x 32 channels of the input shifted by (dx, dy): an im2col tensor map walks the
// positions in (x, y, n) order and delivers zeros outside the image.
__device__ __forceinline__ void im2col_g2s(void* dst_smem, const void* map, int c, int x, int y, int n, int dx, int dy, uint64_t* bar) {
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6], {%7, %8};"
                 ::"r"(smem_u32(dst_smem)), "l"(map), "r"(c), "r"(x), "r"(y), "r"(n), "r"(smem_u32(bar)), "h"((short)dx), "h"((short)dy)
                 : "memory");
}

// The 256 drain threads: a barrier among them, and whether any of them says so.
__device__ __forceinline__ bool drain_any(bool mine) {
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "barrier.cta.red.or.pred q, 1, 256, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)mine)
        : "memory");
    return r != 0;
}

// One output of the depthwise layer in front (SRC_DW), straight from global memory: for the few pixels that are summed again.
template <class T>
__device__ __noinline__ float depthwise_output(const DwArgs& a, int m, int c) {
    constexpr int WI = T::DW::WI, WO = T::DW::WO, S = T::DW::S;
    const int x = m % WO, f = m / WO, y = f % WO;
    const float* const from = a.ex.x + c * a.ex.channel_stride + ((long long)f * S - 1) * WI + x * S - 1;
    float sum = a.dw_b[c];
    for (int t = 0; t < 9; ++t) {
        const int iy = y * S + t / 3 - 1, ix = x * S + t % 3 - 1;
        const float v = (unsigned)iy < (unsigned)WI && (unsigned)ix < (unsigned)WI ? from[t / 3 * WI + t % 3] : 0.0f;
        sum = fmaf(v, a.dw_w[t * a.Cin + c], sum);
    }
    return fmaxf(sum, 0.0f);
}

// All drain threads: sums pixels of the tile that starts at m0 once more, as fp32 FMAs over the kept units.  A pixel with an
// infinity or a NaN in any channel spoils all its split products (0 * inf), also those of pruned weights, which must not see
// it; and sums near the end of the fp32 range may overflow here but not product after product with the bias last, as on the FMA kernels.  `bad` says which of the pixels m0 + 32 * q + lane (q = the warp's place in its warpgroup); a warpgroup wg has `len`
// outputs from n0 + wg * T::COLS on.
// Up to 32 pixels at a time go into shared memory, a row for every (channel, tap), and PS lanes of a warp take a pixel each,
// the others share its units; a warp takes four outputs at a time.  Sums that span several stages of rows wait in `sums`.
// Bound by the latency of the reads of 8 warps.  6 x 25 x 31, 1024 -> 516, half pruned, with three bad pixels: 89 us (a thread
// a pixel, in the middle of the tile loop: 2800; the FMA kernels: 89); with a bad channel in every pixel: 372 us (9600; 88), or
// 2500 with the activations read from global memory.
template <class T>
__device__ __noinline__ void sum_kept_units(const typename T::Args& args, unsigned char* room, float* sums, int m0, bool bad, int n0, int len) {
    const ExactArgs e = args.ex;
    const int W = args.W, H = args.H, Cin = args.Cin, Cout = args.Cout, relu = args.relu, ldy = args.ldy;
    float* const y = args.y;
    const float* const bias = args.bias;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, width = e.G < 4 ? e.G : 4;
    constexpr bool CM = T::SRC == SRC_CM || T::SRC == SRC_CM3 || T::FUSED;
    uint32_t* const found = reinterpret_cast<uint32_t*>(room);
    int* const list = reinterpret_cast<int*>(room + 64);
    int* const where = reinterpret_cast<int*>(room + 1024) + warp * 32;        // 32 (unit, tap) pairs of a warp: place of the row,
    float4* const weight = reinterpret_cast<float4*>(room + 2048) + warp * 32;  // and the weights of its four outputs
    float* const rows = reinterpret_cast<float*>(room + 6144);
    const int capacity = (args.sb * T::B_BYTES + args.sa * T::A_BYTES - 6144) / 4;

    drain_any(false);                                          // nobody still uses the room
    if (tid < 4) found[tid] = 0;
    drain_any(false);
    const uint32_t mine = __ballot_sync(0xffffffffu, bad);
    if (lane == 0 && mine) atomicOr(found + (warp & 3), mine);
    drain_any(false);
    int count = 0;
    for (int q = 0; q < 4; ++q) {
        const uint32_t word = found[q];
        if (warp == 0 && (word >> lane & 1)) list[count + __popc(word & ((1u << lane) - 1))] = m0 + q * 32 + lane;
        count += __popc(word);
    }
    for (int first = 0; first < count; first += 32) {
        const int pixels = min(32, count - first);
        int PS = 1;
        while (PS < pixels) PS *= 2;
        const int p = lane & (PS - 1), us = 32 / PS, u = lane / PS;
        const int stage = capacity / PS / T::TAPS;             // channels at a time
        for (int c0 = 0; c0 < Cin; c0 += stage) {
            const int c1 = min(Cin, c0 + stage);
            drain_any(false);
            // A row holds PS pixels, each moved by the channel's number so that neighbouring channels fall into different banks;
            // eight loads of a thread are in flight.  NHWC: a warp reads the channels of a pixel's tap, channel-major: pixels.
            auto place = [&](int c, int t, int i) { return rows + ((c - c0) * T::TAPS + t) * PS + (i ^ (c & (PS - 1))); };
            auto source = [&](int i, int t) {                  // of channel 0; NULL outside the image
                const int m = list[first + i], dy = T::TAPS == 9 ? t / 3 - 1 : 0, dx = T::TAPS == 9 ? t % 3 - 1 : 0;
                const bool in = T::TAPS == 1 || ((unsigned)(m % W + dx) < (unsigned)W && (unsigned)(m / W % H + dy) < (unsigned)H);
                return in ? e.x + ((long long)m + dy * W + dx) * e.pixel_stride : nullptr;
            };
            float v[8];
            if (CM) {
                for (int t = 0; t < T::TAPS; ++t) {
                    const float* const x = p < pixels ? source(p, t) : nullptr;
                    for (int c = c0 + warp * us + u; c < c1; c += 64 * us) {
                        if constexpr (T::FUSED) {
#pragma unroll 1
                            for (int k = 0; k < 8; ++k)
                                if (c + 8 * us * k < c1) *place(c + 8 * us * k, 0, p) = x ? depthwise_output<T>(args, list[first + p], c + 8 * us * k) : 0.0f;
                            continue;
                        }
#pragma unroll
                        for (int k = 0; k < 8; ++k) v[k] = x && c + 8 * us * k < c1 ? x[(c + 8 * us * k) * e.channel_stride] : 0.0f;
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (c + 8 * us * k < c1) *place(c + 8 * us * k, t, p) = v[k];
                    }
                }
            } else {
                for (int r = warp; r < PS * T::TAPS; r += 8) {
                    const int i = r / T::TAPS, t = r % T::TAPS;
                    const float* const x = i < pixels ? source(i, t) : nullptr;
                    for (int c = c0 + lane; c < c1; c += 256) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) v[k] = x && c + 32 * k < c1 ? x[c + 32 * k] : 0.0f;
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (c + 32 * k < c1) *place(c + 32 * k, t, i) = v[k];
                    }
                }
            }
            drain_any(false);
            const int chunks = 2 * len / width;
            for (int i = warp; i < chunks; i += 8) {
                const int wg = i * width / len, n = n0 + wg * T::COLS + i * width - wg * len;
                if (n >= Cout) continue;
                const int g = n / e.G;
                auto first_unit = [&](int c) {                 // of the group, with a channel from c on
                    int lo = e.group_ptr[g], hi = e.group_ptr[g + 1];
                    while (lo < hi) {
                        const int mid = (lo + hi) / 2;
                        if (e.idx[mid] < c) lo = mid + 1; else hi = mid;
                    }
                    return lo;
                };
                const int lo = c0 > 0 ? first_unit(c0) : e.group_ptr[g], hi = c1 < Cin ? first_unit(c1) : e.group_ptr[g + 1];
                const int items = (hi - lo) * T::TAPS;
                const float* const v = e.val + (size_t)lo * T::TAPS * e.G + n % e.G;
                float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                int c = 0;
                float4 w = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                auto fetch = [&](int item) {                   // a lane's pair of the next 32, while the others are added up
                    if (item >= items) return;
                    c = e.idx[lo + item / T::TAPS];
                    if (T::TAPS == 9 && e.taps && !(e.taps[lo + item / T::TAPS] >> item % T::TAPS & 1)) c = -1;
                    const float* from = v + (size_t)item * e.G;
                    if (width == 4) w = __ldg(reinterpret_cast<const float4*>(from));
                    else w = make_float4(__ldg(from), width > 1 ? __ldg(from + 1) : 0.0f, 0.0f, 0.0f);
                };
                fetch(lane);
                for (int i0 = 0; i0 < items; i0 += 32) {
                    const int limit = min(32, items - i0);
                    __syncwarp();
                    where[lane] = c < 0 ? -1 : (((c - c0) * T::TAPS + (i0 + lane) % T::TAPS) * PS) | (c & (PS - 1));
                    weight[lane] = w;
                    __syncwarp();
                    fetch(i0 + 32 + lane);
                    auto add = [&](int k) {
                        if (T::TAPS == 9 && where[k] < 0) return;
                        const float4 w = weight[k];
                        const float x = rows[where[k] ^ p];
                        s[0] = fmaf(w.x, x, s[0]); s[1] = fmaf(w.y, x, s[1]); s[2] = fmaf(w.z, x, s[2]); s[3] = fmaf(w.w, x, s[3]);
                    };
                    if (us == 1 && limit == 32) {
#pragma unroll
                        for (int k = 0; k < 32; ++k) add(k);
                    } else {
                        for (int k = u; k < limit; k += us) add(k);
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (r >= width) break;
                    for (int d = PS; d < 32; d *= 2) s[r] += __shfl_xor_sync(0xffffffffu, s[r], d);
                    float* const sum = sums + (i * width + r) * 32 + p;
                    if (lane >= pixels) continue;              // (u > 0 or no pixel)
                    if (c0 > 0) s[r] += *sum;
                    if (c1 < Cin) {
                        *sum = s[r];
                    } else {
                        const int m = list[first + p];
                        float out = s[r] + bias[n + r];
                        if (relu) out = fmaxf(out, 0.0f);
                        y[T::OUT_CM ? (size_t)(n + r) * ldy + m : (size_t)m * ldy + n + r] = out;
                    }
                }
            }
        }
    }
}

// Last step of a tile whose steps were shared by the `split` CTAs of a cluster, for the drain threads: chunk c of a
// thread's channels (four of them) belongs to the last CTA r with r * CHUNKS / split <= c (quotients by a factor that comes
// with the launch: with divisions here tiles shared by 8 took 0.1 to 0.2 us longer).  Everybody writes its sums of the
// chunks of others into their shared memory, [sender][chunk][thread], and then adds up and stores its own.  The stages hold the
// exchange: every CTA's MMAs are complete when its drain threads reach the first barrier.
template <class T>
__device__ __forceinline__ void store_shared_tile(const typename T::Args& a, uint64_t (&acc)[T::COLS / 2], unsigned char* room, float* sums, int m0, int tid) {
    constexpr int CHUNKS = T::COLS / 4;
    const uint32_t exchange = smem_u32(room);
    const unsigned char* const mine = room;
    const int m = m0 + (tid & 127), n00 = blockIdx.x / a.split % a.ntiles_n * T::BN, n0 = n00 + (tid >> 7) * T::COLS;
    const int share = a.resident_or_share, rank = (int)cluster_rank(), slots = (share + 65534) >> 16;
    auto first_of = [&](int r) { return r * share >> 16; };
    const int first = first_of(rank), own = first_of(rank + 1) - first;
    __syncwarp();
    cluster_sync();
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
        const int owner = ((c + 1) * a.split - 1) / CHUNKS;
        float4 v;
        unpack2(acc[2 * c], v.x, v.y);
        unpack2(acc[2 * c + 1], v.z, v.w);
        if (owner != rank) store_remote(exchange + ((rank * slots + c - first_of(owner)) * 256 + tid) * 16, owner, v);
    }
    cluster_sync();
    bool redo = false;
#pragma unroll
    for (int c = 0; c < CHUNKS; ++c) {
        if (c < first || c >= first + own) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < a.split; ++s) {
            float4 o = reinterpret_cast<const float4*>(mine)[(s * slots + c - first) * 256 + tid];
            if (s == rank) {
                unpack2(acc[2 * c], o.x, o.y);
                unpack2(acc[2 * c + 1], o.z, o.w);
            }
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        redo |= !(fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, v.w * 0.f))) == 0.f);
        if (a.relu) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
        const int n = n0 + 4 * c;
        if (m < a.M && n < a.Cout) {
            if (T::OUT_CM) {
                float* yp = a.y + (size_t)n * a.ldy + m;
                yp[0] = v.x;
                if (n + 1 < a.Cout) yp[a.ldy] = v.y;
                if (n + 2 < a.Cout) yp[2 * (size_t)a.ldy] = v.z;
                if (n + 3 < a.Cout) yp[3 * (size_t)a.ldy] = v.w;
            } else {
                *reinterpret_cast<float4*>(a.y + (size_t)m * a.ldy + n) = v;   // Cout is a multiple of 4
            }
        }
    }
    redo = redo && m < a.M;
    if (T::IMAGES == 3 && drain_any(redo)) sum_kept_units<T>(a, room, sums, m0, redo, n00 + first * 4, own * 4);
}

__device__ __forceinline__ float shared_f1(uint32_t addr) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float4 shared_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ void store_relu(uint32_t addr, const float (&s)[4]) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};"
                 ::"r"(addr), "f"(fmaxf(s[0], 0.0f)), "f"(fmaxf(s[1], 0.0f)), "f"(fmaxf(s[2], 0.0f)), "f"(fmaxf(s[3], 0.0f))
                 : "memory");
}

// A thread of the split warpgroups in a launch with a depthwise layer (SRC_DW): lanes 8 * i .. 8 * i + 7 of warp q own 8 channels
// of a run of pixels, which they take four at a time.
template <class D>
struct DwThread {
    static constexpr int BLOCKS = D::SUB / 8, GROUPS = D::SUB / 4;    // blocks of 8 channels, groups of 4 pixels
    int c, p0;
    int x, y, r;                                                      // of the tile's first group: its place in the image, and (stride 2) in the stage
    __device__ DwThread(int q, int lane) : c(q % BLOCKS * 8 + (lane & 7)), p0(q / BLOCKS * 32 * BLOCKS + (lane >> 3) * 4 * GROUPS) {}
    __device__ void tile(int m0) {
        const int m = m0 + p0, f = m / D::WO;
        x = m % D::WO;
        y = f % D::WO;
        r = 2 * (f - m0 / D::WO);                                     // box rows r, r + 1, r + 2
    }
    // A stage's depthwise output, bias first and the taps in order as in the depthwise kernels, then ReLU; `zeros`: what is outside.
    // Bound by the latency of one warp's instructions: a stage of 16 channels takes a warpgroup 1000 cycles, 500 more the split.
    // (With a pixel a lane, for every tap a load of each channel and its weight, a 64-channel step took 6000 cycles instead of 4400:
    // the loads fill 11 values for each output.  Four split warpgroups with stages of 8 channels: 82 instead of 69 us for 64
    // images of 56 x 56, 128 -> 128; the columns beside a group summed apart, to save selects: 73.)
    __device__ __forceinline__ void run(uint32_t stage, uint32_t out, uint32_t zeros) const {
        float w[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) w[t] = shared_f1(stage + D::X_BYTES + (t * D::SUB + c) * 4);
        const float bias = shared_f1(stage + D::X_BYTES + (9 * D::SUB + c) * 4);
        const uint32_t to = out + (c * D::PITCH + p0) * 4;
        int x = this->x, y = this->y;
        if constexpr (D::S == 1) {
            uint32_t row[3];                                          // of the first group
#pragma unroll
            for (int i = 0; i < 3; ++i) row[i] = stage + (c * D::PB + D::LEAD + p0 + (D::ROWS3 ? i * D::BOX : (i - 1) * D::WI)) * 4;
            auto at = [&](int i, int y, uint32_t addr) { return i == 1 || (i == 0 ? y > 0 : y < D::WO - 1) ? addr : zeros; };
            float left[3];
            float4 here[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                here[i] = shared_f4(at(i, y, row[i]));
                left[i] = shared_f1(at(i, y, row[i] - 4));
            }
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) {
                const bool first = x == 0, last = x == D::WO - 4;
                const int yn = !last ? y : (y == D::WO - 1 ? 0 : y + 1);
                float4 next[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    if (g < GROUPS - 1) next[i] = shared_f4(at(i, yn, row[i] + 16 * g + 16));
                    else next[i].x = shared_f1(at(i, y, row[i] + 16 * g + 16));
                }
                float s[4] = {bias, bias, bias, bias};
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float v[6] = {first ? 0.0f : left[i], here[i].x, here[i].y, here[i].z, here[i].w, last ? 0.0f : next[i].x};
#pragma unroll
                    for (int t = 0; t < 3; ++t)
#pragma unroll
                        for (int k = 0; k < 4; ++k) s[k] = fmaf(v[k + t], w[3 * i + t], s[k]);
                    left[i] = here[i].w;
                    here[i] = next[i];
                }
                store_relu(to + 16 * g, s);
                x = last ? 0 : x + 4;
                y = yn;
            }
        } else {
            int r = this->r;
            float left[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int g = 0; g < GROUPS; ++g) {
                const bool first = x == 0;
                float s[4] = {bias, bias, bias, bias};
                float4 a[3], b[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const uint32_t row = stage + ((r + i) / D::BR * D::BOX + c * D::PB + (r + i) % D::BR * D::WI + 2 * x) * 4;
                    const bool in = i > 0 || y > 0;
                    a[i] = shared_f4(in ? row : zeros);
                    b[i] = shared_f4(in ? row + 16 : zeros);
                    if (g == 0) left[i] = shared_f1(in && !first ? row - 4 : zeros);
                }
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float v[9] = {first ? 0.0f : left[i], a[i].x, a[i].y, a[i].z, a[i].w, b[i].x, b[i].y, b[i].z, b[i].w};
#pragma unroll
                    for (int t = 0; t < 3; ++t)
#pragma unroll
                        for (int k = 0; k < 4; ++k) s[k] = fmaf(v[2 * k + t], w[3 * i + t], s[k]);
                    left[i] = b[i].w;
                }
                store_relu(to + 16 * g, s);
                x += 4;
                if (x == D::WO) {
                    x = 0;
                    r += 2;
                    y = y == D::WO - 1 ? 0 : y + 1;
                }
            }
        }
    }
};

// The split warps of a launch whose activations are the output of a depthwise layer (SRC_DW).  The two warpgroups take the
// stages in turn (an even number of them, so that a stage always belongs to the same one): depthwise output into shared
// memory, then as for other sources, a pixel a lane, into bf16 images.  A warp that gave up still joins its warpgroup's barriers.
// `wait`, `stages`: as in the kernel.
template <class T, class Stages, class Wait>
__device__ __forceinline__ bool depthwise_split(const DwArgs& a, const unsigned char* ast, float* out, const float4* zeros, Ring ring, uint64_t* xfull,
                                                uint64_t* xempty, uint64_t* afull, uint64_t* aempty, uint32_t lane_base, int half, int q, int lane,
                                                int kb, int ke, Stages stages, Wait wait) {
    using D = typename T::DW;
    auto together = [&] { asm volatile("barrier.cta.sync %0, 128;" ::"r"(2 + half) : "memory"); };
    const float* const pixel = out + q * 32 + lane;
    DwThread<D> thread(q, lane);
    int step = 0;
    bool ok = true;
    if (half) ring.next();
    for (Tiles t(a); t.left(); t.next()) {
        thread.tile(t.m * T::BM);
        for (int k0 = kb; k0 < ke; ++k0, ++step) {
            const int as = step % T::NA, n = stages(k0);
            for (int i = half; i < n; i += 2) {
                // lane 0: the place in tensor memory is free, others: the stage is here
                const bool place = lane == 0 && i == half && step >= T::NA;
                ok = ok && wait(place ? aempty + as : xfull + ring.stage, place ? ((step / T::NA) & 1) ^ 1 : ring.parity);
                if (ok) {
                    tc_fence_after_sync();
                    thread.run(smem_u32(ast) + ring.stage * T::A_BYTES, smem_u32(out), smem_u32(zeros));
                    __syncwarp();
                    if (lane == 0) mbar_arrive(xempty + ring.stage);
                }
                together();
                if (ok) {
                    const uint32_t col = lane_base + as * T::A_COLS + i * D::SUB / 2;
                    uint32_t h[D::SUB / 2], md[D::SUB / 2], lo[D::SUB / 2];
#pragma unroll
                    for (int k = 0; k < D::SUB / 2; ++k)
                        split2(pack2(pixel[2 * k * D::PITCH], pixel[(2 * k + 1) * D::PITCH]), h[k], md[k], lo[k]);
                    tmem_st(col + 32, md);
                    tmem_st(col + 64, lo);
                    tmem_st(col, h);
                }
                together();
                ring.next();
                ring.next();
            }
            if (!ok) continue;
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(afull + as);
        }
    }
    return ok;
}

template <class T>
__global__ void __launch_bounds__(T::NT, 1)
conv_tc_kernel(const __grid_constant__ CUtensorMap amap, const __grid_constant__ CUtensorMap ymap, const __grid_constant__ typename T::Args a) {
    constexpr int NUC = T::NUC, NU = T::NU, BN = T::BN;
    const int SA = a.sa, SB = a.sb;
    const bool resident = !T::SPLIT && a.resident_or_share;
    extern __shared__ unsigned char raw[];
    const uint32_t raw_addr = smem_u32(raw);
    unsigned char* bst = raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);    // weight stages, 1024-byte aligned
    unsigned char* ast = bst + (size_t)SB * T::B_BYTES;                       // activation stages
    unsigned char* ost = ast + (size_t)SA * T::A_BYTES;                       // output staging
    uint64_t* xfull = reinterpret_cast<uint64_t*>(ost + T::OUT_BYTES);
    uint64_t* xempty = xfull + SA;
    uint64_t* bfull = xempty + SA;
    uint64_t* bempty = bfull + 2 * SB;
    uint64_t* afull = bempty + SB;      // A images of a step are in tensor memory
    uint64_t* aempty = afull + T::NA;
    uint64_t* dfull = aempty + T::NA;       // accumulator of a step is complete
    uint64_t* dempty = dfull + 2;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(dempty + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_holder + 1);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wg = warp >> 2;
    float* const dwout = reinterpret_cast<float*>(ost + T::OUT_BYTES + T::CTRL);   // SRC_DW: see DwShape
    float4* const zeros = reinterpret_cast<float4*>(ost + T::OUT_BYTES + T::CTRL - 16);
    if (T::FUSED && tid == 0) *zeros = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (warp == 16 && lane == 0) {
        prefetch_map(&amap);
        prefetch_map(&ymap);
    }
    if (tid == 0) {
        for (int s = 0; s < SA; ++s) { mbar_init(xfull + s, 1); mbar_init(xempty + s, T::FUSED ? 4 : 8); }
        for (int s = 0; s < SB; ++s) { mbar_init(bfull + s, 1); mbar_init(bfull + SB + s, 1); mbar_init(bempty + s, 1); }
        for (int s = 0; s < 2; ++s) {
            mbar_init(dfull + s, 1); mbar_init(dempty + s, T::DEMPTY);
        }
        for (int s = 0; s < T::NA; ++s) { mbar_init(afull + s, 8); mbar_init(aempty + s, NU); }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 18) tmem_alloc(tmem_holder, 512);
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_holder, 0);

    // Whole warp: until the barrier that each lane names has completed its phase; the same result in all lanes.  (A wait
    // costs 60 to 100 cycles even when there is nothing to wait for, so a warp looks at all it needs at once, a barrier a lane.)
    auto wait = [&](uint64_t* bar, uint32_t parity, bool needed = true) {
        uint32_t polls = 0;
        while (!__all_sync(0xffffffffu, (int)mbar_try_wait(bar, parity) | (int)!needed)) {
            if (++polls > 64) {
                if (__any_sync(0xffffffffu, polls > kWaitLimit || *abort_flag)) {
                    *abort_flag = 1;
                    atomicCAS(a.status, 0, SBNN_ERR_TIMEOUT);
                    return false;
                }
                __nanosleep(64);
            }
        }
        // A wait makes the guarded memory visible to the lane that polled; the other lanes get it through this barrier (a vote
        // orders no memory).
        __syncwarp();
        return true;
    };
    // this CTA's steps of its tiles
    int kb = 0, ke = a.steps;
    if (T::SPLIT) {
        const int rank = (int)cluster_rank(), runs = a.steps / T::RUN;
        kb = runs * rank / a.split * T::RUN;
        ke = runs * (rank + 1) / a.split * T::RUN;
    }
    // valid 32-channel halves of a step, and its activation stages
    auto subs = [&](int k) { return a.Cin - (k / T::TAPS) * 64 > 32 ? 2 : 1; };
    auto stages = [&](int k) { return subs(k) * (32 / T::SUB); };

    if (wg >= 2) {
        if (wg < 4) regs_dec<T::SPLIT_REGS>(); else regs_dec<T::AUX_REGS>();
        if (warp == 16) {
            // ---------------- activation copies ----------------
            Ring ring(SA);
            bool ok = true;
            grid_dependency_wait();                       // X comes from the previous kernel of the stream
            grid_dependency_release();                    // (only now: the next kernel must not run beside the one before this)
            for (Tiles t(a); t.left() && ok; t.next()) {
                const int m0 = t.m * T::BM;
                int px = 0, py = 0, pn = 0;
                if (T::SRC == SRC_IM2COL) { px = m0 % a.W; py = (m0 / a.W) % a.H; pn = m0 / (a.W * a.H); }
                for (int k = kb; k < ke && ok; k += T::RUN) {
                    const int c = k / T::TAPS, tap = k - c * T::TAPS, halves = stages(k);
                    // With stages enough both halves of a step are asked for after one wait: a wait and an issue take a warp
                    // 370 cycles, which for 16 KB at a time is slower than the memory.
                    const int batch = SA >= 4 ? (T::FUSED ? 2 : halves) : 1;
                    for (int h = 0; h < halves && ok; h += batch) {
                        Ring second = ring;
                        second.next();
                        const Ring& mine = lane == 1 && batch == 2 ? second : ring;   // lane 1 looks at the second stage
                        if (second.reused() && !(ok = wait(xempty + mine.stage, mine.parity ^ 1, mine.reused()))) break;
                        if (elect_one()) {
                            for (int b = 0; b < batch; ++b) {
                                const int s = b ? second.stage : ring.stage, c0 = c * 64 + (h + b) * T::SUB;
                                unsigned char* dst = ast + (size_t)s * T::A_BYTES;
                                mbar_arrive_expect_tx(xfull + s, T::A_COPIED);
                                if constexpr (T::FUSED) {
                                    using D = typename T::DW;
                                    const int first = D::S == 2 ? (2 * (m0 / D::WO) - 1) * D::WI - D::LEAD : (D::ROWS3 ? m0 - D::WI : m0) - D::LEAD;
#pragma unroll
                                    for (int i = 0; i < D::BOXES; ++i)
                                        tensor_g2s_2d(dst + i * D::SUB * D::PB * 4, &amap, first + i * (D::S == 2 ? D::BR : 1) * D::WI, c0, xfull + s);
                                    tensor_g2s_2d(dst + D::X_BYTES, &a.wmap, c0, 0, xfull + s);
                                    bulk_g2s(dst + D::X_BYTES + 9 * D::SUB * 4, a.dw_b + c0, D::SUB * 4, xfull + s);
                                    continue;
                                }
                                if (T::SRC == SRC_CM) tensor_g2s_2d(dst, &amap, m0, c0, xfull + s);
                                else if (T::SRC == SRC_CM3) tensor_g2s_2d(dst, &amap, (m0 + (tap / 3 - 1) * a.W - 1) & ~3, c0, xfull + s);
                                else if (T::SRC == SRC_NHWC) tensor_g2s_2d(dst, &amap, c0, m0, xfull + s);
                                else im2col_g2s(dst, &amap, c0, px - 1, py - 1, pn, tap % 3, tap / 3, xfull + s);
                            }
                        }
                        __syncwarp();
                        ring.next();
                        if (batch == 2) ring.next();
                    }
                }
            }
            if (!ok) ring.settle(xfull, false);
        } else if (warp == 17) {
            // ---------------- weight copies ----------------
            // The first round of stages is filled while the previous kernel of the stream drains.  No bounded wait starts before
            // that kernel is done, here and in the warps below: its time must not count.
            Ring ring(SB);
            bool ok = true, alone = false;
            for (Tiles t(a); t.left() && ok; t.next()) {
                const int nt = t.n * NU;
                const int batch = SB >= 4 ? NU : 1;         // as above
                for (int k = kb; k < ke && ok; ++k)
                    for (int u = 0; u < NU && ok; u += batch) {
                        Ring second = ring;
                        second.next();
                        const Ring& mine = lane == 1 && batch == 2 ? second : ring;
                        if (second.reused() && !alone) {
                            grid_dependency_wait();
                            alone = true;
                        }
                        if (second.reused() && !(ok = wait(bempty + mine.stage, mine.parity ^ 1, mine.reused()))) break;
                        if (elect_one()) {
                            for (int b = 0; b < batch; ++b) {
                                const Ring& r = b ? second : ring;
                                mbar_arrive_expect_tx(bfull + r.turn(), T::B_BYTES);
                                bulk_g2s(bst + (size_t)r.stage * T::B_BYTES, a.wts + ((size_t)(nt + u + b) * a.steps + k) * (T::B_BYTES / 16), T::B_BYTES,
                                         bfull + r.turn());
                            }
                        }
                        __syncwarp();
                        ring.next();
                        if (batch == 2) ring.next();
                    }
                if (resident) break;
            }
            if (!ok) ring.settle(bfull, true);
        } else if (warp >= 18) {
            // ---------------- MMA issue ----------------
            constexpr uint32_t idesc = instr_desc(NUC);
            // (image of A, image of B), small products first: h = 0, m = 1, l = 2
            constexpr int PA[6] = {2, 0, 1, 1, 0, 0}, PB[6] = {0, 2, 1, 0, 1, 0};
            const int w = warp - 18;
            int step = 0, unit = 0;
            Ring ring(SB);
            bool ok = true;
            grid_dependency_wait();
            // Three images: every step of a column block is a unit with an accumulator of its own, and the warps take turns.
            // One image: a unit is a column block of a tile, warp u takes block u (with one block warp 0 takes all).
            for (Tiles t(a); t.left() && ok; t.next()) {
                for (int k0 = kb; k0 < ke && ok; ++k0, ++step)
                    for (int u = 0; u < NU; ++u, ring.next()) {
                        if (T::IMAGES == 3) {
                            if ((unit++ & 1) != w) continue;
                        } else if (u != w) {
                            continue;
                        }
                        const int mine = T::IMAGES == 3 ? unit - 1 : unit + w, d = mine & 1;
                        const int as = step % T::NA, s = ring.stage;
                        // lane 0: the accumulator is drained, lane 1: the weights are here, others: so are the activations
                        uint64_t* bar = afull + as;
                        uint32_t parity = (step / T::NA) & 1;
                        if (lane == 1) {
                            bar = bfull + ring.turn();
                            parity = ring.turn_parity();
                        } else if (lane == 0 && (T::IMAGES == 3 || k0 == kb) && mine >= 2) {
                            bar = dempty + d;
                            parity = ((mine >> 1) & 1) ^ 1;
                        }
                        if (!(ok = wait(bar, parity))) break;
                        tc_fence_after_sync();
                        const uint32_t a_base = tmem + T::A_COL0 + as * T::A_COLS;
                        const uint64_t b_desc = operand_desc(smem_u32(bst) + (uint32_t)s * T::B_BYTES);
                        const bool whole = subs(k0) == 2;
                        const uint32_t more = T::IMAGES == 1 && k0 > kb ? 1u : 0u;
                        constexpr int P0 = T::IMAGES == 3 ? 0 : 5, NP = 6 - P0;      // one image: just h * h
                        if (elect_one()) {
                            if (whole) {
#pragma unroll
                                for (int i = 0; i < 4 * NP; ++i) {
                                    const int p = P0 + (i >> 2), k = i & 3;
                                    umma_bf16_ta(tmem + d * T::D_COLS, a_base + PA[p] * 32 + k * 8, b_desc + ((PB[p] * (NUC * 128) + k * 32) >> 4),
                                                 idesc, i ? 1u : more);
                                }
                            } else {
#pragma unroll
                                for (int i = 0; i < 2 * NP; ++i) {
                                    const int p = P0 + (i >> 1), k = i & 1;
                                    umma_bf16_ta(tmem + d * T::D_COLS, a_base + PA[p] * 32 + k * 8, b_desc + ((PB[p] * (NUC * 128) + k * 32) >> 4),
                                                 idesc, i ? 1u : more);
                                }
                            }
                            if (!resident) umma_commit(bempty + s);
                            if (T::IMAGES == 3 || k0 == ke - 1) umma_commit(dfull + d);
                            umma_commit(aempty + as);
                        }
                        __syncwarp();
                    }
                if (T::IMAGES == 1) unit += NU;
                if (resident) ring = Ring(SB);            // the same stages again, still full from the first round
            }
        } else if (wg < 4) {
            // ---------------- split into bf16 images ----------------
            const int half = wg - 2, q = warp & 3, p = q * 32 + lane;   // pixel of the tile = tensor-memory lane
            const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16) + T::A_COL0;
            int step = 0;
            Ring ring(SA);
            bool ok = true;
            grid_dependency_wait();
            if constexpr (T::FUSED) {
                ok = depthwise_split<T>(a, ast, dwout + half * T::DW::SUB * T::DW::PITCH, zeros, ring, xfull, xempty, afull, aempty, lane_base, half, q, lane, kb,
                                        ke, stages, wait);
            } else
            for (Tiles t(a); t.left() && ok; t.next()) {
                int px = 0, py = 0;                         // SRC_CM3: the pixel's place in its image
                if (T::SRC == SRC_CM3) {
                    const int m = t.m * T::BM + p;
                    px = m % a.W;
                    py = (m / a.W) % a.H;
                }
                for (int k0 = kb; k0 < ke && ok; ++k0, ++step) {
                    const int as = step % T::NA, halves = subs(k0);
                    const int tap = k0 % T::TAPS, dy = tap / 3 - 1, dx = tap % 3 - 1;
                    const bool inside = T::SRC != SRC_CM3 || ((unsigned)(px + dx) < (unsigned)a.W && (unsigned)(py + dy) < (unsigned)a.H);
                    const int shift = T::SRC == SRC_CM3 ? ((t.m * T::BM + dy * a.W - 1) & 3) + 1 + dx : 0;
                    const uint32_t col = lane_base + as * T::A_COLS + half * 8;
                    // lane 0: the place in tensor memory is free, lane 1: the second half of the step is here, others: the first
                    Ring at = ring;
                    uint64_t* bar = xfull + at.stage;
                    uint32_t parity = at.parity;
                    if (lane == 1 && halves == 2) {
                        Ring second = at;
                        second.next();
                        bar = xfull + second.stage;
                        parity = second.parity;
                    } else if (lane == 0 && step >= T::NA) {
                        bar = aempty + as;
                        parity = ((step / T::NA) & 1) ^ 1;
                    }
                    if (!(ok = wait(bar, parity))) break;
                    tc_fence_after_sync();
                    for (int h = 0; h < halves; ++h, at.next()) {
                        const int s = at.stage;
                        const unsigned char* src = ast + (size_t)s * T::A_BYTES;
                        uint64_t v[8];                // pairs of neighbouring channels
                        if (T::SRC == SRC_CM || T::SRC == SRC_CM3) {
                            const float* row = reinterpret_cast<const float*>(src) + half * 16 * T::PIX + shift + p;
#pragma unroll
                            for (int k = 0; k < 8; ++k)
                                v[k] = inside ? pack2(row[2 * k * T::PIX], row[(2 * k + 1) * T::PIX]) : 0;
                        } else {
                            // 16-byte chunk c of the pixel's row sits at chunk c ^ (p & 7)
                            const uint32_t row = smem_u32(src) + p * 128 + ((p & 7) << 4);
#pragma unroll
                            for (int j = 0; j < 4; ++j) load_shared(row ^ ((half * 4 + j) << 4), v[2 * j], v[2 * j + 1]);
                        }
                        uint32_t hh[8], mm[8], ll[8];
                        if (T::IMAGES == 3) {
#pragma unroll
                            for (int k = 0; k < 8; ++k) split2(v[k], hh[k], mm[k], ll[k]);
                            tmem_st(col + h * 16 + 32, mm);
                            tmem_st(col + h * 16 + 64, ll);
                        } else {
#pragma unroll
                            for (int k = 0; k < 8; ++k) hh[k] = bf16_of(v[k]);
                        }
                        tmem_st(col + h * 16, hh);
                        __syncwarp();
                        if (lane == 0 && tap % T::RUN == T::RUN - 1) mbar_arrive(xempty + s);
                    }
                    if (tap % T::RUN == T::RUN - 1) ring = at;   // else the next tap reads the same stages
                    tmem_st_wait();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(afull + as);
                }
            }
        }
        if (T::SPLIT) {
            __syncwarp();
            cluster_sync();
            cluster_sync();
        }
    } else {
        // ---------------- drain and store ----------------
        regs_inc<T::DRAIN_REGS>();
        const int q = warp & 3;
        const uint32_t lane_base = tmem + ((uint32_t)(q * 32) << 16);
        unsigned char* stage = ost + (size_t)warp * (T::OUT_TILES * 2048);
        int step = 0, copies = 0;                           // copies issued: the two tiles alternate between them
        bool ok = true, again = false;                      // again: some of this lane's pixels have to be summed once more
        grid_dependency_wait();                             // Y may still be read by the previous kernel of the stream
        for (Tiles t(a); t.left() && ok; t.next()) {
            const int m0 = t.m * T::BM, n0 = t.n * BN + wg * T::COLS;
            uint64_t acc[T::COLS / 2];                      // pairs of neighbouring channels, from the bias on
#pragma unroll
            for (int i = 0; i < T::COLS / 4; ++i) {
                ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(a.bias + n0) + i);
                if (T::SPLIT && kb) b = make_ulonglong2(0, 0);
                acc[2 * i] = b.x;
                acc[2 * i + 1] = b.y;
            }
            for (int k = T::IMAGES == 3 ? kb : ke - 1; k < ke; ++k, ++step) {
                // two column blocks: a warpgroup drains its own; one block: both drain their half of every accumulator
                const int unit = NU == 2 ? 2 * step + wg : step, d = unit & 1;
                if (!(ok = wait(dfull + d, (unit >> 1) & 1))) break;
                tc_fence_after_sync();
                const uint32_t col = lane_base + d * T::D_COLS + (NU == 2 ? 0 : wg * T::COLS);
                constexpr int LD = T::BN == 256 ? 16 : 32;      // columns at a time: what registers there are left
#pragma unroll
                for (int c0 = 0; c0 < T::COLS; c0 += LD) {
                    uint32_t v[LD];
                    tmem_ld(col + c0, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < LD / 2; ++i) acc[c0 / 2 + i] = add2(acc[c0 / 2 + i], join2(v[2 * i], v[2 * i + 1]));
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(dempty + d);
            }
            if (T::SPLIT) {
                store_shared_tile<T>(a, acc, bst, reinterpret_cast<float*>(ost), m0, tid);
                break;
            }
            if (!ok) break;
            const int m = m0 + q * 32 + lane;
            // Any sum that is not finite: a bad activation spoils them all, an overflow on the way, which another order of the
            // additions may not have, only its own.  (0 * sum is NaN then, and stays it.)
            bool redo = false;
            if (T::IMAGES == 3) {
                f32x2 probe[4] = {0, 0, 0, 0};
                float lo, hi;
#pragma unroll
                for (int i = 0; i < T::COLS / 2; ++i) fma2(probe[i & 3], acc[i], 0);
                unpack2(add2(add2(probe[0], probe[1]), add2(probe[2], probe[3])), lo, hi);
                redo = m < a.M && !(lo + hi == 0.0f);
            }
            again |= redo;
            // 32 pixels x 16 channels at a time through one of the warp's two staging tiles, stored by tiled copies: rows of 32
            // pixels (channel-major) or of 16 channels (64-byte swizzle).  Rows past Cout or M are clipped by the copy; the last
            // pixels of a channel-major row are stored one by one, so that the padding behind them is left alone.
            // (Stores straight from registers, one row of 32 pixels each, took 100 cycles apiece: 13700 cycles for a tile
            // of 256 channels.)
            const int mw = m0 + q * 32;
#pragma unroll
            for (int c0 = 0; c0 < T::COLS; c0 += 16) {
                if (n0 + c0 < a.Cout && mw < a.M) {         // warp-uniform
                    float o[16];
#pragma unroll
                    for (int i = 0; i < 8; ++i) unpack2(acc[c0 / 2 + i], o[2 * i], o[2 * i + 1]);
                    if (a.relu) {
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = fmaxf(o[i], 0.0f);
                    }
                    if (c0 == 0 && redo) o[0] = __int_as_float(0x7fffffff);   // marks the pixel for the second look below
                    if (T::OUT_CM && mw + 32 > a.M) {
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            if (m < a.M && n0 + c0 + i < a.Cout) a.y[(size_t)(n0 + c0 + i) * a.ldy + m] = o[i];
                    } else {
                        unsigned char* tile = stage + (copies++ & (T::OUT_TILES - 1)) * 2048;
                        if (elect_one()) {                  // the copy that last read this tile is done with it
                            if (T::OUT_TILES == 2) bulk_wait_read_pending1(); else bulk_wait_read_all();
                        }
                        __syncwarp();
                        if (T::OUT_CM) {
#pragma unroll
                            for (int i = 0; i < 16; ++i) reinterpret_cast<float*>(tile)[i * 32 + lane] = o[i];
                        } else {
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                *reinterpret_cast<float4*>(tile + lane * 64 + ((j ^ (lane >> 1 & 3)) << 4)) =
                                    make_float4(o[4 * j], o[4 * j + 1], o[4 * j + 2], o[4 * j + 3]);
                        }
                        fence_async_smem();
                        __syncwarp();
                        if (elect_one()) {                  // (always the same lane)
                            tensor_s2g_2d(&ymap, T::OUT_CM ? mw : n0 + c0, T::OUT_CM ? n0 + c0 : mw, tile);
                            bulk_commit_group();
                        }
                    }
                }
            }
        }
        if (elect_one()) bulk_wait_all();                   // this thread's copies are complete before the CTA gives up its shared memory
        // Pixels that hold an infinity or a NaN: only now, when no warp of the CTA is left in a bounded wait for these.
        if (T::IMAGES == 3 && !T::SPLIT && drain_any(again && ok)) {
            for (Tiles t(a); t.left(); t.next()) {
                const int m = t.m * T::BM + q * 32 + lane, n0 = t.n * BN + wg * T::COLS;
                bool bad = false;
                if (n0 < a.Cout && m < a.M) {
                    const float mark = __ldcg(a.y + (T::OUT_CM ? (size_t)n0 * a.ldy + m : (size_t)m * a.ldy + n0));
                    bad = mark != mark;
                }
                if (drain_any(bad)) sum_kept_units<T>(a, bst, reinterpret_cast<float*>(ost), t.m * T::BM, bad, t.n * BN, T::COLS);
            }
        }
    }
    // common exit: nobody may still be using the tensor memory when it is released
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 18) tmem_dealloc(tmem, 512);
}

// One thread per (kept unit, tap, channel of the group): the weight's bf16 images into their place in the tiles.
__global__ void build_tc_weights_kernel(const int32_t* __restrict__ group_ptr, const int32_t* __restrict__ idx, const float* __restrict__ val,
                                        int G, int taps, int csteps, int nuc, int images, __nv_bfloat16* __restrict__ out) {
    const int g = blockIdx.x, per_unit = taps * G;
    const int lo = group_ptr[g];
    const long long n = (long long)(group_ptr[g + 1] - lo) * per_unit;
    for (long long i = threadIdx.x + (long long)blockIdx.y * blockDim.x; i < n; i += (long long)blockDim.x * gridDim.y) {
        const int j = lo + (int)(i / per_unit), t = (int)(i % per_unit) / G, o = g * G + (int)(i % G), c = idx[j];
        const int row = o % nuc, kk = c & 63;
        const size_t block = (size_t)(o / nuc) * csteps * taps + (size_t)(c >> 6) * taps + t;
        const size_t at = block * images * nuc * 64 + (size_t)row * 64 + ((((kk >> 3) ^ (row & 7)) << 3) | (kk & 7));
        if (images == 1) {
            out[at] = __float2bfloat16_rn(val[(size_t)j * per_unit + i % per_unit]);
            continue;
        }
        const double w = val[(size_t)j * per_unit + i % per_unit] * kTruncation;
        // Round to nearest; magnitudes that would round up to infinity are truncated instead.
        const __nv_bfloat16 h = fabs(w) > 3.3895e38 ? __float2bfloat16_rz(__double2float_rz(w)) : __float2bfloat16_rn((float)w);
        const double r = w - (double)__bfloat162float(h);
        const __nv_bfloat16 m = __float2bfloat16_rn((float)r);
        const __nv_bfloat16 l = __float2bfloat16_rn((float)(r - (double)__bfloat162float(m)));
        out[at] = h;
        out[at + (size_t)nuc * 64] = m;
        out[at + (size_t)2 * nuc * 64] = l;
    }
}

using TcChoice = sbnn_packed::TcChoice;

// Test hooks (sbnn_debug_conv_gs, sbnn_debug_last_route), for the calling thread: how its calls have to run (bn = 0: on the
// FMA kernels), and how the latest ran.
thread_local const TcChoice* forced_choice = nullptr;
thread_local TcChoice last_route = {0, 0, 0.0};

// Weight images of a layer for MMA column blocks of `nuc` output channels, built on first use; NULL if that would be
// in a call of M pixels the layer has been prepared for, which only enqueues, or while `st` is being captured, when nothing
// can be allocated, or if the device has no room for them (which is remembered: they take six bytes for every weight of the
// unpruned layer, many times what is stored of a sparse one).  `ask`: nothing is built, either.
sbnn_status get_tc_weights(const sbnn_packed* p, int nuc, int images, long long M, cudaStream_t st, uint4** out, bool ask = false) {
    std::lock_guard<std::mutex> lk(p->mu);
    *out = nullptr;
    auto it = p->tc_weights.find({nuc, images});
    if (it != p->tc_weights.end()) {
        *out = static_cast<uint4*>(it->second);
        return SBNN_OK;
    }
    if (ask) return SBNN_OK;
    auto prepared = p->tc_prepared.find(images);
    if (!prepare_only() && !forced_choice && prepared != p->tc_prepared.end() && M <= prepared->second) return SBNN_OK;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (!prepare_only() && cudaStreamIsCapturing(st, &cs) != cudaSuccess) cudaGetLastError();
    if (cs != cudaStreamCaptureStatusNone) return SBNN_OK;
    const int taps = p->KH * p->KW, csteps = (p->Cin + 63) / 64;
    const int tiles = nuc == 64 ? (p->Cout + 63) / 64 : (p->Cout + 255) / 256 * 2;    // (a tile of 256 channels reads two blocks of 128)
    const size_t bytes = (size_t)tiles * csteps * taps * images * nuc * 64 * 2;
    void* d = nullptr;
    cudaError_t e = bytes > p->tc_limit ? cudaErrorMemoryAllocation : cudaMalloc(&d, bytes);
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        p->tc_weights[{nuc, images}] = nullptr;
        return SBNN_OK;
    }
    if (e == cudaSuccess) e = cudaMemset(d, 0, bytes);
    if (e == cudaSuccess && p->nnz > 0) {
        build_tc_weights_kernel<<<dim3((unsigned)p->ngroups, 4), 128>>>(p->d_group_ptr, p->d_idx, p->d_val, p->G, taps, csteps, nuc, images,
                                                                       static_cast<__nv_bfloat16*>(d));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
    if (e != cudaSuccess) {
        cudaFree(d);
        cudaGetLastError();
        return fail(SBNN_ERR_CUDA, "building the tensor-core weights: %s", cudaGetErrorString(e));
    }
    p->tc_weights[{nuc, images}] = d;
    *out = static_cast<uint4*>(d);
    return SBNN_OK;
}

struct TcCall {
    const float* x;
    int ldx;           // channel-major sources
    float* y;
    int ldy;
    long long M;
    int N, H, W;       // 3x3
    int relu;
    cudaStream_t st;
    const float* dw_w;  // SRC_DW: the depthwise layer in front, and the pixels of its input
    const float* dw_b;
    long long M_in;
    bool ask;          // launch and build nothing, only say whether the call runs here
};

// ---- which kernel, and how ------------------------------------------------------------------------
// Cycles a launch takes with tiles of bn output channels: rounds of tiles x (steps + fill and store).  A step of 128 or 256
// channels takes about as long as its MMAs (64 cycles for 128 channels, 24 of them), 64 channels as long as the split of the
// activations; one image (bf16 mode) as long as the copies and the barriers around them.  Fitted to launches of 1 to 72
// steps on 1 to 112 CTAs (4.1 us for one step of 64 channels, 0.62 / 0.84 / 1.67 us for each further one of 64 / 128 / 256).
double tc_step(int bn, int images) {
    if (images == 1) return bn == 64 ? 600.0 : (bn == 128 ? 700.0 : 1150.0);
    return bn == 64 ? 1150.0 : 12.5 * bn;
}
double tc_cost(const sbnn_packed* p, long long M, int bn, int images) {
    const long long tiles = (M + 127) / 128 * ((p->Cout + bn - 1) / bn), sms = device_sms();
    const double steps = 0.5 * (double)((p->Cin + 31) / 32) * p->KH * p->KW;
    return (double)((tiles + sms - 1) / sms) * (steps * tc_step(bn, images) + (bn == 64 ? 1300.0 : 1000.0 + 12.0 * bn)) + 4700.0;
}
// Microseconds: long launches run at the clock that the power limit leaves them.
double tc_us(double cycles) { return cycles / (cycles < 1e5 ? 1800.0 : 1600.0); }

// Clusters of `split` CTAs that the device runs at the same time (on 148 SMs 74 of 2, 45 of 3, 33 of 4, 26 of 5, 22 of 6, 15 of 7 and 8).
long long cluster_capacity(int split) {
    static std::mutex mu;
    static std::map<std::pair<int, int>, int> known;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find({dev, split});
    if (it == known.end()) {
        using T = TC<64, SRC_CM, true, true>;
        int n = 0;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(device_sms() / split * split));
        cfg.blockDim = dim3(T::NT);
        cfg.dynamicSmemBytes = 227 * 1024;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = (unsigned)split;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (set_max_dyn_smem(reinterpret_cast<const void*>(&conv_tc_kernel<T>), 227 * 1024) != SBNN_OK ||
            cudaOccupancyMaxActiveClusters(&n, conv_tc_kernel<T>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        it = known.emplace(std::make_pair(dev, split), n).first;
    }
    return it->second;
}

// The same for 64-channel tiles shared by `split` CTAs; infinite when that is not below `limit` or they do not all run at the same time.
double tc_split_cost(const sbnn_packed* p, long long M, int split, int run, int images, double limit) {
    const long long tiles = (M + 127) / 128 * ((p->Cout + 63) / 64), runs = (long long)((p->Cin + 63) / 64) * p->KH * p->KW / run;
    if (runs < split || tiles * split > device_sms()) return 1e30;
    // Clusters of 5 to 7 start later: one 14 x 14 image, 512 -> 512, two steps a CTA in clusters of 4, 5, 6: 6.8, 7.3, 7.6 us; 2 x 28 x
    // 28, 128 -> 128 3x3, 18 steps in clusters of 4 and 5: 9.7 and 10.2.
    const double late = split > 4 && split < 8 ? 1500.0 : 0.0;
    // Steps of a last 64 channels that are 32 or fewer take 0.6 of the others, and count for the CTAs that get them.  3x3 channel-major, 144 ->
    // 32, nine kernel rows, the last three of 16 channels: shared by 4 11.0 us, by 5 11.6.
    const long long half = (p->Cin - 1) % 64 < 32 ? runs - p->KH * p->KW / run : runs;
    double most = 0.0;
    for (int r = 0; r < split; ++r) {
        const long long from = runs * r / split, to = runs * (r + 1) / split, whole = std::min(to, half) - std::min(from, half);
        most = std::max(most, (double)whole + 0.6 * (double)(to - from - whole));
    }
    const double cost = most * run * (tc_step(64, images) + 50.0) + 9800.0 + late;
    if (cost >= limit) return 1e30;
    // Behind another launch the last clusters of 3 and of 5 of a full device find no place before others have ended.  In clusters of 3, of
    // which 45 run at a time: 9 x 5 tiles of 6 steps 10.3 us (unshared 7.5), 5 x 9 of 10 steps 11.9 (of 2: 9.6), 44 tiles of 4 steps 9.0, 43
    // and fewer take what they are modelled at.  26 tiles of 17 steps in clusters of 5: 10.6 (of 4: 9.0).
    const long long capacity = cluster_capacity(split), spare = split == 3 || split == 5 ? capacity / 16 : 0;
    return tiles <= capacity - spare ? cost : 1e30;
}

TcChoice tc_choose(const sbnn_packed* p, long long M, int run, int images) {
    TcChoice best{64, 1, tc_cost(p, M, 64, images)};
    for (int bn : {128, 256}) {
        const double cost = tc_cost(p, M, bn, images);
        if (cost < best.cost) best = {bn, 1, cost};
    }
    // (every number: a layer of 16 tiles gets no clusters of 8, of which 15 run at a time, but clusters of 6.  5 x 7 x 7, 512 -> 512
    // 3x3, 72 steps: 17.9 us shared by 4, 15.0 by 6)
    for (int split = 2; split <= 8; ++split) {
        const double cost = tc_split_cost(p, M, split, run, images, best.cost);
        if (cost < best.cost) best = {64, split, cost};
    }
    return best;
}

// Whether a call is faster here than on the FMA kernels, in microseconds of both, fitted to measured times.  Layers of
// 64-1024 channels on 49 to 50176 pixels, G = 4 and 8, 0 / 50 / 70 / 90 % pruned, in short bursts (in a long loop the largest
// run at the power limit, 460 us instead of 390 here): channel-major 1x1 calls gain up to 70 %
// pruning (256 x 14 x 14, 1024 -> 1024: 1969 -> 404, 1025 -> 386, 669 -> 366 us; 9 x 14 x 14, 512 -> 512: 89 -> 12, 53 -> 12,
// 39 -> 12 us) and lose where next to nothing is left to do (the first at 90 %: 289 and 338 us; one 14 x 14 image, 256 -> 512,
// 50 %: 4.5 and 6.0 us); NHWC calls, which the FMA kernels convert first, and 3x3 calls gain nearly everywhere
// (32 x 28 x 28, 256 -> 256: 305 -> 119 us at 50 %, 120 -> 111 at 90 %; in groups of 8 106 and 111).
// `choice` is how; it is remembered with the layer for each kind of call and number of pixels.
enum Call { CALL_1X1_NHWC, CALL_1X1_CM, CALL_3X3, CALL_3X3_CM, CALL_BF16 };
double fma_us(const sbnn_packed* p, long long M, Call call) {
    const double bytes = 4.0 * M * (p->Cin + p->Cout), mem = bytes / 6.5e6;
    const double dense = 1e-6 * M * p->Cin * p->Cout;                        // 1e6 multiply-adds of the unpruned layer, a tap
    double kept = 1e-6 * M * p->nnz * p->G * (p->KH * p->KW);                // and of what is kept
    if (!p->tap_mask.empty()) kept *= (double)count_kept_taps(p) / ((double)p->nnz * p->KH * p->KW);
    if (call == CALL_3X3 || call == CALL_3X3_CM) return 25.0 + kept * (p->G >= 8 ? 0.050 : 0.075);
    if (call == CALL_1X1_CM && conv1x1_few_tiles(p, M)) return conv1x1_small_us(p, M);
    if (call == CALL_1X1_CM || (p->Cin >= 128 && M >= 2048)) {
        const double conversion = call == CALL_1X1_NHWC ? 2.0 + 8.0 * M * p->Cin / 4.5e6 : 0.0;   // to channel-major
        return 4.5 + 0.034 * kept + 0.0011 * dense + 0.65 * mem + conversion;
    }
    return 2.0 + (p->Cin >= 128 ? 2.0 : 0.0) + 0.012 * p->Cin + 0.1 * kept;
}
TcChoice decide(const sbnn_packed* p, long long M, Call call) {
    TcChoice choice = {0, 0, 0.0};
    if (call == CALL_BF16) return tc_choose(p, M, 1, 1);
    if (!p->finite || p->nnz == 0) return choice;
    choice = tc_choose(p, M, call == CALL_3X3_CM ? 3 : 1, 3);
    // (Few-pixel calls need no margin between the two models: of 4924 timed on both sides 36 run on a side that is more than 3 % slower
    // than the one an older model had picked, and 266 on one that is faster by that; the other FMA kernels' model is rougher.)
    const double least = call == CALL_1X1_CM && conv1x1_few_tiles(p, M) ? 1.0 : 0.95;
    if (std::max(tc_us(choice.cost), 4.0 * M * (p->Cin + p->Cout) / 6.5e6) >= least * fma_us(p, M, call)) choice.bn = 0;
    return choice;
}

// A block of the network (a depthwise layer with images of `side` pixels a row and the 1x1 layer behind it, N images): the
// tile of the launch that does both, bn = 0 where two launches are faster.  What one launch saves of the time of the network whose other
// blocks run as the rule has them, in microseconds, mean of 0 to 70 % pruned, at 1, 4, 6, 9, 12, 16, 28, 40 and 64 images (of 114, 158,
// 168, 200, 222, 263, 407, 467 and 668):
//   112 x 112, 32 -> 64           1.5   2.1   2.4   2.1   2.9   3.1   6.4  12.2  20.8
//   112 -> 56, 64 -> 128         -1.3   0.7   2.5   0.1   2.9   1.8  -0.3   2.7   7.7
//   56 x 56, 128 -> 128          -2.1   1.0   1.5  -0.6   2.3   2.1  -0.2   3.5  16.7
//   56 -> 28, 128 -> 256         -4.4  -1.9  -2.1   0.0   0.8   2.2  -2.7  10.6  23.6
//   28 x 28, 256 -> 256          -6.6  -3.7  -5.8  -2.8  -1.5   1.1  -6.2   5.1   8.9
// (Whole rounds of tiles on both sides make it go up and down, and a launch less saves more in a chain than the same pair called again
// and again: three of these were slower in one launch by that measure.)  Over 89 batch sizes and densities the rule is 0.06 us off the
// better side on average for a block, at most 1.9.  Tiles of 64 channels shared by 2 to 4 CTAs, for few images, save nothing: +2.0 to
// -2.1 at one image, -3 to -9 at two.
// The depthwise layer is computed again for every tile of output channels, on the split warps, so a step takes 3000 (64 or 128
// channels a tile) to 3300 cycles longer than without (twice that at stride 2, whose stages hold 8 channels); layers with
// smaller maps, more channels and less to move (14 x 14, 512 -> 512: 9 + 30 us at 64 images) stay apart.
double block_step(int bn, int stride) {
    if (stride == 2) return bn == 64 ? 6500.0 : (bn == 128 ? 7200.0 : 9500.0);
    return bn == 64 ? 4400.0 : (bn == 128 ? 5000.0 : 5600.0);
}
TcChoice decide_block(const sbnn_packed* p, int N, int side, int stride) {
    const long long out = side / stride, M = N * out * out, M_in = (long long)N * side * side, sms = device_sms();
    TcChoice best = {0, 0, 0.0};
    if (!p->finite || p->nnz == 0 || side < 28 || out < 28) return best;
    const double depthwise = 4.0 * (M_in + M) * p->Cin;              // bytes of the depthwise launch
    const double steps = p->Cin / 64.0, mem = 4.0 * (M_in * p->Cin + M * p->Cout) / 5.2e6;
    double us = 0.0;
    for (int bn : {64, 128, 256}) {
        if (bn > p->Cout || (bn == 256 && out > 28)) continue;
        const long long tiles = (M + 127) / 128 * ((p->Cout + bn - 1) / bn);
        const double cycles = (double)((tiles + sms - 1) / sms) * (steps * block_step(bn, stride) + (bn == 64 ? 1300.0 : 1000.0 + 12.0 * bn)) + 4700.0;
        const double t = std::max(cycles / 1800.0, mem);
        if (best.bn == 0 || t < us) {
            best = {bn, 1, cycles};
            us = t;
        }
    }
    const TcChoice layer = decide(p, M, CALL_1X1_CM);
    const double apart = (layer.bn ? std::max(tc_us(layer.cost), 4.0 * M * (p->Cin + p->Cout) / 6.5e6) : fma_us(p, M, CALL_1X1_CM)) + 2.0 +
                         depthwise / (depthwise < 1e8 ? 4.2e6 : 4.4e6);
    if (us >= 0.94 * apart) best.bn = 0;
    return best;
}
bool tc_profits(const sbnn_packed* p, long long M, Call call, TcChoice* choice = nullptr) {
    if (forced_choice) {
        if (choice) *choice = *forced_choice;
        return forced_choice->bn != 0;
    }
    const long long key = M * 8 + call;
    {
        std::lock_guard<std::mutex> lk(p->mu);
        auto it = p->tc_choices.find(key);
        if (it != p->tc_choices.end()) {
            if (choice) *choice = it->second;
            return it->second.bn != 0;
        }
    }
    const TcChoice c = decide(p, M, call);
    std::lock_guard<std::mutex> lk(p->mu);
    if (p->tc_choices.size() > 64) p->tc_choices.clear();
    p->tc_choices[key] = c;
    if (choice) *choice = c;
    return c.bn != 0;
}

}  // namespace

// Calls with fewer pixels can be faster here although the largest is not, and in tiles of another width: what they choose is
// looked up for every number of pixel tiles up to 512 and in steps of a 64th from there, with the fewest and with the most
// pixels of these tiles.
sbnn_status prepare_tc(const sbnn_packed* p, long long M, int images) {
    bool wanted[2] = {false, false};                  // blocks of 64 and of 128 channels
    auto look = [&](long long m) {
        for (Call call : {CALL_1X1_NHWC, CALL_1X1_CM, CALL_3X3, CALL_BF16}) {   // (channel-major 3x3 calls gain no oftener than NHWC ones)
            if (images == 1 ? call != CALL_BF16 : call == CALL_BF16 || (call == CALL_3X3) != (p->KH == 3)) continue;
            const int bn = decide(p, m, call).bn;
            if (bn) wanted[bn != 64] = true;
        }
    };
    for (long long t = (M + 127) / 128; t > 0 && !(wanted[0] && (wanted[1] || p->Cout <= 64)); t -= t > 512 ? t / 64 : 1) {
        look(std::min(M, 128 * t));
        look(128 * (t - 1) + 1);
    }
    uint4* wts = nullptr;
    PrepareScope scope;
    for (int k = 0; k < 2; ++k)
        if (wanted[k]) {
            const sbnn_status r = get_tc_weights(p, k ? 128 : 64, images, M, nullptr, &wts);
            if (r != SBNN_OK) return r;
        }
    std::lock_guard<std::mutex> lk(p->mu);
    long long& known = p->tc_prepared[images];
    known = std::max(known, M);
    return SBNN_OK;
}

namespace {

template <class T>
sbnn_status launch_tc(const sbnn_packed* p, const TcCall& c, int split, bool* done) {
    sbnn_status r = set_max_dyn_smem(reinterpret_cast<const void*>(&conv_tc_kernel<T>), 227 * 1024);
    if (r != SBNN_OK) return r;
    // The warpgroups' register shares add up to LAUNCH_REGS a thread: a build that starts with fewer must not be launched,
    // since the drain warps would wait for registers that nobody returns.  The FMA kernels run then.
    static std::atomic<int> known{0};
    int regs = known.load();
    if (regs == 0) {
        cudaFuncAttributes fa = {};
        SBNN_CUDA_TRY(cudaFuncGetAttributes(&fa, conv_tc_kernel<T>));
        known = regs = fa.numRegs;
    }
    if (regs != T::LAUNCH_REGS) return SBNN_OK;
    typename T::Args a = {};
    uint4* wts = nullptr;
    if ((r = get_tc_weights(p, T::NUC, T::IMAGES, c.M, c.st, &wts, c.ask)) != SBNN_OK || !wts) return r;
    if ((r = async_status_word(&a.status)) != SBNN_OK) return r;
    *done = true;
    if (prepare_only() || c.ask) return SBNN_OK;
    const long long ntiles_n = (p->Cout + T::BN - 1) / T::BN, total = (c.M + T::BM - 1) / T::BM * ntiles_n;
    if (total > 0x7fffffffLL) return fail(SBNN_ERR_SHAPE, "too many tiles");
    a.wts = wts; a.bias = p->d_bias; a.y = c.y; a.ldy = c.ldy; a.M = (int)c.M; a.Cin = p->Cin; a.Cout = p->Cout;
    a.steps = (p->Cin + 63) / 64 * T::TAPS; a.ntiles_m = (int)((c.M + T::BM - 1) / T::BM); a.ntiles_n = (int)ntiles_n;
    a.W = c.W; a.H = c.H; a.relu = c.relu; a.split = T::SPLIT ? split : 1;
    const bool cm = T::SRC == SRC_CM || T::SRC == SRC_CM3 || T::FUSED;
    a.ex = {c.x, cm ? 1 : p->Cin, cm ? c.ldx : 1, p->d_group_ptr, p->d_idx, p->d_val, use_tap_lists(p) ? p->d_taps : nullptr, p->G};
    CUtensorMap amap, ymap;
    if constexpr (T::FUSED) {
        using D = typename T::DW;
        a.dw_w = c.dw_w; a.dw_b = c.dw_b;
        const unsigned long long dims[2] = {(unsigned long long)c.M_in, (unsigned long long)p->Cin}, wdims[2] = {(unsigned long long)p->Cin, 9};
        const unsigned long long strides[1] = {(unsigned long long)c.ldx * 4}, wstrides[1] = {(unsigned long long)p->Cin * 4};
        const unsigned box[2] = {(unsigned)D::PB, (unsigned)D::SUB}, wbox[2] = {(unsigned)D::SUB, 9u};
        if ((r = encode_tiled_map(&amap, c.x, 4, 2, dims, strides, box)) != SBNN_OK) return r;
        if ((r = encode_tiled_map(&a.wmap, c.dw_w, 4, 2, wdims, wstrides, wbox)) != SBNN_OK) return r;
    } else if (T::SRC == SRC_IM2COL) {
        if ((r = encode_im2col_3x3_map(&amap, c.x, c.N, c.H, c.W, p->Cin, T::SUB, T::BM)) != SBNN_OK) return r;
    } else if (cm) {
        const unsigned long long dims[2] = {(unsigned long long)c.M, (unsigned long long)p->Cin};
        const unsigned long long strides[1] = {(unsigned long long)c.ldx * 4};
        const unsigned box[2] = {(unsigned)T::PIX, (unsigned)T::SUB};
        if ((r = encode_tiled_map(&amap, c.x, 4, 2, dims, strides, box)) != SBNN_OK) return r;
    } else {
        const unsigned long long dims[2] = {(unsigned long long)p->Cin, (unsigned long long)c.M};
        const unsigned long long strides[1] = {(unsigned long long)p->Cin * 4};
        const unsigned box[2] = {(unsigned)T::SUB, (unsigned)T::BM};
        if ((r = encode_tiled_map(&amap, c.x, 4, 2, dims, strides, box, 128)) != SBNN_OK) return r;
    }
    {
        const unsigned long long dims[2] = {(unsigned long long)(T::OUT_CM ? c.M : p->Cout), (unsigned long long)(T::OUT_CM ? p->Cout : c.M)};
        const unsigned long long strides[1] = {(unsigned long long)c.ldy * 4};
        const unsigned box[2] = {T::OUT_CM ? 32u : 16u, T::OUT_CM ? 16u : 32u};
        if ((r = encode_tiled_map(&ymap, c.y, 4, 2, dims, strides, box, T::OUT_CM ? 0 : 64)) != SBNN_OK) return r;
    }
    const unsigned grid = T::SPLIT ? (unsigned)(total * split) : (unsigned)std::min<long long>(total, device_sms());
    a.dm = T::SPLIT ? a.ntiles_m : (int)(grid / (unsigned)ntiles_n);
    a.dn = T::SPLIT ? 0 : (int)(grid % (unsigned)ntiles_n);
    const bool resident = !T::SPLIT && ntiles_n == 1 && a.steps * T::NU <= T::SB_MAX && a.steps * T::NU * T::B_BYTES + (T::FUSED ? T::SA_MIN : 3) * T::A_BYTES <= T::ROOM;
    a.resident_or_share = T::SPLIT ? T::COLS / 4 * 65536 / split + 1 : resident;   // (r * share / 65536 = r * chunks / split for all r <= split <= 8)
    a.sb = resident ? a.steps * T::NU : T::SB;
    a.sa = std::min(T::SA_MAX, (T::ROOM - a.sb * T::B_BYTES) / T::A_BYTES);
    if (T::FUSED) a.sa &= ~1;   // (see depthwise_split)
    const size_t smem = (size_t)a.sb * T::B_BYTES + (size_t)a.sa * T::A_BYTES + T::OUT_BYTES + T::CTRL + T::DW::OUTPUT + 1024;
    last_route = {T::BN, a.split, 0.0};
    ChainedLaunchScope early;   // before their waits the kernel's warps read the layer's own arrays only
    SBNN_CUDA_TRY(launch_kernel_cluster(conv_tc_kernel<T>, dim3(grid), dim3(T::NT), smem, c.st, (unsigned)a.split, amap, ymap, a));
    return SBNN_OK;
}

template <int SRC, bool OUT_CM>
sbnn_status dispatch_tc(const sbnn_packed* p, const TcCall& c, const TcChoice& ch, bool* done) {
    if (ch.split > 1) return launch_tc<TC<64, SRC, OUT_CM, true>>(p, c, ch.split, done);
    switch (ch.bn) {
        case 256: return launch_tc<TC<256, SRC, OUT_CM>>(p, c, 1, done);
        case 128: return launch_tc<TC<128, SRC, OUT_CM>>(p, c, 1, done);
        default: return launch_tc<TC<64, SRC, OUT_CM>>(p, c, 1, done);
    }
}

}  // namespace

// The kernel numbers pixels with ints and adds up to a tile and a row of 224 to them.
constexpr long long kMaxPixels = 0x7fffffffLL - 1024;

sbnn_status conv1x1_tc(const sbnn_packed* p, const float* x, float* y, long long M, int relu, cudaStream_t st, bool* done) {
    *done = false;
    last_route = {0, 0, 0.0};
    TcChoice ch;
    sbnn_status r;
    if (prepare_only() && (r = prepare_tc(p, M)) != SBNN_OK) return r;
    if (p->Cin % 4 || p->Cout % 4 || M > kMaxPixels || !tc_profits(p, M, CALL_1X1_NHWC, &ch)) return SBNN_OK;
    const TcCall c{x, 0, y, p->Cout, M, 0, 0, 0, relu, st};
    return dispatch_tc<SRC_NHWC, false>(p, c, ch, done);
}

// bf16 mode, dense over the masked weights.  (Activations rounded to bf16 by a pass of their own and multiplied from shared
// memory took 154 us for 1024 -> 1024 on 256 x 14 x 14, 40 of them for that pass.)
sbnn_status conv1x1_tc_bf16(const sbnn_packed* p, const float* x, float* y, long long M, int relu, cudaStream_t st, bool* done) {
    *done = false;
    last_route = {0, 0, 0.0};
    if (p->Cin % 4 || p->Cout % 4 || M > kMaxPixels) return SBNN_OK;
    if (prepare_only()) {
        const sbnn_status r = prepare_tc(p, M, 1);
        if (r != SBNN_OK) return r;
    }
    TcChoice ch;
    tc_profits(p, M, CALL_BF16, &ch);
    const TcCall c{x, 0, y, p->Cout, M, 0, 0, 0, relu, st};
    if (ch.split > 1) return launch_tc<TC<64, SRC_NHWC, false, true, 1>>(p, c, ch.split, done);
    switch (ch.bn) {
        case 256: return launch_tc<TC<256, SRC_NHWC, false, false, 1>>(p, c, 1, done);
        case 128: return launch_tc<TC<128, SRC_NHWC, false, false, 1>>(p, c, 1, done);
        default: return launch_tc<TC<64, SRC_NHWC, false, false, 1>>(p, c, 1, done);
    }
}

sbnn_status conv1x1_tc_cm(const sbnn_packed* p, const float* x, int ldx, float* y, int ldy, long long M, int relu, bool out_cm, cudaStream_t st,
                          bool* done) {
    *done = false;
    last_route = {0, 0, 0.0};
    TcChoice ch;
    sbnn_status r;
    if (prepare_only() && (r = prepare_tc(p, M)) != SBNN_OK) return r;
    if (p->Cout % 4 || M > kMaxPixels || !tc_profits(p, M, CALL_1X1_CM, &ch)) return SBNN_OK;
    const TcCall c{x, ldx, y, ldy, M, 0, 0, 0, relu, st};
    return out_cm ? dispatch_tc<SRC_CM, true>(p, c, ch, done) : dispatch_tc<SRC_CM, false>(p, c, ch, done);
}

sbnn_status conv3x3_tc(const sbnn_packed* p, const float* x, float* y, int N, int H, int W, int relu, cudaStream_t st, bool* done) {
    *done = false;
    last_route = {0, 0, 0.0};
    TcChoice ch;
    const long long M = (long long)N * H * W;
    sbnn_status r;
    if (prepare_only() && (r = prepare_tc(p, M)) != SBNN_OK) return r;
    if (p->Cin % 4 || p->Cout % 4 || M > kMaxPixels || !tc_profits(p, M, CALL_3X3, &ch)) return SBNN_OK;
    const TcCall c{x, 0, y, p->Cout, M, N, H, W, relu, st};
    return dispatch_tc<SRC_IM2COL, false>(p, c, ch, done);
}

sbnn_status conv3x3_tc_cm(const sbnn_packed* p, const float* x, int ldx, float* y, int ldy, int N, int H, int W, int relu, bool out_cm, cudaStream_t st,
                          bool* done) {
    *done = false;
    last_route = {0, 0, 0.0};
    TcChoice ch;
    const long long M = (long long)N * H * W;
    sbnn_status r;
    if (prepare_only() && (r = prepare_tc(p, M)) != SBNN_OK) return r;
    // (the entry point takes rows of up to 224 pixels)
    if (W > 224 || ldy % 4 || p->Cout % 4 || M > kMaxPixels || !tc_profits(p, M, CALL_3X3_CM, &ch)) return SBNN_OK;
    const TcCall c{x, ldx, y, ldy, M, N, H, W, relu, st};
    return out_cm ? dispatch_tc<SRC_CM3, true>(p, c, ch, done) : dispatch_tc<SRC_CM3, false>(p, c, ch, done);
}

namespace {
template <int WI, int S>
sbnn_status dispatch_dw(const sbnn_packed* p, const TcCall& c, const TcChoice& ch, bool* done) {
    if constexpr (WI < 112) {                     // (steps to share)
        if (ch.split > 1) return launch_tc<TC<64, SRC_DW, true, true, 3, WI, S>>(p, c, ch.split, done);
    }
    if constexpr (WI / S <= 28) {                 // 256 outputs
        if (ch.bn == 256) return launch_tc<TC<256, SRC_DW, true, false, 3, WI, S>>(p, c, 1, done);
    }
    if constexpr (WI / S < 112) {
        if (ch.bn == 128) return launch_tc<TC<128, SRC_DW, true, false, 3, WI, S>>(p, c, 1, done);
    }
    return ch.bn == 64 ? launch_tc<TC<64, SRC_DW, true, false, 3, WI, S>>(p, c, 1, done) : SBNN_OK;
}
}  // namespace

sbnn_status dwconv3x3_conv1x1_tc_cm(const sbnn_packed* p, const float* dw_w, const float* dw_b, const float* x, int ldx, float* y, int ldy, int N,
                                    int side, int stride, cudaStream_t st, bool* done, bool ask) {
    *done = false;
    if (!ask) last_route = {0, 0, 0.0};
    const int out = side / stride;
    const long long M = (long long)N * out * out, M_in = (long long)N * side * side;
    if ((p->Cin != 32 && p->Cin % 64) || p->Cin > kMaxDwChannels || p->Cout % 4 || M_in > kMaxPixels || !aligned16(x) || !aligned16(y) || !aligned16(dw_w) || !aligned16(dw_b)) return SBNN_OK;
    TcChoice ch;
    if (forced_choice) ch = *forced_choice;
    else ch = decide_block(p, N, side, stride);
    if (ch.split > (p->Cin + 63) / 64) return SBNN_OK;
    const TcCall c{x, ldx, y, ldy, M, N, out, out, 1, st, dw_w, dw_b, M_in, ask};
    switch (side * 4 + stride) {
        case 112 * 4 + 1: return dispatch_dw<112, 1>(p, c, ch, done);
        case 112 * 4 + 2: return dispatch_dw<112, 2>(p, c, ch, done);
        case 56 * 4 + 1: return dispatch_dw<56, 1>(p, c, ch, done);
        case 56 * 4 + 2: return dispatch_dw<56, 2>(p, c, ch, done);
        case 28 * 4 + 1: return dispatch_dw<28, 1>(p, c, ch, done);
        default: return SBNN_OK;
    }
}

sbnn_status prepare_block_tc(const sbnn_packed* p, int max_batch, int side, int stride) {
    bool wanted[2] = {false, false};                  // blocks of 64 and of 128 channels
    for (int n = max_batch; n > 0; n -= n > 64 ? n / 64 : 1) {
        const int bn = decide_block(p, n, side, stride).bn;
        if (bn) wanted[bn != 64] = true;
    }
    uint4* wts = nullptr;
    PrepareScope scope;
    for (int k = 0; k < 2; ++k)
        if (wanted[k]) {
            const sbnn_status r = get_tc_weights(p, k ? 128 : 64, 3, 0, nullptr, &wts);
            if (r != SBNN_OK) return r;
        }
    return SBNN_OK;
}

sbnn_status check_forced_choice(int tile, int split) {
    if (tile != 0 && tile != 64 && tile != 128 && tile != 256) return fail(SBNN_ERR_UNSUPPORTED, "tile=%d is not 0, 64, 128 or 256", tile);
    if (split < 1 || split > 8 || (split > 1 && tile != 64))
        return fail(SBNN_ERR_UNSUPPORTED, "split=%d is not 1, or up to 8 with 64-channel tiles", split);
    return SBNN_OK;
}
ForcedChoiceScope::ForcedChoiceScope(int tile, int split) : choice{tile, split, 0.0} { forced_choice = &choice; }
ForcedChoiceScope::~ForcedChoiceScope() { forced_choice = nullptr; }

void free_tc_weights(sbnn_packed* p) {
    for (auto& kv : p->tc_weights) cudaFree(kv.second);
    p->tc_weights.clear();
}

}  // namespace sbnn

using namespace sbnn;

extern "C" sbnn_status sbnn_debug_last_route(int* tile, int* split) {
    clear_error();
    if (!tile || !split) return fail(SBNN_ERR_NULL, "tile and split must not be NULL");
    *tile = last_route.bn;
    *split = last_route.split;
    return SBNN_OK;
}

extern "C" sbnn_status sbnn_debug_limit_images(sbnn_packed* w, long long bytes) {
    clear_error();
    if (!w) return fail(SBNN_ERR_NULL, "packed weights must not be NULL");
    if (bytes < 0) return fail(SBNN_ERR_SHAPE, "bytes must not be negative");
    w->tc_limit = (size_t)bytes;
    return SBNN_OK;
}

extern "C" sbnn_status sbnn_debug_conv_gs(const sbnn_packed* w, const float* x_dev, int ldx, float* y_dev, int ldy, int N, int H, int W, int flags,
                                          int tile, int split, void* cuda_stream) {
    clear_error();
    if (!w) return fail(SBNN_ERR_NULL, "packed weights must not be NULL");
    sbnn_status r = check_forced_choice(tile, split);
    if (r != SBNN_OK) return r;
    const int runs = (w->Cin + 63) / 64 * w->KH * (ldx ? 1 : w->KW);   // (channel-major 3x3: the taps of a kernel row stay together)
    if (runs < split) return fail(SBNN_ERR_UNSUPPORTED, "the layer has %d steps to split, not %d", runs, split);
    const ForcedChoiceScope scope(tile, split);
    last_route = {0, 0, 0.0};
    if (ldx == 0 && ldy == 0)
        r = w->KH == 3 ? sbnn_conv3x3_gs(w, x_dev, y_dev, N, H, W, flags, cuda_stream) : sbnn_conv1x1_gs(w, x_dev, y_dev, N, H, W, flags, cuda_stream);
    else if (w->KH == 3)
        r = sbnn_conv3x3_gs_cm(w, x_dev, ldx, y_dev, ldy, N, H, W, flags, cuda_stream);
    else if (N < 0 || H < 0 || W < 0 || (long long)N * H * W > 0x7fffffff)
        r = fail(SBNN_ERR_SHAPE, "bad shape %dx%dx%d", N, H, W);
    else
        r = sbnn_conv1x1_gs_cm(w, x_dev, ldx, y_dev, ldy, N * H * W, flags, 0, 0, 0, 0, cuda_stream);
    if (r == SBNN_OK && (last_route.bn != tile || (tile && last_route.split != split)))
        return fail(SBNN_ERR_UNSUPPORTED, "the tensor-core kernel does not take this call; it ran on another kernel");
    return r;
}
