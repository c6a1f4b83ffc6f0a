// 3x3 convolutions of the learned stage on the tcgen05 tensor cores, tiled: the
// kernels that run every layer of the network (at most 64 channels on either
// side); conv_tc.cu holds the general form for more input channels.
//
// A convolution is the contraction D[m][n] = sum_k A[m][k] B[n][k], m an output
// pixel, n an output channel, k = (input channel, ky, kx) (the input gradient:
// channels exchanged, A the output gradient through the transposed stencil, B the
// weights transposed).  Its cost is building A: nine shifted copies of every
// input value.  Here the nine copies are made from registers.  A tile is 128
// output pixels (2 rows x 64 or 4 rows x 32).  A producer thread reads 8 pixels
// of one input row and channel (float4), rounds them to bfloat16, forms the three
// x-shifted 16-byte chunks and stores them as the k rows of every (output row,
// ky) that needs this input row: one global read feeds up to 18 chunks, with no
// index arithmetic per value.  In shared memory a k row is 64 consecutive
// pixels, 128 bytes, in the 128-byte swizzle: the tensor core reads the
// rows as an M-major operand for the convolution and the input gradient, and the
// same image as a K-major operand (M = k, K = pixels) for the weight gradient.
//
// One persistent CTA per SM, warps specialised: 8 produce A (three stages of 16
// channels, 144 k rows), 1 issues the MMAs and commits them to the stages'
// mbarriers, 4 load the weights once (all k, 72 KB), then read finished accumulators
// back (two of them, so that the epilogue of one tile runs under the MMAs of the
// next) and apply bias, relu, skip, or the gradient's mask, sum and 2 x 2 pooling.
//
// k runs in the order (channel, ky, kx), 16 per MMA, as in the general form: the
// same products enter the same accumulation steps, so the results are the same
// to the last bit.  (Any other order moves an activation's float32 sum by an ulp,
// now and then across a bfloat16 rounding boundary, and six layers turn that into
// 5e-4 of the output.)
//
// What bounds it, measured by leaving parts out (64 -> 32 channels onto 1088^2 pixels,
// 200 us, 218 TFLOP/s; SM clock 2.07 GHz): the MMAs, 140 us for the 2196 of an SM, 130
// cycles each; on top of them the stores of A 12 us, the epilogue 11 us, the loads'
// latency 37 us.  The weights and the launch cost some 10 us a kernel, which is most of a
// layer on a batch of 32 crops of 64 x 64; as dependent launches they run under the
// kernel before (forward and gradients of that batch 0.50 ms, before these kernels
// 4.28 ms).  One forward pass on 1088^2: 0.68 ms, before 2.98 ms.
//
// Every wait on an mbarrier is bounded; on timeout the kernel sets *err, the issuer and
// the epilogue leave their loops, the producers run to their end without waiting, the
// issuer waits (bounded) for its last commit, and the tensor memory is freed.
#include <algorithm>
#include <cstdint>

#include "mxp_internal.h"

namespace mxp {

namespace {

constexpr long long kPollLimit = 1ll << 22;   // try_wait polls (each suspends briefly): well over a second
constexpr int kProd = 256;                    // producer threads (warps 5 .. 12)
constexpr int kThreads = 128 + 32 + kProd;
constexpr int kStageCh = 16;                  // input channels per stage
constexpr int kStageK = 9 * kStageCh;         // its k rows
constexpr int kBlk = kStageK * 128;           // bytes of one 64-pixel block of a stage
constexpr int kMaxCh = 64;
constexpr int kSlots = 3;                     // stages in shared memory

enum ConvMode { kF1, kF2, kFU, kD1, kD2 };    // forward stride 1, 2, upsampled; input gradient stride 1, 2

__device__ __forceinline__ uint32_t su32(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void bar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(bar)), "r"(count));
}

__device__ __forceinline__ void bar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(bar)) : "memory");
}

// Waits until the phase of the given parity has completed; false on timeout or
// when another role gave up.  The lanes of a warp may differ in that, and must not part
// over it in front of warp-wide instructions: the producers go on either way (to the end
// of their tiles without waiting, into their own shared memory), the MMA issuer is one
// lane, the epilogue warps vote.
__device__ __forceinline__ bool bar_wait(uint64_t *bar, unsigned parity, volatile int *abort)
{
    const uint32_t a = su32(bar);
    for (long long it = 0; it < kPollLimit; ++it) {
        uint32_t done = 0;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
        if (*abort) return false;
    }
    *abort = 1;
    return false;
}

// true in all of the 4 epilogue warps when it is in each (they meet in the pooling
// epilogue, so they leave their loop together)
__device__ __forceinline__ bool all_of_128(bool ok)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, 128, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((int)ok)
        : "memory");
    return r != 0;
}

// Programmatic dependent launch: the next kernel's set-up (barriers, tensor memory,
// weights) may run under this kernel's last tiles; its activations wait for this one.
// It is let go when this kernel no longer waits itself: before that, the CTAs of kernels
// further on took SMs and shared memory from the next one's (forward pass on 30 x 34
// 82 -> 71 us, on 1088^2 701 -> 676 us, with gradients on 32 crops of 64^2 545 -> 534 us).
__device__ __forceinline__ void wait_for_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void commit_to(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
                 : "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, int acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}

// Shared-memory descriptor: address and byte offsets in 16-byte units, version 1;
// swz = 2 for the 128-byte swizzle, 0 for none.
__device__ __forceinline__ uint64_t desc(uint32_t addr, uint32_t lbo, uint32_t sbo, uint64_t swz)
{
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46) | (swz << 61);
}

// kind::f16: float32 accumulator, bfloat16 operands; amn: A is M-major
__device__ __forceinline__ uint32_t idesc_bf16(int n, int amn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)amn << 15) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
}

__device__ __forceinline__ uint32_t pk(float lo, float hi)
{
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// Predicated loads, zero where the predicate is false, issued where they stand and
// straight into their registers: written as conditions, the compiler moves the loaded
// values when the branches join, and waits for them there.
// Plain loads, not .nc: a chained kernel starts while its predecessor still writes what
// it will read, and .nc is for memory that is read-only as long as the kernel runs.
__device__ __forceinline__ void ld4(float *v, const float *p, bool ok)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\tmov.f32 %2, 0f00000000;\n\tmov.f32 %3, 0f00000000;\n\t"
        "@p ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=&f"(v[0]), "=&f"(v[1]), "=&f"(v[2]), "=&f"(v[3])
        : "l"(p), "r"((int)ok));
}

__device__ __forceinline__ void ld1(float &v, const float *p, bool ok)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %2, 0;\n\t"
        "mov.f32 %0, 0f00000000;\n\t"
        "@p ld.global.f32 %0, [%1];\n\t}"
        : "=&f"(v)
        : "l"(p), "r"((int)ok));
}

__device__ __forceinline__ float ldg_now(const float *p)
{
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}

// Input values behind 8 output pixels of one input row: v[1 .. LEN], with the
// neighbours v[0] and v[LEN + 1].
template <int M> struct Chunk {
    static constexpr int LEN = (M == kF2) ? 16 : (M == kFU || M == kD2) ? 4 : 8;
    float v[LEN + 2];
    __device__ __forceinline__ static int xstart(int ox) { return M == kF2 ? 2 * ox : (M == kFU || M == kD2) ? ox / 2 : ox; }

    // row: the channel's input row (ok = false: all zero); ws its length; first / last:
    // the lane to the left / right does not hold the neighbouring chunk of this row
    template <bool VEC>
    __device__ __forceinline__ void load(const float *row, bool ok, int xs, int ws, bool first, bool last)
    {
        const float *x = row + xs;
        if (VEC) {
#pragma unroll
            for (int q = 0; q < LEN / 4; ++q) ld4(&v[1 + 4 * q], x + 4 * q, ok && xs + 4 * q < ws);
        } else {
#pragma unroll
            for (int q = 0; q < LEN; ++q) ld1(v[1 + q], x + q, ok && xs + q < ws);
        }
        ld1(v[0], x - 1, ok && first && M != kD2 && xs > 0 && xs - 1 < ws);
        if (M != kF2) ld1(v[LEN + 1], x + LEN, ok && last && xs + LEN < ws);
    }
    __device__ __forceinline__ void exchange(bool first, bool last)
    {
        const float l = __shfl_up_sync(0xffffffffu, v[LEN], 1), r = __shfl_down_sync(0xffffffffu, v[1], 1);
        if (!first) v[0] = l;
        if (!last) v[LEN + 1] = r;
    }
    // 8 bfloat16 of the k row with x tap kx
    __device__ __forceinline__ uint4 shifted(int kx) const
    {
        const float *s = v + 1;
        if (M == kF2) {        // in[2 ox + kx - 1]
            if (kx == 1) return make_uint4(pk(s[0], s[2]), pk(s[4], s[6]), pk(s[8], s[10]), pk(s[12], s[14]));
            if (kx == 2) return make_uint4(pk(s[1], s[3]), pk(s[5], s[7]), pk(s[9], s[11]), pk(s[13], s[15]));
            return make_uint4(pk(v[0], s[1]), pk(s[3], s[5]), pk(s[7], s[9]), pk(s[11], s[13]));
        } else if (M == kFU) { // in[(ox + kx - 1) >> 1]
            if (kx == 1) return make_uint4(pk(s[0], s[0]), pk(s[1], s[1]), pk(s[2], s[2]), pk(s[3], s[3]));
            if (kx == 0) return make_uint4(pk(v[0], s[0]), pk(s[0], s[1]), pk(s[1], s[2]), pk(s[2], s[3]));
            return make_uint4(pk(s[0], s[1]), pk(s[1], s[2]), pk(s[2], s[3]), pk(s[3], s[4]));
        } else if (M == kD2) { // g[(ox + 1 - kx) / 2] where that is whole
            if (kx == 1) return make_uint4(pk(s[0], 0.f), pk(s[1], 0.f), pk(s[2], 0.f), pk(s[3], 0.f));
            if (kx == 0) return make_uint4(pk(0.f, s[1]), pk(0.f, s[2]), pk(0.f, s[3]), pk(0.f, s[4]));
            return make_uint4(pk(0.f, s[0]), pk(0.f, s[1]), pk(0.f, s[2]), pk(0.f, s[3]));
        } else {               // forward in[ox + kx - 1], gradient g[ox + 1 - kx]
            const int d = (M == kD1) ? 2 - kx : kx;
            const float *t = v + d;
            return make_uint4(pk(t[0], t[1]), pk(t[2], t[3]), pk(t[4], t[5]), pk(t[6], t[7]));
        }
    }
};

// Input rows of a tile of TH output rows from oy0: row index sr stands for input
// row ybase + sr; the (output row r, ky) pairs reading it are those with
// src(r, ky) == sr.
template <int M, int TH> struct Rows {
    static constexpr int SR = (M == kF2) ? 2 * TH + 1 : (M == kFU) ? (TH == 1 ? 2 : TH / 2 + 2) : (M == kD2) ? TH / 2 + 1 : TH + 2;
    __device__ __forceinline__ static int ybase(int oy0)
    {
        return M == kF2 ? 2 * oy0 - 1 : M == kFU ? (oy0 - 1) >> 1 : M == kD2 ? oy0 / 2 : oy0 - 1;
    }
    // -1: this (r, ky) reads no row (zero)
    __device__ __forceinline__ static int src(int oy0, int r, int ky)
    {
        if (M == kF2) return 2 * r + ky;
        if (M == kFU && TH > 1) return ((r + ky - 1) >> 1) + 1;          // oy0 is even
        if (M == kFU) return ((oy0 + ky - 1) >> 1) - ((oy0 - 1) >> 1);
        if (M == kD2) return ((r + 1 - ky) & 1) ? -1 : (r + 1 - ky) / 2;
        if (M == kD1) return r + 2 - ky;
        return r + ky;
    }
};

// Address of 16-byte chunk c (8 pixels) of k row k in a 64-pixel block.
__device__ __forceinline__ uint32_t row_chunk(int k, int c) { return (uint32_t)(k * 128 + ((c ^ (k & 7)) << 4)); }

struct ConvArgs {
    const float *in;
    int Cin, Hs, Ws;
    const __nv_bfloat16 *w;
    const float *bias;
    int Cout, Ho, Wo;
    int relu;
    ConvOut o;
    int ntx, nty, ntiles;
    int NT, KT;              // N tile (16, 32, 64); k rows in all, padded per stage
    bool chain;
    unsigned *err;
};

struct TilePos {
    int img, oy0, ox0;
};
// Steps whose input values are in flight ahead of the one being stored: two where
// the registers allow it, since a step is shorter than a load under traffic.
template <int M> constexpr int ahead() { return M == kF2 ? 1 : 2; }

// Walks a CTA's (tile, 16-channel group) steps: tiles blockIdx.x, + gridDim.x, ...
// as (column, row, image), advanced by additions.
struct Cursor {
    int left, s, x, y, img;          // tiles left; group; tile coordinates
    int dx, dy, dimg, ntx, nty;
    __device__ __forceinline__ Cursor(int ntiles, int ntx_, int nty_) : s(0), ntx(ntx_), nty(nty_)
    {
        const int t = blockIdx.x, d = gridDim.x;
        left = t < ntiles ? (ntiles - t + d - 1) / d : 0;
        x = t % ntx;
        y = t / ntx % nty;
        img = t / ntx / nty;
        dx = d % ntx;
        dy = d / ntx % nty;
        dimg = d / ntx / nty;
    }
    __device__ __forceinline__ void next(int ngrp)
    {
        if (++s == ngrp) {
            s = 0;
            left -= left > 0;
            x += dx;
            y += dy;
            img += dimg;
            if (x >= ntx) { x -= ntx; ++y; }
            if (y >= nty) { y -= nty; ++img; }
        }
    }
    __device__ __forceinline__ TilePos pos(int TH, int TW) const { return TilePos{img, y * TH, x * TW}; }
};

// One stage's (or 16-channel group's) share of a producer warp: NI items, an item
// one input row of 32 / NC channels, 8 pixels per lane.  The row is uniform over
// the warp, so the (output row, ky) pairs that need it are uniform branches; 8 lanes
// of a quarter warp write 8 different 16-byte columns (with 4 chunks a row the lanes'
// two channels are 4 apart: their swizzles differ in the other half).  The loop over
// stages is bound by instructions, so what depends on the thread only is made once.
template <int M, int TW, int TH> struct Items {
    static constexpr int NC = TW / 8, SR = Rows<M, TH>::SR, CPW = 32 / NC;
    static constexpr int TOTAL = kStageCh / CPW * SR, NI = (TOTAL + kProd / 32 - 1) / (kProd / 32);
    static constexpr bool TABLE = M != kF2;      // kF2 has no registers left for it
    int pc;
    int sr[NI], c0[NI], ci[NI];                  // input row, first channel of the warp, the lane's channel
    uint32_t sw[TABLE ? NI : 1][8];              // its k rows' chunk offsets, by tap mod 8

    __device__ __forceinline__ uint32_t offset(int it, int t) const
    {
        // k = 9 ci + tap: byte 128 k, 16-byte column pc ^ (k & 7), k & 7 = (ci + tap) & 7
        return TABLE ? sw[TABLE ? it : 0][t & 7] + t * 128
                     : (uint32_t)(ci[it] * 1152 + t * 128 + ((pc ^ ((ci[it] + t) & 7)) << 4));
    }
    __device__ __forceinline__ Items(int pwarp, int lane)
    {
        pc = lane % NC;
#pragma unroll
        for (int it = 0; it < NI; ++it) {
            const int wi = it * (kProd / 32) + pwarp, cg = wi / SR;
            sr[it] = (wi + cg) % SR;             // rows feed one or two output rows: spread them over the warps
            c0[it] = wi < TOTAL ? cg * CPW : kStageCh;
            ci[it] = wi < TOTAL ? cg * CPW + (NC == 8 ? lane >> 3 : (lane >> 3) + (lane & 4)) : kStageCh;
            if (TABLE) {
#pragma unroll
                for (int u = 0; u < 8; ++u) sw[it][u] = (uint32_t)(ci[it] * 1152 + ((pc ^ ((ci[it] + u) & 7)) << 4));
            }
        }
    }

    // channels ch0 .. ch0 + nch - 1 of image p.img (nch <= 0: none).  No branches around
    // the loads: a register that is loaded on one side only is copied where they join.
    template <bool VEC>
    __device__ __forceinline__ void load(Chunk<M> (&c)[NI], const float *in, const TilePos &p, int Cin, int ch0, int nch,
                                         int Hs, int Ws) const
    {
        const int yb = Rows<M, TH>::ybase(p.oy0), xs = Chunk<M>::xstart(p.ox0 + 8 * pc);
        const float *plane = in + ((int64_t)p.img * Cin + ch0) * Hs * Ws;
#pragma unroll
        for (int it = 0; it < NI; ++it) {
            const int ys = yb + sr[it];
            const bool ok = ci[it] < nch && ys >= 0 && ys < Hs;
            c[it].template load<VEC>(plane + ((int64_t)ci[it] * Hs + ys) * Ws, ok, xs, Ws, pc == 0, pc == NC - 1);
        }
    }

    // Store the chunks as k rows of `base`.  PIX: pixels beyond the output's edge are
    // stored as zero (the contraction runs over pixels).
    template <bool PIX>
    __device__ __forceinline__ void store(Chunk<M> (&c)[NI], uint8_t *base, const TilePos &p, int nch, int Ho, int Wo) const
    {
#pragma unroll
        for (int it = 0; it < NI; ++it) {
            if (c0[it] >= nch) continue;
            c[it].exchange(pc == 0, pc == NC - 1);
            if (ci[it] >= nch) continue;
            uint4 s[3];
#pragma unroll
            for (int kx = 0; kx < 3; ++kx) s[kx] = c[it].shifted(kx);
            if (PIX) {
                const int nv = Wo - (p.ox0 + 8 * pc);
                if (nv < 8) {
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        uint32_t *q = reinterpret_cast<uint32_t *>(&s[kx]);
#pragma unroll
                        for (int h = 0; h < 4; ++h)
                            q[h] = nv <= 2 * h ? 0u : nv == 2 * h + 1 ? (q[h] & 0xFFFFu) : q[h];
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < TH; ++r) {
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) {
                    if (Rows<M, TH>::src(p.oy0, r, ky) != sr[it]) continue;
                    // 64-pixel block of the output row; the second row of a block is its other half
                    const int b = TW == 64 ? r : r >> 1;
                    const uint32_t half = TW == 64 ? 0u : (uint32_t)(r & 1) * 64u;
                    const bool live = !PIX || p.oy0 + r < Ho;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx)
                        *reinterpret_cast<uint4 *>(base + b * kBlk + (offset(it, ky * 3 + kx) ^ half)) =
                            live ? s[kx] : make_uint4(0, 0, 0, 0);
                }
            }
        }
    }
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
        "%13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Weights as the K-major operand, no swizzle: 8 x 16-byte core matrices, k groups
// 128 bytes apart, channel groups KT * 16 bytes apart.
__device__ __forceinline__ void load_weights(uint8_t *sB, const ConvArgs &a, bool grad, int tid, int nthr)
{
    const int K = a.Cin * 9, KT = a.KT;
    auto off = [&](int n, int k) { return (uint32_t)((n >> 3) * KT * 16 + (k >> 3) * 128 + (n & 7) * 16 + (k & 7) * 2); };
    const bool v16 = !grad && K % 8 == 0 && (reinterpret_cast<uintptr_t>(a.w) & 15) == 0;
    if (v16) {                                             // W[co = n][k]: whole 16-byte groups
        const int per = KT / 8;
        for (int i = tid; i < a.NT * per; i += nthr) {
            const int n = i / per, kg = i % per;
            uint4 v = make_uint4(0, 0, 0, 0);
            if (n < a.Cout && kg * 8 < K) v = *reinterpret_cast<const uint4 *>(a.w + (int64_t)n * K + kg * 8);
            *reinterpret_cast<uint4 *>(sB + off(n, kg * 8)) = v;
        }
        return;
    }
    const __nv_bfloat16 z = __float2bfloat16_rn(0.f);
    if (!grad) {
        for (int i = tid; i < a.NT * KT; i += nthr) {
            const int n = i / KT, k = i % KT;
            *reinterpret_cast<__nv_bfloat16 *>(sB + off(n, k)) = (n < a.Cout && k < K) ? a.w[(int64_t)n * K + k] : z;
        }
    } else {                                               // W[co][ci = n][tap], k = co * 9 + tap
        if (a.NT != a.Cout || KT != K) {                   // channels or k rows that fill up: zero
            for (int i = tid; i < a.NT * KT / 8; i += nthr) reinterpret_cast<uint4 *>(sB)[i] = make_uint4(0, 0, 0, 0);
            asm volatile("bar.sync 1, 128;" ::: "memory");
        }
        const int row = a.Cout * 9;
        if (row % 8 == 0 && (reinterpret_cast<uintptr_t>(a.w) & 15) == 0) {
#pragma unroll 4
            for (int i = tid; i < a.Cin * row / 8; i += nthr) {
                const uint4 v = reinterpret_cast<const uint4 *>(a.w)[i];
                const int co = i * 8 / row, r0 = i * 8 - co * row;
                const __nv_bfloat16 *e = reinterpret_cast<const __nv_bfloat16 *>(&v);
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int n = (r0 + u) / 9, k = co * 9 + (r0 + u) - 9 * n;
                    *reinterpret_cast<__nv_bfloat16 *>(sB + off(n, k)) = e[u];
                }
            }
        } else {
            for (int i = tid; i < a.Cin * row; i += nthr) {
                const int co = i / row, r = i % row, n = r / 9, k = co * 9 + r % 9;
                *reinterpret_cast<__nv_bfloat16 *>(sB + off(n, k)) = a.w[i];
            }
        }
    }
}

struct ConvShared {
    uint64_t full[kSlots], empty[kSlots], acc_full[2], acc_empty[2], wready;
    uint32_t tmem;
    int abort;
    float bias[kMaxCh];
    float pool[16][32];      // first rows' pair sums of 16 channels (2 x 2 pooling)
};

template <int M, int TW, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) k_conv_tile(const __grid_constant__ ConvArgs a)
{
    constexpr int TH = 128 / TW;
    constexpr bool GRAD = M == kD1 || M == kD2;
    extern __shared__ uint8_t raw[];
    __shared__ ConvShared sh;
    uint8_t *sA = raw + ((1024u - (su32(raw) & 1023u)) & 1023u);   // [kSlots][2 blocks][kBlk]
    uint8_t *sB = sA + kSlots * 2 * kBlk;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nst = (a.Cin + kStageCh - 1) / kStageCh;
    const int NT = a.NT, tcols = 2 * NT < 32 ? 32 : 2 * NT;

    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sh.tmem)), "r"(tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < kSlots; ++s) {
            bar_init(&sh.full[s], kProd / 32);
            bar_init(&sh.empty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            bar_init(&sh.acc_full[s], 1);
            bar_init(&sh.acc_empty[s], 4);
        }
        bar_init(&sh.wready, 4);
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (M == kD2) {
        // the (row, ky) pairs without a source stay zero for the whole kernel
        for (int i = tid; i < kSlots * 2 * kBlk / 16; i += kThreads) reinterpret_cast<uint4 *>(sA)[i] = make_uint4(0, 0, 0, 0);
        fence_async_smem();
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = sh.tmem;
    volatile int *abort = &sh.abort;
    const int t0 = blockIdx.x, dt = gridDim.x;

    if (warp >= 5) {
        // ------------------------------------------------ producers
        const int ptid = tid - 160, pwarp = warp - 5;
        using It = Items<M, TW, TH>;
        const It items(pwarp, lane);
        constexpr int D = ahead<M>();
        Chunk<M> q[D + 1][It::NI];
        Cursor at(a.ntiles, a.ntx, a.nty), ld = at;
        auto load = [&](Chunk<M> (&c)[It::NI]) {
            items.template load<VEC>(c, a.in, ld.pos(TH, TW), a.Cin, ld.s * kStageCh,
                                     ld.left > 0 ? min(kStageCh, a.Cin - ld.s * kStageCh) : 0, a.Hs, a.Ws);
            ld.next(nst);
        };
        int slot = 0, par = 1;
        // store one stage while the values of a later one are on their way; false at the end
        auto stage = [&](Chunk<M> (&now)[It::NI], Chunk<M> (&later)[It::NI]) -> bool {
            if (at.left <= 0) return false;
            load(later);
            const TilePos p = at.pos(TH, TW);
            const int nch = min(kStageCh, a.Cin - at.s * kStageCh);
            // parity 1 of a fresh barrier counts as complete: the first round finds its slots free
            bar_wait(&sh.empty[slot], par, abort);
            uint8_t *base = sA + slot * 2 * kBlk;
            items.template store<false>(now, base, p, nch, a.Ho, a.Wo);
            const int k0 = nch * 9, k1 = (k0 + 15) / 16 * 16;
            for (int i = ptid; i < (k1 - k0) * 16; i += kProd) {      // k rows that fill up the last MMA
                const int k = k0 + i / 16, c = i % 16;
                *reinterpret_cast<uint4 *>(base + (c >> 3) * kBlk + row_chunk(k, c & 7)) = make_uint4(0, 0, 0, 0);
            }
            fence_async_smem();
            __syncwarp();
            if (lane == 0) bar_arrive(&sh.full[slot]);
            if (++slot == kSlots) {
                slot = 0;
                par ^= 1;
            }
            at.next(nst);
            return true;
        };
        wait_for_previous();
#pragma unroll
        for (int d = 0; d < D; ++d) load(q[d]);
        // buffers by name, not shifted: a move of a value still in flight would wait for it
        if constexpr (D == 1) {
            while (stage(q[0], q[1]) && stage(q[1], q[0])) {}
        } else {
            while (stage(q[0], q[2]) && stage(q[1], q[0]) && stage(q[2], q[1])) {}
        }
    } else if (warp == 4) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            const uint32_t id = idesc_bf16(NT, 1);
            bool ok = bar_wait(&sh.wready, 0, abort);
            int n = 0, slot = 0, par = 0, last = -1, lastpar = 0;
            for (int t = t0; ok && t < a.ntiles; t += dt, ++n) {
                const int acc = n & 1;
                if (n >= 2) ok = bar_wait(&sh.acc_empty[acc], ((n >> 1) - 1) & 1, abort);
                for (int s = 0; ok && s < nst; ++s) {
                    ok = bar_wait(&sh.full[slot], par, abort);
                    if (!ok) break;
                    tc_after();
                    // a lone warp runs at instruction latency: descriptors by addition, unrolled
                    // (with a loop that formed them the MMAs of a tile took 1.8 times as long)
                    const int nch = min(kStageCh, a.Cin - s * kStageCh);
                    const uint32_t dcol = tmem + acc * NT;
                    const uint64_t ad = desc(su32(sA + slot * 2 * kBlk), kBlk, 1024, 2);
                    const uint64_t bd = desc(su32(sB) + s * (kStageK / 8) * 128, 128, a.KT * 16, 0);
                    if (nch == kStageCh) {
#pragma unroll
                        for (int q = 0; q < kStageK / 16; ++q) mma_bf16(dcol, ad + q * 128, bd + q * 16, id, s > 0 || q > 0);
                    } else {
                        for (int q = 0; q < (nch * 9 + 15) / 16; ++q)
                            mma_bf16(dcol, ad + q * 128, bd + q * 16, id, s > 0 || q > 0);
                    }
                    commit_to(&sh.empty[slot]);
                    if (s == nst - 1) commit_to(&sh.acc_full[acc]);
                    last = slot;
                    lastpar = par;
                    if (++slot == kSlots) {
                        slot = 0;
                        par ^= 1;
                    }
                }
            }
            // before the tensor memory is freed: every MMA issued has completed
            if (last >= 0) {
                volatile int none = 0;
                bar_wait(&sh.empty[last], lastpar, &none);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ weights, then epilogue
        load_weights(sB, a, GRAD, tid, 128);
        if (tid < kMaxCh) sh.bias[tid] = (a.bias && tid < a.Cout) ? a.bias[tid] : 0.f;
        fence_async_smem();
        __syncwarp();
        if (lane == 0) bar_arrive(&sh.wready);
        asm volatile("bar.sync 1, 128;" ::: "memory");
        wait_for_previous();
        const int64_t hw = (int64_t)a.Ho * a.Wo;
        const int r = TW == 64 ? warp >> 1 : warp, px = TW == 64 ? (warp & 1) * 32 + lane : lane;
        Cursor at(a.ntiles, a.ntx, a.nty);
        for (int n = 0; at.left > 0; ++n, at.next(1)) {
            const TilePos p = at.pos(TH, TW);
            const int acc = n & 1;
            if (!all_of_128(bar_wait(&sh.acc_full[acc], (n >> 1) & 1, abort))) break;
            tc_after();
            const int oy = p.oy0 + r, ox = p.ox0 + px;
            const bool valid = oy < a.Ho && ox < a.Wo;
            const int64_t rr = (int64_t)oy * a.Wo + ox;
            const uint32_t taddr = tmem + acc * NT + ((uint32_t)(warp * 32) << 16);
            for (int c0 = 0; c0 < a.Cout; c0 += 16) {
                const int nc = min(16, a.Cout - c0);
                const int64_t q0 = ((int64_t)p.img * a.Cout + c0) * hw + rr;
                // reads of the epilogue's other operands before its first store
                float ad[16], mk[16];
                if (valid && !a.o.pool) {
                    if (a.o.add) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j < nc) ad[j] = ldg_now(a.o.add + q0 + (int64_t)j * hw);
                    }
                    if (GRAD && a.o.mask) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j < nc) mk[j] = ldg_now(a.o.mask + q0 + (int64_t)j * hw);
                    }
                }
                uint32_t d[16];
                tmem_ld16(taddr + c0, d);
                if (GRAD && a.o.pool) {
                    // sum of each 2 x 2 block in the order of the plain sum: the warps of the
                    // block's first row hand their pair sums to those of its second row
                    const bool top = (r & 1) == 0;
                    const int at = (TW == 64 ? (warp & 1) : (warp >> 1)) * 16 + lane / 2;
                    float s[16];
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float v = __uint_as_float(d[j]);
                        const float e = __shfl_down_sync(0xffffffffu, v, 1);
                        s[j] = e;
                        if (top && (lane & 1) == 0) sh.pool[j][at] = v + e;
                    }
                    const bool owner = !top && (lane & 1) == 0 && valid;
                    const int64_t hw4 = hw / 4;
                    const int64_t q4 = ((int64_t)p.img * a.Cout + c0) * hw4 + (int64_t)(oy / 2) * (a.Wo / 2) + ox / 2;
                    if (owner && a.o.mask) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (j < nc) mk[j] = ldg_now(a.o.mask + q4 + j * hw4);
                    }
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                    if (owner) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            if (j >= nc) continue;
                            float v = sh.pool[j][at] + __uint_as_float(d[j]);
                            v += s[j];
                            if (a.o.mask && !(mk[j] > 0.f)) v = 0.f;
                            a.o.out[q4 + j * hw4] = v;
                        }
                    }
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                } else if (valid) {
                    float *o1 = a.o.out + q0, *o2 = a.o.out2 + q0;
                    if (!GRAD) {
#pragma unroll
                        for (int j = 0; j < 16; ++j) {
                            float v = __uint_as_float(d[j]);
                            if (a.bias) v += sh.bias[c0 + j];
                            if (a.relu) v = fmaxf(v, 0.f);
                            d[j] = __float_as_uint(v);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (a.o.add) d[j] = __float_as_uint(__uint_as_float(d[j]) + ad[j]);
                    }
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (j >= nc) continue;
                        const float v = __uint_as_float(d[j]);
                        o1[(int64_t)j * hw] = GRAD && a.o.mask && !(mk[j] > 0.f) ? 0.f : v;
                        if (a.o.out2) o2[(int64_t)j * hw] = GRAD ? v : v + ad[j];
                    }
                }
            }
            tc_before();
            __syncwarp();
            if (lane == 0) bar_arrive(&sh.acc_empty[acc]);
        }
    }
    tc_before();
    __syncthreads();
    if (tid == 0 && sh.abort) atomicExch(a.err, 1u);
    if (warp == 4) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
}

// Weight gradient gW[co][k] = sum over pixels of X[p][k] g[co][p], X the shifted input
// copies: M = k (128 per accumulator, up to 5 of them), N = co, K = pixels, 64 per
// step.  A step holds every k row of 64 pixels (72 KB) and the gradients of the same
// pixels; all accumulators stay in tensor memory over the CTA's pixel tiles and are
// added to gW once at the end.  The producers read the gradient tiles anyway and sum
// them for the bias gradient: each CTA leaves its sums, and k_bias_sum adds those of all
// layers in the CTAs' order, so that the same inputs give the same bits (with atomicAdd
// they did not; added up by the last CTA of each layer it cost 3 to 5 us a layer, in one
// launch behind them all 2 to 4 us in all).
struct WgradArgs {
    const float *x;
    int Cin, Hs, Ws;
    const float *g;
    int Cout, Ho, Wo;
    int vecg;
    float *gw, *part;        // part nullable: [CTA][kMaxCh] sums of g
    int ntx, nty, ntiles, NT, nmb;
    bool chain;
    unsigned *err;
};

struct WgradShared {
    uint64_t full[2], empty[2], done;
    uint32_t tmem;
    int abort;
};

template <int M, int TW, bool VEC>
__global__ void __launch_bounds__(kThreads, 1) k_wgrad_tile(const __grid_constant__ WgradArgs a)
{
    constexpr int TH = 64 / TW;
    extern __shared__ uint8_t raw[];
    __shared__ WgradShared sh;
    uint8_t *smem = raw + ((1024u - (su32(raw) & 1023u)) & 1023u);
    const int NT = a.NT, asz = a.nmb * 128 * 128, slotsz = asz + NT * 128;    // [A | B] per slot
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int K = a.Cin * 9, ngrp = (a.Cin + kStageCh - 1) / kStageCh;
    int tcols = 32;
    while (tcols < a.nmb * NT) tcols *= 2;

    if (warp == 4) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sh.tmem)), "r"(tcols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) {
            bar_init(&sh.full[s], kProd / 32);
            bar_init(&sh.empty[s], 1);
        }
        bar_init(&sh.done, 1);
        sh.abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_before();
    __syncthreads();
    tc_after();
    const uint32_t tmem = sh.tmem;
    volatile int *abort = &sh.abort;
    const int t0 = blockIdx.x, dt = gridDim.x;

    if (warp >= 5) {
        const int ptid = tid - 160, pwarp = warp - 5;
        using It = Items<M, TW, TH>;
        const It items(pwarp, lane);
        constexpr int D = ahead<M>();
        Chunk<M> q[D + 1][It::NI];
        float bsum[2] = {0.f, 0.f};
        Cursor at(a.ntiles, a.ntx, a.nty), ld = at;
        auto load = [&](Chunk<M> (&c)[It::NI]) {
            items.template load<VEC>(c, a.x, ld.pos(TH, TW), a.Cin, ld.s * kStageCh,
                                     ld.left > 0 ? min(kStageCh, a.Cin - ld.s * kStageCh) : 0, a.Hs, a.Ws);
            ld.next(ngrp);
        };
        // this thread's 8 pixels of two gradient channels
        const int gc = ptid & 7, gco = ptid >> 3;
        float gv[2][8];
        int slot = 0, par = 1;
        auto stage = [&](Chunk<M> (&now)[It::NI], Chunk<M> (&later)[It::NI]) -> bool {
            if (at.left <= 0) return false;
            load(later);
            const TilePos p = at.pos(TH, TW);
            uint8_t *base = smem + slot * slotsz;
            const int gi = at.s;
            if (gi == 0) {
                const int oy = p.oy0 + (TW == 64 ? 0 : gc >> 2), ox = p.ox0 + 8 * (TW == 64 ? gc : gc & 3);
#pragma unroll
                for (int it = 0; it < 2; ++it) {
                    const int co = gco + 32 * it;
                    const bool ok = co < a.Cout && oy < a.Ho;
                    const float *row = a.g + (((int64_t)p.img * a.Cout + (ok ? co : 0)) * a.Ho + (ok ? oy : 0)) * a.Wo;
                    if (a.vecg) {
#pragma unroll
                        for (int e = 0; e < 2; ++e) ld4(&gv[it][4 * e], row + ox + 4 * e, ok && ox + 4 * e < a.Wo);
                    } else {
#pragma unroll
                        for (int e = 0; e < 8; ++e) ld1(gv[it][e], row + ox + e, ok && ox + e < a.Wo);
                    }
                }
                bar_wait(&sh.empty[slot], par, abort);
            }
            items.template store<true>(now, base + gi * kStageK * 128, p, min(kStageCh, a.Cin - gi * kStageCh), a.Ho, a.Wo);
            if (gi == ngrp - 1) {
#pragma unroll
                for (int it = 0; it < 2; ++it) {
                    const int co = gco + 32 * it;
                    const float *v = gv[it];
                    if (co < NT)
                        *reinterpret_cast<uint4 *>(base + asz + row_chunk(co, gc)) =
                            make_uint4(pk(v[0], v[1]), pk(v[2], v[3]), pk(v[4], v[5]), pk(v[6], v[7]));
                    bsum[it] += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
                }
                fence_async_smem();
                __syncwarp();
                if (lane == 0) bar_arrive(&sh.full[slot]);
                slot ^= 1;
                if (slot == 0) par ^= 1;
            }
            at.next(ngrp);
            return true;
        };
        wait_for_previous();
#pragma unroll
        for (int d = 0; d < D; ++d) load(q[d]);
        if constexpr (D == 1) {
            while (stage(q[0], q[1]) && stage(q[1], q[0])) {}
        } else {
            while (stage(q[0], q[2]) && stage(q[1], q[0]) && stage(q[2], q[1])) {}
        }
        if (a.part) {
            unsigned cta;        // read here: held since the kernel's start it costs a register in the loop
            asm volatile("mov.u32 %0, %%ctaid.x;" : "=r"(cta));
#pragma unroll
            for (int it = 0; it < 2; ++it) {
                for (int o = 1; o < 8; o <<= 1) bsum[it] += __shfl_xor_sync(0xffffffffu, bsum[it], o);
                if (gc == 0) a.part[cta * kMaxCh + gco + 32 * it] = bsum[it];
            }
        }
    } else if (warp == 4) {
        if (lane == 0) {
            const uint32_t id = idesc_bf16(NT, 0);
            bool ok = true;
            int n = 0;
            for (int t = t0; t < a.ntiles; t += dt, ++n) {
                const int slot = n & 1;
                ok = bar_wait(&sh.full[slot], (n >> 1) & 1, abort);
                if (!ok) break;
                tc_after();
                const uint32_t ab = su32(smem + slot * slotsz);
                uint64_t ad = desc(ab, 16, 1024, 2);
                const uint64_t bd = desc(ab + asz, 16, 1024, 2);
                uint32_t dcol = tmem;
#pragma unroll 1
                for (int mb = 0; mb < a.nmb; ++mb, ad += 1024, dcol += NT) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) mma_bf16(dcol, ad + q * 2, bd + q * 2, id, n > 0 || q > 0);
                }
                commit_to(&sh.empty[slot]);
                if (t + dt >= a.ntiles) commit_to(&sh.done);
            }
            if (n > 0) {
                volatile int none = 0;
                bar_wait(&sh.empty[(n - 1) & 1], ((n - 1) >> 1) & 1, &none);
            }
        }
        __syncwarp();
    } else if (__all_sync(0xffffffffu, bar_wait(&sh.done, 0, abort))) {
        wait_for_previous();
        tc_after();
        for (int mb = 0; mb < a.nmb; ++mb) {
            const int krow = mb * 128 + warp * 32 + lane;
            for (int c0 = 0; c0 < a.Cout; c0 += 16) {
                uint32_t d[16];
                tmem_ld16(tmem + mb * NT + c0 + ((uint32_t)(warp * 32) << 16), d);
                if (krow < K) {
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        if (c0 + j < a.Cout) atomicAdd(a.gw + (int64_t)(c0 + j) * K + krow, __uint_as_float(d[j]));
                }
            }
        }
        tc_before();
    }
    __syncthreads();
    if (tid == 0 && sh.abort) atomicExch(a.err, 1u);
    if (warp == 4) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols));
}

// One block per layer: gb[co] += sum over its CTAs of part[CTA][co].  It is a few loads'
// latency behind the last layer, so a thread takes every sixteenth CTA: up to twelve
// loads at once, added in order, then the sixteen sums in order.
constexpr int kSumWays = 16, kSumLoads = 12;

__global__ void __launch_bounds__(kSumWays * kMaxCh) k_bias_sum(const __grid_constant__ BiasSums b)
{
    __shared__ float sum[kSumWays][kMaxCh];
    const BiasSums::Layer L = b.layer[blockIdx.x];
    const int co = threadIdx.x % kMaxCh, q = threadIdx.x / kMaxCh;
    float t = 0.f;
    wait_for_previous();
    for (int c0 = q; c0 < L.ctas; c0 += kSumWays * kSumLoads) {
        float v[kSumLoads];
#pragma unroll
        for (int i = 0; i < kSumLoads; ++i)
            ld1(v[i], L.part + (c0 + i * kSumWays) * kMaxCh + co, c0 + i * kSumWays < L.ctas);
#pragma unroll
        for (int i = 0; i < kSumLoads; ++i) t += v[i];
    }
    sum[q][co] = t;
    __syncthreads();
    if (q == 0 && co < L.Cout) {
        for (int w = 1; w < kSumWays; ++w) t += sum[w][co];
        L.gb[co] += t;
    }
}

template <typename... P, typename A>
bool launch_chained(void (*fn)(P...), unsigned grid, int smem, cudaStream_t st, bool chain, const A &a, int threads = kThreads)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = chain ? 1 : 0;
    count_launch();
    return cudaLaunchKernelEx(&cfg, fn, a) == cudaSuccess;
}

// Dynamic shared memory above the default, once per kernel and device.
template <typename F>
bool opt_in(F *fn, int bytes, std::atomic<int> (&done)[64])
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
    if (done[dev].load() >= bytes) return true;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
    done[dev].store(bytes);
    return true;
}

// Tile width: the one that covers the output with fewer pixels, 64 on a tie
// (whole 128-byte rows in the epilogue's stores).
bool narrow(int Ho, int Wo, int pixels)
{
    auto cover = [&](int tw) {
        const int th = pixels / tw;
        return (int64_t)((Wo + tw - 1) / tw) * tw * ((Ho + th - 1) / th) * th;
    };
    return cover(32) < cover(64);
}

bool aligned4(const float *p, int w) { return w % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

constexpr int kConvSmem = 1024 + kSlots * 2 * kBlk + kMaxCh * 9 * kMaxCh * 2;
constexpr int kWgradSmem = 1024 + 2 * (5 * 128 * 128 + kMaxCh * 128);

template <int M, int TW, bool VEC>
bool launch_conv(ConvArgs &a, int N, cudaStream_t st)
{
    constexpr int TH = 128 / TW;
    static std::atomic<int> done[64];
    a.ntx = (a.Wo + TW - 1) / TW;
    a.nty = (a.Ho + TH - 1) / TH;
    const int64_t nt = (int64_t)N * a.ntx * a.nty;
    if (nt > INT32_MAX) return false;
    a.ntiles = (int)nt;
    const int smem = 1024 + kSlots * 2 * kBlk + a.NT * a.KT * 2;
    if (!opt_in(k_conv_tile<M, TW, VEC>, kConvSmem, done)) return false;
    return launch_chained(k_conv_tile<M, TW, VEC>, (unsigned)(nt < sm_count() ? nt : sm_count()), smem, st, a.chain, a);
}

template <int M>
bool launch_conv_w(ConvArgs &a, int N, cudaStream_t st)
{
    const bool nar = narrow(a.Ho, a.Wo, 128);
    if (aligned4(a.in, a.Ws)) return nar ? launch_conv<M, 32, true>(a, N, st) : launch_conv<M, 64, true>(a, N, st);
    return nar ? launch_conv<M, 32, false>(a, N, st) : launch_conv<M, 64, false>(a, N, st);
}

template <int M, int TW, bool VEC>
bool launch_wgrad_t(WgradArgs &a, int N, cudaStream_t st)
{
    constexpr int TH = 64 / TW;
    static std::atomic<int> done[64];
    a.ntx = (a.Wo + TW - 1) / TW;
    a.nty = (a.Ho + TH - 1) / TH;
    const int64_t nt = (int64_t)N * a.ntx * a.nty;
    if (nt > INT32_MAX) return false;
    a.ntiles = (int)nt;
    const int smem = 1024 + 2 * (a.nmb * 128 * 128 + a.NT * 128);
    if (!opt_in(k_wgrad_tile<M, TW, VEC>, kWgradSmem, done)) return false;
    return launch_chained(k_wgrad_tile<M, TW, VEC>, (unsigned)(nt < sm_count() ? nt : sm_count()), smem, st, a.chain, a);
}

template <int M>
bool launch_wgrad_w(WgradArgs &a, int N, cudaStream_t st)
{
    const bool nar = narrow(a.Ho, a.Wo, 64);
    if (aligned4(a.x, a.Ws)) return nar ? launch_wgrad_t<M, 32, true>(a, N, st) : launch_wgrad_t<M, 64, true>(a, N, st);
    return nar ? launch_wgrad_t<M, 32, false>(a, N, st) : launch_wgrad_t<M, 64, false>(a, N, st);
}

int n_tile(int channels) { return channels <= 16 ? 16 : channels <= 32 ? 32 : 64; }

}  // namespace

size_t bias_part_floats() { return (size_t)sm_count() * kMaxCh; }

bool launch_bias_sums(const BiasSums &b, cudaStream_t st)
{
    return launch_chained(k_bias_sum, b.n, 0, st, true, b, kSumWays * kMaxCh);
}

bool conv_tile_fits(int Cin, int Cout) { return Cin >= 1 && Cin <= kMaxCh && Cout >= 1 && Cout <= kMaxCh; }

bool conv_tile(bool grad, int S, int UPS, const float *in, int N, int Cin, int Hs, int Ws, const __nv_bfloat16 *w,
               const float *bias, int Cout, int Ho, int Wo, int relu, const ConvOut &o, unsigned *err, cudaStream_t st,
               bool chain)
{
    ConvArgs a{};
    a.chain = chain;
    a.in = in;
    a.Cin = Cin;
    a.Hs = Hs;
    a.Ws = Ws;
    a.w = w;
    a.bias = bias;
    a.Cout = Cout;
    a.Ho = Ho;
    a.Wo = Wo;
    a.relu = relu;
    a.o = o;
    a.NT = n_tile(Cout);
    const int full = (Cin - 1) / kStageCh;
    a.KT = full * kStageK + ((Cin - full * kStageCh) * 9 + 15) / 16 * 16;
    a.err = err;
    if (grad) return S == 2 ? launch_conv_w<kD2>(a, N, st) : launch_conv_w<kD1>(a, N, st);
    if (UPS) return launch_conv_w<kFU>(a, N, st);
    return S == 2 ? launch_conv_w<kF2>(a, N, st) : launch_conv_w<kF1>(a, N, st);
}

bool wgrad_tile(int S, int UPS, const float *x, int N, int Cin, int Hs, int Ws, const float *g, int Cout, int Ho,
                int Wo, float *gw, float *gb, float *part, BiasSums *sums, unsigned *err, cudaStream_t st, bool chain)
{
    WgradArgs a{};
    a.part = part;
    a.chain = chain;
    a.x = x;
    a.Cin = Cin;
    a.Hs = Hs;
    a.Ws = Ws;
    a.g = g;
    a.Cout = Cout;
    a.Ho = Ho;
    a.Wo = Wo;
    a.vecg = aligned4(g, Wo);
    a.gw = gw;
    a.NT = n_tile(Cout);
    a.nmb = (Cin * 9 + 127) / 128;
    a.err = err;
    const bool ok = UPS ? launch_wgrad_w<kFU>(a, N, st) : S == 2 ? launch_wgrad_w<kF2>(a, N, st) : launch_wgrad_w<kF1>(a, N, st);
    if (ok && part) sums->layer[sums->n++] = {part, gb, std::min(a.ntiles, sm_count()), Cout};
    return ok;
}

}  // namespace mxp
