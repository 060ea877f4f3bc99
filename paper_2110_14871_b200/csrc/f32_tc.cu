// The fp32 forward with its pointwise products on the tensor cores (3 x 3 and 5 x 5 filters, NCHW and NHWC).
//
// z is computed on the ALUs in fp32, tap by tap as in fused_f32_kernel.  The pointwise stage is a contraction, and bf16 products
// with fp32 sums can carry it at full fp32 precision: an fp32 value is the exact sum of three bf16 values (its 24 significant
// bits in pieces of 8), z = z1 + z2 + z3 and P = p1 + p2 + p3 with every piece at most 2^-8 of the one before, and
//     z P = z1 p1 + (z1 p2 + z2 p1) + (z1 p3 + z2 p2 + z3 p1) + what is below 2^-24 of the product
// (2^-27.5 in the root mean square).
// The tensor cores add to their accumulators without rounding to nearest, which would cost a long sum more than fp32 arithmetic
// does.  An accumulator therefore holds one chunk of kF32TcChunk intermediate channels only, smallest products first, and the chunks'
// sums are added in fp32 registers: fewer roundings than one multiply-add per channel.
//
// bf16 ends where fp32 does, so the lower pieces of small values would leave its range: taps and weights are taken times 2^24 (exact)
// and y times 2^-48.  Multiples of 2^-149, fp32's smallest step, are then multiples of 2^-125 and so are their pieces.  (Without, at
// weights of 2^-110 the error was 5e-7 and at 2^-123 4e-3.)  At the other end outputs beyond 2^79 and z and weights beyond 2^103
// overflow and are worked out again like those that are not finite.
//
// Error against 64 bits (2-norm), this kernel over the ALU kernel, G intermediate channels, 3 x 3 | 5 x 5 taps: 1.20 | 1.07 at G = 1, 1.04 |
// 1.01 at 4, 0.98 | 0.96 at 8, 0.80 | 0.88 at 16, 0.71 | 0.78 at 32, 0.42 | 0.52 at 128, 0.22 | 0.18 at 648 | 1693 (positive values: 1.05 |
// 1.09 at 8, 0.79 | 0.81 at 16).  With few terms the tensor cores' truncation outweighs the roundings saved: from kF32TcLeast on only.
//
// What bounds it: the serial instruction streams of the warps that load and cut (3900 cycles a chunk if nothing else runs) and that
// compute z (3500), which share four schedulers at two instructions per cycle; the products (12 of 128 x N x 16, 768 cycles a chunk at
// N = 128) keep the tensor pipe busy for 14 %.  16 x 128 -> 128 channels at 28 x 28, G = 619: 83.5 us in fused_f32_kernel, 53.6 here
// (timed with a role's work left out: without z 43, without input staging 45, without products 49).  The roles' loops are kept
// short: the first version, all unrolled, was 186 KB of code and took 127 us.  1 x 249 -> 25 channels at 18 x 17: 46.6 | 11.4 us (eight
// blocks share a tile), 39 x 10 -> 17 at 116 x 145, NHWC: 362 | 124.
// Roles (one block of 24 warps per SM, register shares by setmaxnreg): warps 0-3 add up the chunks (thread = one pixel x up to
// 128 output channels) and store y, 4-11 compute z (a warp: 64 pixels x 8 channels of a chunk), 12-19 cut the weights into pieces
// and stage input rows, filters and the table of channels a chunk ahead, 20 issues the products.
// Layers with few tiles: the blocks of a cluster share a tile's chunks and add their sums through distributed shared memory.
#include <float.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "sm100.cuh"

namespace gdws {

constexpr int kF32TcChunk = 32;          // intermediate channels per chunk: 64-byte rows of bf16
constexpr int kF32TcLeast = 16;          // intermediate channels from which on it is as exact as the ALUs (above)
constexpr int kF32TcThreads = 24 * 32;
constexpr int kF32TcZWarp = 4, kF32TcLoadWarp = 12, kF32TcMmaWarp = 20;
// Registers per thread after the split: setmaxnreg.inc can only claim what other warpgroups of the same block released, so the sum
// must stay within the block's allocation at launch (768 threads x 80; f32tc_launch checks the kernel for it).
constexpr int kF32TcRegsLaunch = 80, kF32TcRegsSum = 168, kF32TcRegsZ = 80, kF32TcRegsLoad = 56, kF32TcRegsMma = 40;
static_assert(kF32TcRegsSum + 2 * kF32TcRegsZ + 2 * kF32TcRegsLoad + kF32TcRegsMma <= 6 * kF32TcRegsLaunch,
              "register split exceeds the block's allocation: setmaxnreg.inc would wait forever");
template <int N> __device__ __forceinline__ void f32tc_regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void f32tc_regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
constexpr int kF32TcMaxPos = 1024;       // staged positions of a tile
constexpr uint32_t kF32TcSw64 = 4u << 29;     // descriptor high word: layout type "64-byte swizzle"
constexpr int kF32TcMaxStages = 3;
constexpr float kF32TcScale = 16777216.f, kF32TcUnscale = 1.f / (kF32TcScale * kF32TcScale);      // 2^24: see above
constexpr uint32_t kF32TcA = 128 * 64;        // bytes of one piece of z

struct F32TcParams {
    const float *x, *dw, *pw, *bias;
    const int32_t *chan;
    float *y;
    int *status;
    int H, W, D, G, stride, pad, Ho, Wo, relu;
    long long xn, xc, xh, xw, yn, yc, yh, yw;      // element strides
    int N, TN, PH, PW, IH, IW, np, pitch, tiles_h, tiles_w, ntiles;
    int nq, Nd, ns;                                // chunks; columns of the products (output channels of a block, a multiple of 16); stages
    uint32_t b_piece, ab_bytes, off_x, x_bytes, off_f, off_slot, off_tab, off_bias;
};

// Bounded like the other waits; inline, because ptxas finds no registers for calls in roles with register shares of their own.
__device__ __forceinline__ void f32tc_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (mbar_try_wait(bar, parity)) return;
#pragma unroll 1
    for (uint32_t it = 0; it < (1u << 20) && !*abort_flag; ++it)
        if (mbar_try_wait_suspend(bar, parity, 4096u)) return;
    if (*abort_flag) return;
    *abort_flag = 1;
    atomicOr(status, code);
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&r)[16])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
        ::"r"(taddr), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]), "f"(r[4]), "f"(r[5]), "f"(r[6]), "f"(r[7]),
          "f"(r[8]), "f"(r[9]), "f"(r[10]), "f"(r[11]), "f"(r[12]), "f"(r[13]), "f"(r[14]), "f"(r[15]) : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Three bf16 pieces of each of two fp32 values, packed: the first value in the low halves.
__device__ __forceinline__ void split3(float a, float b, uint32_t &p1, uint32_t &p2, uint32_t &p3)
{
    auto rest = [&](uint32_t p) {                // both values less their pieces, one issue slot for the two
        asm("{\n\t.reg .b64 v, h;\n\tmov.b64 v, {%0, %1};\n\tmov.b64 h, {%2, %3};\n\tsub.rn.f32x2 v, v, h;\n\tmov.b64 {%0, %1}, v;\n\t}"
            : "+f"(a), "+f"(b) : "r"(p << 16), "r"(p & 0xFFFF0000u));
    };
    p1 = pack_bf16x2(a, b);
    rest(p1);
    p2 = pack_bf16x2(a, b);
    rest(p2);
    p3 = pack_bf16x2(a, b);
}

// Outputs that are not finite, once more in fp32 on the ALUs (pieces of an infinity are an infinity and NaN).  The warps that add
// up the chunks leave NaN in their places in y; when a block's tiles are done, they look for them and work such a tile's columns c0
// to c1 out from the inputs, 64 pixels and 32 intermediate channels at a time through shared memory, added in fused_f32_kernel's order.
// Nobody waits for the block in a bounded wait meanwhile.  (Each such output summed up by its own thread took 89 ms where one tap of
// 16 x 128 -> 128 channels at 28 x 28 is infinite, and its code beside the hot loops 2 us of every call; here 0.53 ms, an ordinary call 54 us.)
constexpr int kF32TcRedoZ = 65, kF32TcRedoW = 129;       // pitches of z and of the weights: odd, for stores down a column
template <int K, int NB, bool NHWC>
__device__ __forceinline__ void f32tc_redo(const F32TcParams &P, uint8_t *base, const float *bias, volatile int *any, int tile0, int step, int c0, int c1)
{
    constexpr int K2 = K * K, CH = kF32TcChunk, T = 128, COLS = 4 * NB;
    float *const zs = reinterpret_cast<float *>(base), *const ws = zs + CH * kF32TcRedoZ, *const taps = ws + CH * kF32TcRedoW;
    int *const pn = reinterpret_cast<int *>(taps + CH * K2), *const ph0 = pn + 128, *const pw0 = ph0 + 128, *const py = pw0 + 128;      // py: pixel of the image
    static_assert(4 * (CH * (kF32TcRedoZ + kF32TcRedoW + K2) + 4 * 128) <= 2 * (3 * kF32TcA + 3 * 16 * 64), "two stages of operands hold it");
    const int tid = threadIdx.x, d0 = (int)blockIdx.y * 128 + c0, nd = c1 - c0, pg = tid & 15, dg = tid >> 4;
#pragma unroll 1
    for (int tile = tile0; tile < P.ntiles; tile += step) {
        const int hw = P.tiles_h * P.tiles_w, ppi = P.PH * P.PW, nl = tid / ppi, ph = (tid - nl * ppi) / P.PW, pw = tid - nl * ppi - ph * P.PW;
        const int bn = tile / hw, bh = (tile - bn * hw) / P.tiles_w, bw = tile - bn * hw - bh * P.tiles_w;
        const int n = bn * P.TN + nl, ho = bh * P.PH + ph, wo = bw * P.PW + pw;
        const bool live = nl < P.TN && n < P.N && ho < P.Ho && wo < P.Wo;
        pn[tid] = live ? n : -1; ph0[tid] = ho * P.stride - P.pad; pw0[tid] = wo * P.stride - P.pad; py[tid] = ho * P.Wo + wo;
        if (tid == 0) *any = 0;
        named_bar_sync(2, T);
        const float *const yl = P.y + n * P.yn + ho * P.yh + wo * P.yw;
        bool found = false;
#pragma unroll 4
        for (int d = 0; d < nd; ++d)
            if (live) { const float v = yl[(d0 + d) * P.yc]; found = found || v != v; }
        if (found) *any = 1;
        named_bar_sync(2, T);
        const bool go = *any != 0;
        named_bar_sync(2, T);
#pragma unroll 1
        for (int half = 0; go && half < 128; half += 64) {
            float acc[4][COLS] = {};             // pixels half + pg + 16 j, columns dg + 8 e
#pragma unroll 1
            for (int i0 = 0; i0 < P.G; i0 += CH) {
                const int ni = min(CH, P.G - i0);
#pragma unroll 4
                for (int t = tid; t < ni * K2; t += T) taps[t % K2 * CH + t / K2] = __ldg(P.dw + (size_t)i0 * K2 + t);
                if ((tid & (CH - 1)) < ni) {
                    const float *const w = P.pw + (size_t)d0 * P.G + i0 + (tid & (CH - 1));
#pragma unroll 8
                    for (int d = tid / CH; d < nd; d += T / CH) ws[(tid & (CH - 1)) * kF32TcRedoW + d] = __ldg(w + (size_t)d * P.G);
                }
                named_bar_sync(2, T);
#pragma unroll 2
                for (int e = tid; e < CH * 64; e += T) {
                    const int rh = NHWC ? e / CH : e & 63, r = half + rh, i = NHWC ? e & (CH - 1) : e >> 6;
                    if (i < ni && pn[r] >= 0) {
                        const float *const x = P.x + pn[r] * P.xn + __ldg(P.chan + i0 + i) * P.xc;
                        const int h0 = ph0[r], w0 = pw0[r];
                        float z = 0.f;
#pragma unroll
                        for (int t = 0; t < K2; ++t) {
                            const int h = h0 + t / K, w = w0 + t % K;
                            z = fmaf(taps[t * CH + i], h >= 0 && h < P.H && w >= 0 && w < P.W ? __ldg(x + h * P.xh + w * P.xw) : 0.f, z);
                        }
                        zs[i * kF32TcRedoZ + rh] = z;
                    }
                }
                named_bar_sync(2, T);
#pragma unroll 1
                for (int i = 0; i < ni; ++i) {   // rows and columns outside: whatever is there, not stored below
                    float z[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) z[j] = zs[i * kF32TcRedoZ + pg + 16 * j];
#pragma unroll
                    for (int e = 0; e < COLS; ++e) {
                        const float w = ws[i * kF32TcRedoW + dg + 8 * e];
#pragma unroll
                        for (int j = 0; j < 4; ++j) acc[j][e] = fmaf(z[j], w, acc[j][e]);
                    }
                }
                named_bar_sync(2, T);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int r = half + pg + 16 * j, px = py[r];
                if (pn[r] < 0) continue;
                float *const yr = P.y + pn[r] * P.yn + px * P.yw + d0 * P.yc;        // pixels of an image are yw apart in either layout
#pragma unroll
                for (int e = 0; e < COLS; ++e) {
                    const int d = dg + 8 * e;
                    float *const y = yr + d * P.yc;
                    if (d >= nd || *y == *y) continue;
                    const float v = acc[j][e] + bias[c0 + d];
                    *y = P.relu ? fmaxf(v, 0.f) : v;
                }
            }
        }
        named_bar_sync(2, T);                    // the table is written anew
    }
}

// Floats per filter in shared memory: 3 x 3 taps twice each (the packed multiply-adds of two pixels take them as pairs).
__host__ __device__ constexpr int f32tc_filt_pitch(int k) { return k == 3 ? 20 : (k * k + 3) / 4 * 4; }

__device__ __forceinline__ float f32tc_lds(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint64_t f32tc_pair(float lo, float hi)
{
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
    return v;
}
__device__ __forceinline__ void f32tc_unpair(uint64_t v, float &lo, float &hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }

__device__ __forceinline__ void f32tc_scale(float &a, float &b)
{
    uint64_t v = f32tc_pair(a, b);
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(v) : "l"(f32tc_pair(kF32TcScale, kF32TcScale)));
    f32tc_unpair(v, a, b);
}

// z of 4 channels at 64 pixels (two groups of 32), 3 x 3 taps, cut into pieces: o[piece][pixel group][pair of channels].  The two
// pixels of a thread share the packed multiply-adds.  xs: address of the staged rows, pos: of the pixels' windows in them.
__device__ __forceinline__ void f32tc_z3(uint32_t xs, uint32_t iw4, uint32_t fs, const int4 &off4, const uint32_t (&pos)[2], uint32_t (&o)[3][2][2], uint64_t (&xr)[9], int &have)
{
    const int off[4] = {off4.x, off4.y, off4.z, off4.w};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float z[2][2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int of = off[2 * j + e];
            if (of != have && of >= 0) {         // the next input channel's windows: the same for the whole warp
                have = of;
                uint32_t a = xs + (uint32_t)of + pos[0], b = xs + (uint32_t)of + pos[1];
#pragma unroll
                for (int u = 0; u < 3; ++u, a += iw4, b += iw4)
#pragma unroll
                    for (int v = 0; v < 3; ++v) xr[3 * u + v] = f32tc_pair(f32tc_lds(a + 4u * v), f32tc_lds(b + 4u * v));
            }
            uint64_t acc = 0, w[10];
#pragma unroll
            for (int t = 0; t < 5; ++t) asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(w[2 * t]), "=l"(w[2 * t + 1]) : "r"(fs + (uint32_t)((2 * j + e) * 80 + 16 * t)));
#pragma unroll
            for (int t = 0; t < 9; ++t) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(xr[t]), "l"(w[t]));
            if (of < 0) acc = 0;                 // beyond G: zero, not 0 * x
            f32tc_unpair(acc, z[e][0], z[e][1]);
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) split3(z[0][g], z[1][g], o[0][g][j], o[1][g][j], o[2][g][j]);
    }
}
// The same for 5 x 5 taps and 32 pixels: 25 window values are enough registers.
__device__ __forceinline__ void f32tc_z5(uint32_t xs, uint32_t iw4, uint32_t fs, const int4 &off4, uint32_t pos, uint32_t (&o)[3][2], float (&xr)[25], int &have)
{
    const int off[4] = {off4.x, off4.y, off4.z, off4.w};
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float z[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int of = off[2 * j + e];
            if (of != have && of >= 0) {
                have = of;
                uint32_t a = xs + (uint32_t)of + pos;
#pragma unroll
                for (int u = 0; u < 5; ++u, a += iw4)
#pragma unroll
                    for (int v = 0; v < 5; ++v) xr[5 * u + v] = f32tc_lds(a + 4u * v);
            }
            float acc = 0.f;
#pragma unroll
            for (int t = 0; t < 7; ++t) {
                float w[4];
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(w[0]), "=f"(w[1]), "=f"(w[2]), "=f"(w[3]) : "r"(fs + (uint32_t)((2 * j + e) * 112 + 16 * t)));
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (4 * t + i < 25) acc = fmaf(w[i], xr[4 * t + i], acc);
            }
            z[e] = of >= 0 ? acc : 0.f;
        }
        split3(z[0], z[1], o[0][j], o[1][j], o[2][j]);
    }
}

// NB: 32-column blocks of the sums.
template <int K, int NB, bool NHWC>
__global__ void __launch_bounds__(kF32TcThreads, 1) f32_tc_kernel(const __grid_constant__ F32TcParams P, int split)
{
    extern __shared__ uint8_t smem_raw[];
    // xfull[2] xfree[2] | full[3] free[3] | accfull[2] accfree[2] | drain
    __shared__ __align__(8) uint64_t bars[16];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, redo, redo_any;           // redo: an output of this block is not finite
    constexpr int FP = f32tc_filt_pitch(K), K2 = K * K;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    uint8_t *const base = smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
    const uint32_t ab_s = smem_u32(base), x_s = ab_s + P.off_x, f_s = ab_s + P.off_f, slot_s = ab_s + P.off_slot;
    int *const tab = reinterpret_cast<int *>(base + P.off_tab);
    float *const bias_sm = reinterpret_cast<float *>(base + P.off_bias);
    const uint32_t bar_xfull = smem_u32(&bars[0]), bar_xfree = bar_xfull + 16, bar_full = bar_xfull + 32, bar_free = bar_full + 8 * kF32TcMaxStages;
    const uint32_t bar_accfull = bar_free + 8 * kF32TcMaxStages, bar_accfree = bar_accfull + 16, bar_drain = bar_accfree + 16;
    if (tid == 0) {
        abort_flag = redo = 0;
#pragma unroll 1
        for (int i = 0; i < 2; ++i) { mbar_init(bar_xfull + 8 * i, 8); mbar_init(bar_xfree + 8 * i, 8); mbar_init(bar_accfull + 8 * i, 1); mbar_init(bar_accfree + 8 * i, 4); }
#pragma unroll 1
        for (int i = 0; i < kF32TcMaxStages; ++i) { mbar_init(bar_full + 8 * i, 16); mbar_init(bar_free + 8 * i, 1); }
        mbar_init(bar_drain, 1);
        fence_mbar_init();
    }
    grid_launch_dependents();
    if (warp == kF32TcMmaWarp) tmem_alloc(smem_u32(&tmem_slot), 64u * NB);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_wait();
    const uint32_t tmem = tmem_slot;
    const int rank = split > 1 ? (int)cluster_rank() : 0, cluster = (int)blockIdx.x / split, nclusters = (int)gridDim.x / split;
    const int q0 = rank * P.nq / split, q1 = (rank + 1) * P.nq / split;
    const int d0 = (int)blockIdx.y * 128, dn = min(P.D - d0, P.Nd);      // this block's output channels
    const int hw = P.tiles_h * P.tiles_w;

    if (warp < kF32TcZWarp) {
        // ---------------- sums of the chunks, y ----------------
        f32tc_regs_inc<kF32TcRegsSum>();
        const int r = tid, ppi = P.PH * P.PW;
        const int nl = r / ppi, ph = (r - nl * ppi) / P.PW, pw = r - nl * ppi - ph * P.PW;
        for (int d = tid; d < 32 * NB; d += 128) bias_sm[d] = P.bias && d < dn ? __ldg(P.bias + d0 + d) : 0.f;
        named_bar_sync(2, 128);
        int cnt = 0;
#pragma unroll 1
        for (int tile = cluster; tile < P.ntiles; tile += nclusters) {
            uint64_t sum[2 * NB][8];             // pairs of columns
#pragma unroll
            for (int b = 0; b < 2 * NB; ++b)
#pragma unroll
                for (int e = 0; e < 8; ++e) sum[b][e] = 0;
            const uint32_t t0 = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
            for (int q = q0; q < q1; ++q, ++cnt) {
                const int buf = cnt & 1;
                if (lane == 0) f32tc_wait(bar_accfull + 8 * buf, (uint32_t)(cnt >> 1) & 1u, &abort_flag, P.status, kStatusWaitMma);
                __syncwarp();
                tc_fence_after();
                const uint32_t t = t0 + (uint32_t)(buf * 32 * NB);
#pragma unroll
                for (int b = 0; b < 2 * NB; ++b) {
                    uint32_t v[16];
                    tmem_ld16(t + 16 * b, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 8; ++e) asm("add.rn.f32x2 %0, %0, %1;" : "+l"(sum[b][e]) : "l"(f32tc_pair(__uint_as_float(v[2 * e]), __uint_as_float(v[2 * e + 1]))));
                }
                if (q == q1 - 1) {               // the tile's sums take the last chunk's place, from where a short loop finishes them
#pragma unroll
                    for (int b = 0; b < 2 * NB; ++b) {
                        float v[16];
#pragma unroll
                        for (int e = 0; e < 8; ++e) f32tc_unpair(sum[b][e], v[2 * e], v[2 * e + 1]);
                        tmem_st16(t + 16 * b, v);
                    }
                    tmem_st_wait();
                    if (split > 1) break;        // a cluster has one tile: the sums meet below
                    const int bn = tile / hw, bh = (tile - bn * hw) / P.tiles_w, bw = tile - bn * hw - bh * P.tiles_w;
                    const int n = bn * P.TN + nl, ho = bh * P.PH + ph, wo = bw * P.PW + pw;
                    const bool live = nl < P.TN && n < P.N && ho < P.Ho && wo < P.Wo;
                    float *yp = P.y + n * P.yn + ho * P.yh + wo * P.yw + d0 * P.yc;
                    // NHWC: 32 pixels x 16 channels turn in shared memory, so that a store covers two pixels' 16 channels
                    float *const turn = bias_sm + 32 * NB + warp * 32 * 17;
                    const int mask = live ? 1 : 0;
#pragma unroll 1
                    for (int c = 0; c < dn; c += 16) {
                        uint32_t a[16];
                        tmem_ld16(t + c, a);
                        tmem_ld_wait();
                        uint32_t odd = 0;        // columns that are not finite
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            float v = __uint_as_float(a[e]);
                            if (!(fabsf(v) <= FLT_MAX)) odd |= 1u << e;
                            v = fmaf(v, kF32TcUnscale, bias_sm[c + e]);
                            if (P.relu) v = fmaxf(v, 0.f);
                            a[e] = __float_as_uint(v);
                        }
                        if constexpr (NHWC) {
#pragma unroll
                            for (int e = 0; e < 16; ++e) turn[lane * 17 + e] = __uint_as_float(a[e]);
                            __syncwarp();
                            const bool in = c + (lane & 15) < dn;
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                const int px = 2 * e + (lane >> 4);
                                float *dst = reinterpret_cast<float *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(yp), px));
                                const int ok = __shfl_sync(0xffffffffu, mask, px);
                                if (ok && in) dst[c + (lane & 15)] = turn[px * 17 + (lane & 15)];
                            }
                            __syncwarp();
                        } else if (live) {
                            float *yc = yp + c * P.yc;
#pragma unroll
                            for (int e = 0; e < 16; ++e, yc += P.yc)
                                if (c + e < dn) *yc = __uint_as_float(a[e]);
                        }
#pragma unroll 1
                        for (odd = live ? odd : 0u; odd; odd &= odd - 1) {
                            const int d = c + __ffs(odd) - 1;
                            if (d >= dn) break;
                            yp[d * P.yc] = __uint_as_float(0x7fffffffu);
                            redo = 1;
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_accfree + 8 * buf);
            }
            if (split > 1) break;
        }
        int c0 = 0, c1 = dn;                     // columns that this block stores
        if (split > 1) {                         // all products are done: the operands' memory takes the sums, [column][pixel]
            float *part = reinterpret_cast<float *>(base);
            const uint32_t t = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(((q1 - q0 - 1) & 1) * 32 * NB);
#pragma unroll 1
            for (int c = 0; c < 32 * NB; c += 16) {
                uint32_t a[16];
                tmem_ld16(t + c, a);
                tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 16; ++e) part[(c + e) * 128 + r] = __uint_as_float(a[e]);
            }
            cluster_sync();                      // rank r of the cluster finishes its share of the output channels, at least 4
            const int bn = cluster / hw, bh = (cluster - bn * hw) / P.tiles_w, bw = cluster - bn * hw - bh * P.tiles_w;
            const int n = bn * P.TN + nl, ho = bh * P.PH + ph, wo = bw * P.PW + pw;
            const bool live = nl < P.TN && n < P.N && ho < P.Ho && wo < P.Wo;
            float *yp = P.y + n * P.yn + ho * P.yh + wo * P.yw + d0 * P.yc;
            c0 = rank * (32 * NB / split); c1 = min(c0 + 32 * NB / split, dn);
#pragma unroll 1
            for (int c = c0; live && c < c1; c += 4) {
                float v[4] = {};
#pragma unroll 1
                for (int o0 = 0; o0 < split; o0 += 4) {      // in the chunks' order, sixteen reads in flight
                    float w[4][4];
#pragma unroll
                    for (int o = 0; o < 4; ++o) {
                        if (o0 + o >= split) break;
                        const uint32_t src = map_shared(ab_s + (uint32_t)(c * 128 + r) * 4u, (uint32_t)(o0 + o));
#pragma unroll
                        for (int e = 0; e < 4; ++e) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(w[o][e]) : "r"(src + 512u * e));
                    }
#pragma unroll
                    for (int o = 0; o < 4; ++o)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (o0 + o < split) v[e] += w[o][e];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (c + e >= c1) break;
                    const bool fine = fabsf(v[e]) <= FLT_MAX;
                    if (!fine) redo = 1;
                    v[e] = fmaf(v[e], kF32TcUnscale, bias_sm[c + e]);
                    if (P.relu) v[e] = fmaxf(v[e], 0.f);
                    yp[(c + e) * P.yc] = fine ? v[e] : __uint_as_float(0x7fffffffu);
                }
            }
            __syncwarp();
            cluster_sync();                      // every block's sums have been read
        }
        named_bar_sync(2, 128);
        if (*(volatile int *)&redo) f32tc_redo<K, NB, NHWC>(P, base, bias_sm, &redo_any, cluster, nclusters, c0, c1);
    } else if (warp < kF32TcLoadWarp) {
        // ---------------- z ----------------
        f32tc_regs_dec<kF32TcRegsZ>();
        const int zw = warp - kF32TcZWarp, half = zw & 1, oct = zw >> 1, ppi = P.PH * P.PW;
        uint32_t pos[2], row[2];
#pragma unroll
        for (int g = 0; g < 2; ++g) {
            const int r = half * 64 + g * 32 + lane, nl = r / ppi, ph = (r - nl * ppi) / P.PW, pw = r - nl * ppi - ph * P.PW;
            pos[g] = nl < P.TN ? 4u * (uint32_t)((nl * P.IH + ph * P.stride) * P.IW + pw * P.stride) : 0u;
            row[g] = (uint32_t)r * 64u + (uint32_t)((oct ^ ((r >> 1) & 3)) << 4);
        }
        int cnt = 0, st = 0;
        uint32_t par = 1;
#pragma unroll 1
        for (int tile = cluster; tile < P.ntiles; tile += nclusters) {
#pragma unroll 1
            for (int q = q0; q < q1; ++q, ++cnt) {
                const int buf = cnt & 1;
                f32tc_wait(bar_xfull + 8 * buf, (uint32_t)(cnt >> 1) & 1u, &abort_flag, P.status, kStatusWaitOperand);
                f32tc_wait(bar_free + 8 * st, par, &abort_flag, P.status, kStatusWaitStage);
                const uint32_t xs = x_s + (uint32_t)buf * P.x_bytes, fs = f_s + (uint32_t)((buf * kF32TcChunk + oct * 8) * FP * 4), sl = slot_s + (uint32_t)((buf * kF32TcChunk + oct * 8) * 4);
                const uint32_t a_s = ab_s + (uint32_t)st * P.ab_bytes, iw4 = 4u * (uint32_t)P.IW;
                auto offsets = [&](int h) {
                    int4 v;
                    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(sl + 16u * (uint32_t)h));
                    return v;
                };
                if constexpr (K == 3) {
                    uint64_t xr[9];
                    int have = -1;
#pragma unroll 1
                    for (int h = 0; h < 2; ++h) {
                        uint32_t o[3][2][2];
                        f32tc_z3(xs, iw4, fs + (uint32_t)(h * 4 * FP * 4), offsets(h), pos, o, xr, have);
#pragma unroll
                        for (int e = 0; e < 3; ++e)
#pragma unroll
                            for (int g = 0; g < 2; ++g)
                                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a_s + (uint32_t)e * kF32TcA + row[g] + 8u * h), "r"(o[e][g][0]), "r"(o[e][g][1]) : "memory");
                    }
                } else {
#pragma unroll 1
                    for (int g = 0; g < 2; ++g) {
                        float xr[25];
                        const uint32_t pg = g ? pos[1] : pos[0], dst = a_s + (g ? row[1] : row[0]);
                        int have = -1;
#pragma unroll 1
                        for (int h = 0; h < 2; ++h) {
                            uint32_t o[3][2];
                            f32tc_z5(xs, iw4, fs + (uint32_t)(h * 4 * FP * 4), offsets(h), pg, o, xr, have);
#pragma unroll
                            for (int e = 0; e < 3; ++e)
                                asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst + (uint32_t)e * kF32TcA + 8u * h), "r"(o[e][0]), "r"(o[e][1]) : "memory");
                        }
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(bar_xfree + 8 * buf);
                    mbar_arrive(bar_full + 8 * st);
                }
                if (++st == P.ns) { st = 0; par ^= 1u; }
            }
        }
    } else if (warp < kF32TcMmaWarp) {
        // ---------------- weights of a chunk, input rows, filters and channel table of the next; loads a step ahead in registers ----------------
        f32tc_regs_dec<kF32TcRegsLoad>();
        const int lt = tid - kF32TcLoadWarp * 32, lw = warp - kF32TcLoadWarp;
        // weights: thread = two neighbouring channels of rows dr, dr + 16, ...
        const int ip = lt & 15, dr = lt >> 4, wrow = 16 * P.G;
        float wv[2 * NB][2];
        uint32_t rows = 0;                       // which of the thread's rows are output channels
#pragma unroll
        for (int j = 0; j < 2 * NB; ++j) rows |= (uint32_t)(dr + 16 * j < dn) << j;
        const float *const w0 = P.pw + (size_t)(d0 + (dr < dn ? dr : 0)) * P.G + 2 * ip;
        auto load_w = [&](int j, const float *w, bool in0, bool in1) {
            const bool in = (rows >> j) & 1u;
            wv[j][0] = in && in0 ? __ldg(w + j * wrow) : 0.f;
            wv[j][1] = in && in1 ? __ldg(w + j * wrow + 1) : 0.f;
        };
        // input: a round is 8 channels x 256 positions.  NCHW: thread = position, 8 channels; NHWC: thread = one of 8 neighbouring
        // channels, 8 positions 32 apart (whole sectors in, 32 different banks out)
        constexpr int NF = (kF32TcChunk * K2 + 255) / 256;
        float xv[8], fv[NF];
        int c = -1, c_next = -1, nslots = 0, xtile = cluster, xq = q0, xcnt = 0;
        const int iw_ih = P.IW * P.IH, xc = (int)P.xc;
        const float *xt = P.x;
        const uint32_t list_s = slot_s + (uint32_t)((2 + lw) * kF32TcChunk * 4);      // this warp's list of the chunk's input channels, as offsets in x
        const int a_first = NHWC ? lw * 4 + (lane >> 3) : lt;
        auto load_round = [&](int s0, int a0) {
            if constexpr (!NHWC) {
                const int a = a0 + a_first, o = a < P.np ? tab[a] : -1;
                int co[8];
                asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(co[0]), "=r"(co[1]), "=r"(co[2]), "=r"(co[3]) : "r"(list_s + 4u * (uint32_t)s0));
                asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(co[4]), "=r"(co[5]), "=r"(co[6]), "=r"(co[7]) : "r"(list_s + 4u * (uint32_t)s0 + 16u));
#pragma unroll
                for (int j = 0; j < 8; ++j) xv[j] = s0 + j < nslots && o >= 0 ? __ldg(xt + co[j] + o) : 0.f;
            } else {
                int co;
                asm volatile("ld.shared.s32 %0, [%1];" : "=r"(co) : "r"(list_s + 4u * (uint32_t)(s0 + (lane & 7))));
                const bool ok = s0 + (lane & 7) < nslots;
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int a = a0 + a_first + 32 * j, o = ok && a < P.np ? tab[a] : -1;
                    xv[j] = o >= 0 ? __ldg(xt + co + o) : 0.f;
                }
            }
        };
        auto store_round = [&](uint32_t xs, int s0, int a0) {
            const uint32_t dst = xs + 4u * (uint32_t)(NHWC ? (s0 + (lane & 7)) * P.pitch + a0 + a_first : s0 * P.pitch + a0 + a_first);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bool in = NHWC ? s0 + (lane & 7) < nslots && a0 + a_first + 32 * j < P.np : s0 + j < nslots && a0 + a_first < P.np;
                if (in) asm volatile("st.shared.f32 [%0], %1;" ::"r"(dst + (NHWC ? 128u * j : 4u * (uint32_t)(j * P.pitch))), "f"(xv[j]) : "memory");
            }
        };
        auto chan_of = [&](int q) { const int i = q * kF32TcChunk + lane; return i < P.G ? __ldg(P.chan + i) : -1; };
        c_next = chan_of(q0);
        for (int j = lt; j < P.np; j += 256) {   // positions of a tile: image, row, column (read again by the thread that writes them)
            const int nl = j / iw_ih, ih = (j - nl * iw_ih) / P.IW;
            tab[P.np + j] = nl << 20 | ih << 10 | (j - nl * iw_ih - ih * P.IW);
        }
        int q = q0, left = (P.ntiles - cluster + nclusters - 1) / nclusters * (q1 - q0), st = 0;     // weights: chunks to go
        int slot = 0;
        uint32_t par = 1;
#pragma unroll
        for (int j = 0; j < 2 * NB; ++j) load_w(j, w0 + q0 * kF32TcChunk, q0 * kF32TcChunk + 2 * ip < P.G, q0 * kF32TcChunk + 2 * ip + 1 < P.G);
        // step s: input s + 2 is asked for, input s + 1 stored, weights s stored
#pragma unroll 1
        for (int s = -2; left > 0; ++s) {
            if (s >= -1 && nslots > 0) {         // asked for in the step before
                const int buf = xcnt & 1;
                const uint32_t xs = x_s + (uint32_t)buf * P.x_bytes;
                f32tc_wait(bar_xfree + 8 * buf, ((uint32_t)(xcnt >> 1) & 1u) ^ 1u, &abort_flag, P.status, kStatusWaitStage);
#pragma unroll
                for (int j = 0; j < NF; ++j) {
                    const int t = lt + 256 * j, kk = t / K2;
                    const uint32_t f = f_s + (uint32_t)((buf * kF32TcChunk + kk) * FP * 4);
                    if (t < kF32TcChunk * K2) {
                        if constexpr (K == 3) asm volatile("st.shared.v2.f32 [%0], {%1, %1};" ::"r"(f + 8u * (uint32_t)(t - kk * K2)), "f"(fv[j] * kF32TcScale) : "memory");
                        else asm volatile("st.shared.f32 [%0], %1;" ::"r"(f + 4u * (uint32_t)(t - kk * K2)), "f"(fv[j] * kF32TcScale) : "memory");
                    }
                }
                if (lw == 0) asm volatile("st.shared.s32 [%0], %1;" ::"r"(slot_s + (uint32_t)(buf * kF32TcChunk + lane) * 4u), "r"(c >= 0 ? slot * P.pitch * 4 : -1) : "memory");
#pragma unroll 1
                for (int s0 = 0; s0 < nslots; s0 += 8)
#pragma unroll 1
                    for (int a0 = 0; a0 < P.np; a0 += 256) {
                        if (s0 + a0) load_round(s0, a0);
                        store_round(xs, s0, a0);
                    }
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_xfull + 8 * buf);
                ++xcnt;
                if (++xq == q1) { xq = q0; xtile += nclusters; }
            }
            if (xtile < P.ntiles) {
                if (xq == q0) {                  // the next tile's table of positions
                    const int bn = xtile / hw, bh = (xtile - bn * hw) / P.tiles_w, bw = xtile - bn * hw - bh * P.tiles_w;
                    named_bar_sync(3, 256);      // the last tile's is not read any more
#pragma unroll 1
                    for (int j = lt; j < P.np; j += 256) {
                        const int px = tab[P.np + j], nl = px >> 20, ih = (px >> 10) & 1023, iw = px & 1023;
                        const int hi = bh * P.PH * P.stride - P.pad + ih, wi = bw * P.PW * P.stride - P.pad + iw;
                        const bool in = bn * P.TN + nl < P.N && hi >= 0 && hi < P.H && wi >= 0 && wi < P.W;
                        tab[j] = in ? (int)(nl * P.xn + hi * P.xh + wi * P.xw) : -1;
                    }
                    named_bar_sync(3, 256);
                    xt = P.x + (long long)bn * P.TN * P.xn;
                }
                c = c_next;
                c_next = chan_of(xq + 1 < q1 ? xq + 1 : q0);
#pragma unroll
                for (int j = 0; j < NF; ++j) {
                    const int t = lt + 256 * j;
                    fv[j] = t < kF32TcChunk * K2 && xq * kF32TcChunk * K2 + t < P.G * K2 ? __ldg(P.dw + xq * kF32TcChunk * K2 + t) : 0.f;
                }
                const int before = __shfl_up_sync(0xffffffffu, c, 1);
                const bool fresh = c >= 0 && (lane == 0 || c != before);       // a channel that begins a new input channel: a slot each
                const uint32_t m = __ballot_sync(0xffffffffu, fresh);
                nslots = __popc(m);
                slot = __popc(m & ((2u << lane) - 1u)) - 1;
                __syncwarp();
                if (fresh) asm volatile("st.shared.s32 [%0], %1;" ::"r"(list_s + 4u * (uint32_t)slot), "r"(c * xc) : "memory");
                __syncwarp();
                load_round(0, 0);
            } else {
                nslots = 0;
            }
            if (s >= 0) {
                f32tc_wait(bar_free + 8 * st, par, &abort_flag, P.status, kStatusWaitStage);
                const uint32_t b_s = ab_s + (uint32_t)st * P.ab_bytes + 3u * kF32TcA + (uint32_t)((ip & 3) * 4);
                if (++q == q1) q = q0;
                const float *const w = w0 + q * kF32TcChunk;
                const bool in0 = q * kF32TcChunk + 2 * ip < P.G, in1 = q * kF32TcChunk + 2 * ip + 1 < P.G;
                const uint32_t swz = b_s + (uint32_t)dr * 64u + (uint32_t)(((ip >> 2) ^ ((dr >> 1) & 3)) << 4);      // rows 16 apart are swizzled alike
#pragma unroll
                for (int j = 0; j < 2 * NB; ++j) {
                    uint32_t p1, p2, p3;
                    f32tc_scale(wv[j][0], wv[j][1]);
                    split3(wv[j][0], wv[j][1], p1, p2, p3);
                    load_w(j, w, in0, in1);
                    if (dr + 16 * j < P.Nd) {
                        const uint32_t a = swz + 1024u * j;
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(p1) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(a + P.b_piece), "r"(p2) : "memory");
                        asm volatile("st.shared.b32 [%0], %1;" ::"r"(a + 2u * P.b_piece), "r"(p3) : "memory");
                    }
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar_full + 8 * st);
                if (++st == P.ns) { st = 0; par ^= 1u; }
                --left;
            }
        }
    } else {
        f32tc_regs_dec<kF32TcRegsMma>();
        if (warp == kF32TcMmaWarp && elect_one()) {
            // ---------------- products ----------------
            const uint32_t idesc = make_idesc(P.Nd, false), hi = (512u >> 4) | (1u << 14) | kF32TcSw64;
            int cnt = 0, st = 0;
            uint32_t par = 0;
#pragma unroll 1
            for (int tile = cluster; tile < P.ntiles; tile += nclusters) {
#pragma unroll 1
                for (int q = q0; q < q1; ++q, ++cnt) {
                    const int buf = cnt & 1;
                    if (cnt >= 2) f32tc_wait(bar_accfree + 8 * buf, (uint32_t)((cnt >> 1) - 1) & 1u, &abort_flag, P.status, kStatusWaitStage);
                    f32tc_wait(bar_full + 8 * st, par, &abort_flag, P.status, kStatusWaitOperand);
                    tc_fence_after();
                    const uint32_t a = ((ab_s + (uint32_t)st * P.ab_bytes) & 0x3FFFFu) >> 4 | (1u << 16), b = ((ab_s + (uint32_t)st * P.ab_bytes + 3u * kF32TcA) & 0x3FFFFu) >> 4 | (1u << 16);
                    const uint32_t d = tmem + (uint32_t)(buf * 32 * NB);
                    // smallest products first: what the accumulator drops when it adds is a share of its value
                    constexpr int za[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
#pragma unroll
                    for (int e = 0; e < 6; ++e)
#pragma unroll
                        for (int k = 0; k < 2; ++k)
                            umma_bf16_words(d, a + za[e] * (kF32TcA >> 4) + 2u * k, hi, b + pb[e] * (P.b_piece >> 4) + 2u * k, hi, idesc, e | k ? 1u : 0u);
                    umma_commit(bar_free + 8 * st);
                    umma_commit(bar_accfull + 8 * buf);
                    if (++st == P.ns) { st = 0; par ^= 1u; }
                }
            }
            // Teardown: one more commit covers every product issued.
            umma_commit(bar_drain);
            mbar_wait_drain(bar_drain, 0);
        }
        __syncwarp();
    }
    if (split > 1 && warp >= kF32TcZWarp) {      // the two of the warps that finish y
        cluster_sync();
        cluster_sync();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kF32TcMmaWarp) tmem_dealloc(tmem, 64u * NB);
}

namespace {

// Most distinct input channels that a chunk reads.
int f32tc_slots(const gdws_plan_s *p)
{
    int most = 0;
    for (int i0 = 0; i0 < p->G; i0 += kF32TcChunk) {
        int n = 0;
        for (int i = i0; i < std::min(p->G, i0 + kF32TcChunk); ++i) n += i == i0 || p->chan[i] != p->chan[i - 1];
        most = std::max(most, n);
    }
    return most;
}

struct F32TcGeom {
    int TN = 0, PH = 0, PW = 0, IH = 0, IW = 0, np = 0, pitch = 0, tiles_h = 0, tiles_w = 0, ns = 0, nb = 0, Nd = 0, split = 1;
    long long tiles = 0;
    double us = 0;
};

struct F32TcLaunch {
    LaunchKey key;
    F32TcGeom g;
    bool taken = false;
    int alu = -1;                // fused_f32_kernel's tile
    int slots = 0;               // most distinct input channels that a chunk reads
};

size_t f32tc_smem(const gdws_plan_s *p, int slots, const F32TcGeom &g)
{
    return 1024 + (size_t)g.ns * (3 * kF32TcA + 3 * (size_t)g.Nd * 64) + 2 * (size_t)slots * g.pitch * 4 + (2 * (size_t)f32tc_filt_pitch(p->k) + 10) * kF32TcChunk * 4 +
           (size_t)g.np * 8 + 4 * 32 * (size_t)g.nb + 4 * 32 * 17 * 4 + 64;
}

// Tile shape: the pixels of a tile are a patch of one image or whole small images, whatever fills 128 rows best.
bool f32tc_geometry(const gdws_plan_s *p, int n, int Ho, int Wo, long long xn, int slots, F32TcGeom *out)
{
    if ((p->k != 3 && p->k != 5) || p->G < 1) return false;
    const int sms = sm_count_of(p), nq = (p->G + kF32TcChunk - 1) / kF32TcChunk;
    const int parts = (p->D + 127) / 128;
    bool found = false;
    auto consider = [&](int TN, int PH, int PW) {
        F32TcGeom g;
        g.TN = TN; g.PH = PH; g.PW = PW;
        g.IH = (PH - 1) * p->stride + p->k; g.IW = (PW - 1) * p->stride + p->k;
        const long long np = (long long)TN * g.IH * g.IW;
        if (np > kF32TcMaxPos || TN * xn > 0x7fffffffLL) return;
        g.np = (int)np;
        g.pitch = (g.np + 3) / 8 * 8 + 4;        // an odd multiple of 4: 8 channels x 4 positions fall into 32 banks
        g.tiles_h = (Ho + PH - 1) / PH; g.tiles_w = (Wo + PW - 1) / PW;
        g.tiles = (long long)((n + TN - 1) / TN) * g.tiles_h * g.tiles_w;
        g.Nd = parts > 1 ? 128 : (p->D + 15) / 16 * 16;
        g.nb = g.Nd <= 32 ? 1 : (g.Nd <= 64 ? 2 : 4);
        for (g.ns = kF32TcMaxStages; g.ns >= 2; --g.ns)
            if (f32tc_smem(p, slots, g) <= (size_t)kMaxSmem) break;
        if (g.ns < 2) return;
        const long long waves = (g.tiles * parts + sms - 1) / sms;
        // Fitted to 40 layers: a chunk takes 1.5 us and more with more output channels and rounds of staged input (8 channels x 256
        // positions), a tile what its stores take, clusters the adding up.
        const int rounds = (slots + 7) / 8 * ((g.np + 255) / 256);
        const double chunk = (p->k == 3 ? 1.5 : 1.9) + 0.006 * g.Nd + 0.35 * (rounds - 1);
        for (g.split = 1; g.split <= 8 && g.split <= nq; g.split *= 2) {
            if (g.split > 1 && g.tiles * parts > cluster_capacity(p, g.split)) break;        // one wave
            g.us = 5.0 + (double)waves * ((nq + g.split - 1) / g.split * chunk + 0.01 * g.Nd) + (g.split > 1 ? 2.5 : 0.0) + 1e-4 * g.np;
            if (!found || g.us < out->us) { *out = g; found = true; }
        }
    };
    // A row or column in so many equal parts: only those numbers are visited that change the parts' size (500 x 500 outputs: 700 us of a
    // first call with all of them).
    auto next = [](int total, int parts) { const int size = (total + parts - 1) / parts; return size > 1 ? (total + size - 2) / (size - 1) : total + 1; };
    for (int j = (Wo + 127) / 128; j <= Wo; j = next(Wo, j)) {
        const int PW = (Wo + j - 1) / j, most = 128 / PW;
        if (PW < 4 && PW < Wo) break;
        for (int i = (Ho + most - 1) / most; i <= Ho; i = next(Ho, i)) {
            const int PH = (Ho + i - 1) / i;
            if (i == 1 && j == 1) {
                for (int TN = std::min(n, 128 / (PH * PW)); TN >= 1; --TN) consider(TN, PH, PW);
            } else {
                consider(1, PH, PW);
            }
            if (PH * PW < 32) break;
        }
    }
    return found && out->tiles <= 0x3fffffffLL;
}

template <int K, int NB, bool NHWC> gdws_status_t f32tc_launch(gdws_plan_s *p, const F32TcGeom &g, const F32TcParams &P, size_t smem, cudaStream_t st)
{
    auto kernel = f32_tc_kernel<K, NB, NHWC>;
    static bool attr_set[64] = {};
    if (!attr_set[p->device & 63]) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(f32_tc_kernel)");
        cudaFuncAttributes a;
        if (cudaFuncGetAttributes(&a, kernel) != cudaSuccess || a.numRegs < kF32TcRegsLaunch) return fail(GDWS_ERR_UNSUPPORTED, "f32_tc_kernel: register split needs %d registers at launch", kF32TcRegsLaunch);
        attr_set[p->device & 63] = true;
    }
    const int parts = (p->D + 127) / 128;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.split * std::min<long long>(g.tiles, std::max(1, sm_count_of(p) / (g.split * parts)))), (unsigned)parts);
    cfg.blockDim = dim3(kF32TcThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)g.split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = g.split > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, P, g.split);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "f32_tc_kernel launch"); }
    p->launches++;
    return GDWS_OK;
}

}  // namespace

// Whether a forward of this size runs here; the geometry is worked out once per size.
static const F32TcLaunch *f32tc_prepared(gdws_plan_s *p, int n, int h, int w)
{
    const LaunchKey key = {n, h, w, p->opt_dw_math};
    if (const F32TcLaunch *l = LaunchCache<F32TcLaunch>::find(p->launch_cache[kCacheF32], key)) return l;
    std::unique_ptr<F32TcLaunch> e(new (std::nothrow) F32TcLaunch);
    if (!e) return nullptr;
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    e->key = key;
    e->alu = f32_alu_config(p, (long long)n * Ho * Wo, Wo);
    if (p->opt_dw_math != 1) {
        e->slots = f32tc_slots(p);
        e->taken = f32tc_geometry(p, n, Ho, Wo, (long long)p->C * h * w, e->slots, &e->g);
    }
    // The other kernel's estimate is too long for short calls (5 x 32 -> 81 channels at 11 x 9, stride 2: 17.6 for 11.9 us, where this one
    // takes 14.8) and up to twice too short for large NHWC ones.
    const double alu = f32_alu_us(p, n, h, w);
    if (e->taken && p->opt_dw_math != 2) e->taken = p->G >= kF32TcLeast && e->g.us < (alu < 24.0 ? 3.0 + 0.65 * (alu - 3.0) : 1.1 * alu);
    return LaunchCache<F32TcLaunch>::add(p->launch_cache[kCacheF32], std::move(e));
}

bool f32_tc_takes(gdws_plan_s *p, int n, int h, int w, int *alu)
{
    const F32TcLaunch *l = f32tc_prepared(p, n, h, w);
    if (l) *alu = l->alu;
    return l && l->taken;
}

// Estimate of an fp32 forward of n images, for gdws_forward_host.
double f32_forward_us(gdws_plan_s *p, int n, int h, int w)
{
    const F32TcLaunch *l = f32tc_prepared(p, n, h, w);
    return l && l->taken ? l->g.us : f32_alu_us(p, n, h, w);
}

gdws_status_t f32_fused_tc(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, const float *pw_w, const float *bias, gdws_tensor_t *y, cudaStream_t st)
{
    const F32TcLaunch *l = f32tc_prepared(p, x->n, x->h, x->w);
    if (!l || !l->taken) return fail(GDWS_ERR_UNSUPPORTED, "fp32 tensor-core path: layer not covered");
    const F32TcGeom &g = l->g;
    const long long xn = (long long)x->c * x->h * x->w, yn = (long long)y->c * y->h * y->w;
    const bool nhwc = x->layout == GDWS_NHWC;
    F32TcParams P;
    memset(&P, 0, sizeof(P));
    P.x = (const float *)x->ptr; P.dw = dw_w; P.pw = pw_w; P.bias = bias; P.chan = p->d_chan; P.y = (float *)y->ptr; P.status = p->d_status;
    P.N = x->n; P.H = x->h; P.W = x->w; P.D = p->D; P.G = p->G; P.stride = p->stride; P.pad = p->pad; P.Ho = y->h; P.Wo = y->w; P.relu = p->opt_relu;
    P.xn = xn; P.yn = yn;
    P.xc = nhwc ? 1 : (long long)x->h * x->w; P.xw = nhwc ? x->c : 1; P.xh = P.xw * x->w;
    P.yc = nhwc ? 1 : (long long)y->h * y->w; P.yw = nhwc ? y->c : 1; P.yh = P.yw * y->w;
    P.TN = g.TN; P.PH = g.PH; P.PW = g.PW; P.IH = g.IH; P.IW = g.IW; P.np = g.np; P.pitch = g.pitch; P.tiles_h = g.tiles_h; P.tiles_w = g.tiles_w; P.ntiles = (int)g.tiles;
    P.nq = (p->G + kF32TcChunk - 1) / kF32TcChunk; P.Nd = g.Nd; P.ns = g.ns;
    const int slots = l->slots;
    P.b_piece = (uint32_t)g.Nd * 64u; P.ab_bytes = 3u * kF32TcA + 3u * P.b_piece;
    P.x_bytes = (uint32_t)slots * (uint32_t)g.pitch * 4u;
    P.off_x = (uint32_t)g.ns * P.ab_bytes;
    P.off_f = P.off_x + 2u * P.x_bytes;
    P.off_slot = P.off_f + 2u * kF32TcChunk * (uint32_t)f32tc_filt_pitch(p->k) * 4u;
    P.off_tab = P.off_slot + 10u * kF32TcChunk * 4u;      // two chunks' offsets, the eight loading warps' lists
    P.off_bias = P.off_tab + ((uint32_t)g.np * 8u + 15u) / 16u * 16u;
    size_t smem = f32tc_smem(p, slots, g);
    if (g.split > 1) smem = std::max(smem, (size_t)1024 + 128 * 32 * (size_t)g.nb * 4);      // the sums on their way
    const auto launch = [&](auto k) -> gdws_status_t {
        constexpr int K = decltype(k)::value;
        if (nhwc) return g.nb == 1 ? f32tc_launch<K, 1, true>(p, g, P, smem, st) : (g.nb == 2 ? f32tc_launch<K, 2, true>(p, g, P, smem, st) : f32tc_launch<K, 4, true>(p, g, P, smem, st));
        return g.nb == 1 ? f32tc_launch<K, 1, false>(p, g, P, smem, st) : (g.nb == 2 ? f32tc_launch<K, 2, false>(p, g, P, smem, st) : f32tc_launch<K, 4, false>(p, g, P, smem, st));
    };
    return p->k == 3 ? launch(std::integral_constant<int, 3>()) : launch(std::integral_constant<int, 5>());
}

}  // namespace gdws
