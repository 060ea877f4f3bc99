// fp32 kernels (NCHW or NHWC through explicit strides).  Plain FFMA on both stages: the tensor cores have no full-fp32 mode and TF32
// would miss the 1e-4 parity bound.  Larger layers of 3 x 3 and 5 x 5 filters run in f32_tc.cu (three bf16 pieces per value).
#include <algorithm>

#include "gdws_internal.h"

namespace gdws {

struct F32Shape {
    int N, C, H, W, D, G, k, stride, pad, Ho, Wo, relu;
    // element strides of x (xn, xc, xh, xw), of z / y (channel count G / D) in the same layout
    long long xn, xc, xh, xw;
    long long zn, zc, zh, zw;
    long long yn, yc, yh, yw;
};

static F32Shape make_shape(const gdws_plan_s *p, gdws_layout_t layout, int N, int H, int W)
{
    F32Shape s;
    s.N = N; s.C = p->C; s.H = H; s.W = W; s.D = p->D; s.G = p->G; s.k = p->k; s.stride = p->stride; s.pad = p->pad;
    s.Ho = gdws_out_dim(H, p->k, p->stride, p->pad);
    s.Wo = gdws_out_dim(W, p->k, p->stride, p->pad);
    s.relu = p->opt_relu;
    if (layout == GDWS_NCHW) {
        s.xw = 1; s.xh = W; s.xc = (long long)H * W; s.xn = s.xc * s.C;
        s.zw = 1; s.zh = s.Wo; s.zc = (long long)s.Ho * s.Wo; s.zn = s.zc * s.G;
        s.yw = 1; s.yh = s.Wo; s.yc = (long long)s.Ho * s.Wo; s.yn = s.yc * s.D;
    } else {
        s.xc = 1; s.xw = s.C; s.xh = (long long)W * s.C; s.xn = s.xh * H;
        s.zc = 1; s.zw = s.G; s.zh = (long long)s.Wo * s.G; s.zn = s.zh * s.Ho;
        s.yc = 1; s.yw = s.D; s.yh = (long long)s.Wo * s.D; s.yn = s.yh * s.Ho;
    }
    return s;
}

// One depthwise output: sum over the k x k window of channel c at output (ho, wo), zero padding.
__device__ __forceinline__ float dw_point(const F32Shape &s, const float *__restrict__ xc,
                                          const float *__restrict__ ker, int ho, int wo)
{
    float acc = 0.f;
    for (int u = 0; u < s.k; ++u) {
        const int hi = ho * s.stride + u - s.pad;
        if (hi < 0 || hi >= s.H) continue;
        for (int v = 0; v < s.k; ++v) {
            const int wi = wo * s.stride + v - s.pad;
            if (wi < 0 || wi >= s.W) continue;
            acc = fmaf(__ldg(ker + u * s.k + v), __ldg(xc + hi * s.xh + wi * s.xw), acc);
        }
    }
    return acc;
}

// z[n,i,ho,wo]: one thread per element; threads run along wo (NCHW) so reads of x coalesce.
__global__ void gdw_f32_kernel(F32Shape s, const float *__restrict__ x, const float *__restrict__ dw,
                               const int32_t *__restrict__ chan, float *__restrict__ z)
{
    const long long total = (long long)s.N * s.G * s.Ho * s.Wo;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int wo = (int)(t % s.Wo);
        long long r = t / s.Wo;
        const int ho = (int)(r % s.Ho);
        r /= s.Ho;
        const int i = (int)(r % s.G);
        const int n = (int)(r / s.G);
        const int c = chan[i];
        const float v = dw_point(s, x + n * s.xn + c * s.xc, dw + (size_t)i * s.k * s.k, ho, wo);
        z[n * s.zn + i * s.zc + ho * s.zh + wo * s.zw] = v;
    }
}

// y[n,d,ho,wo] = bias[d] + sum_i P[d,i] z[n,i,ho,wo]: one thread per element.
__global__ void pw_f32_kernel(F32Shape s, const float *__restrict__ z, const float *__restrict__ pw,
                              const float *__restrict__ bias, float *__restrict__ y)
{
    const long long total = (long long)s.N * s.D * s.Ho * s.Wo;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int wo = (int)(t % s.Wo);
        long long r = t / s.Wo;
        const int ho = (int)(r % s.Ho);
        r /= s.Ho;
        const int d = (int)(r % s.D);
        const int n = (int)(r / s.D);
        const float *zp = z + n * s.zn + ho * s.zh + wo * s.zw;
        const float *pp = pw + (size_t)d * s.G;
        float acc = 0.f;
        for (int i = 0; i < s.G; ++i) acc = fmaf(__ldg(pp + i), __ldg(zp + i * s.zc), acc);
        acc += bias ? __ldg(bias + d) : 0.f;
        if (s.relu) acc = fmaxf(acc, 0.f);
        y[n * s.yn + d * s.yc + ho * s.yh + wo * s.yw] = acc;
    }
}

// Fused fp32 forward: y[pixels x D] = z[pixels x G] P^T as a register-tiled product whose z operand is produced on the way.
// A block owns PT output pixels (consecutive in n, h', w') x DT output channels; a thread TP x TD of them.  K runs over
// chunks of kF32KC intermediate channels, staged two chunks ahead by 4-byte asynchronous copies: the pointwise weights
// (transposed on the way to [channel][output channel]), the filters, and of each input channel the rows the tile's windows
// read, zeros outside the image filled in.  NP producer threads start the copies and compute the next chunk's z from
// shared memory while the other threads multiply this chunk; one barrier per chunk.  (In the multiplying threads' own
// program order, copies and z cost their full latency on top: 105 us for 16 x 128 -> 128 channels at 28 x 28,
// G = 640, NCHW, 39 of them for the products; 84 now.)
// KS groups of threads share a tile: each multiplies its share of a chunk's channels, and the sums meet in shared memory at
// the end.  (One group of 8 x 8 thread tiles leaves 1.5 warps per scheduler, which cannot cover their own latencies.)
// What bounds it: the FFMA pipe (G (k^2 + D) multiply-adds per pixel; nothing faster keeps fp32 products and sums).  The
// packed form (two multiply-adds per instruction, same rate) leaves every other issue slot to loads and staging.  Large
// thread tiles need fewer loads per multiply-add, small ones spread small layers over more SMs (f32_config chooses).  z straight from global memory, without the staging, took 870 cycles per
// channel and thread: 139 us on that layer.
constexpr int kF32KC = 16;

__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, bool valid)
{
    const int n = valid ? 4 : 0;      // 0: the four bytes are filled with zeros
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}

// Elements e of a thread's T along an axis of N threads: groups of 4 that neighbouring threads interleave.
template <int T, int N> __device__ __forceinline__ constexpr int f32_pos(int idx, int e)
{
    return T == 8 ? (e >> 2) * (N * 4) + idx * 4 + (e & 3) : idx * T + e;
}
template <int T, int N> __device__ __forceinline__ void f32_frag(const float *row, int idx, float (&v)[T])
{
    if constexpr (T >= 4) {
#pragma unroll
        for (int q = 0; q < T / 4; ++q) {
            const float4 f = *reinterpret_cast<const float4 *>(row + f32_pos<T, N>(idx, 4 * q));
            v[4 * q] = f.x; v[4 * q + 1] = f.y; v[4 * q + 2] = f.z; v[4 * q + 3] = f.w;
        }
    } else if constexpr (T == 2) {
        const float2 f = *reinterpret_cast<const float2 *>(row + 2 * idx);
        v[0] = f.x; v[1] = f.y;
    } else {
        v[0] = row[idx];
    }
}
__device__ __forceinline__ void named_bar(int id, int count) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory"); }
// acc.{lo, hi} += a.{lo, hi} * b.{lo, hi}, each with one rounding.
__device__ __forceinline__ void ffma2(float &lo, float &hi, float a0, float a1, float b0, float b1)
{
    asm("{\n\t.reg .b64 a, b, c;\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "mov.b64 b, {%4, %5};\n\t"
        "mov.b64 c, {%0, %1};\n\t"
        "fma.rn.f32x2 c, a, b, c;\n\t"
        "mov.b64 {%0, %1}, c;\n\t}"
        : "+f"(lo), "+f"(hi) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// Positions of a tile's staged input rows: output pixel j of the tile (0 .. PT-1) lies in the tile's r-th output row; its
// window starts at position j * stride + r * max(0, k - stride) of each of the k staged rows, so that windows of one output
// row overlap as they do in the image and different output rows do not touch.
__host__ __device__ inline int f32_row_len(int pt, int Wo, int k, int stride)
{
    const int rows = (pt + Wo - 2) / Wo + 1;
    return pt * stride + rows * (k > stride ? k - stride : 0);
}
__host__ __device__ constexpr int f32_filt_pitch(int k2) { return (k2 + 3) / 4 * 4; }

// K: filter size with the input window in registers (1, 3, 5), 0: any.
template <int PT, int DT, int TP, int TD, int KS, int NP, int K, bool NHWC>
__global__ void __launch_bounds__((PT / TP) * (DT / TD) * KS + NP, TP * TD <= 16 ? 3 : (TP * TD == 32 ? 2 : 1))
fused_f32_kernel(F32Shape s, const float *__restrict__ x, const float *__restrict__ dw, const float *__restrict__ pw,
                 const float *__restrict__ bias, const int32_t *__restrict__ chan, float *__restrict__ y)
{
    constexpr int NX = PT / TP, NY = DT / TD, NC = NX * NY * KS, T = NC + NP, KC = kF32KC, WC = NC / 32, WP = NP / 32;
    static_assert(WC % KS == 0 && WP % 2 == 0 && KC % KS == 0, "warps share staging and chunks evenly");
    constexpr int LX = NX % 8 == 0 ? 8 : 4, NXW = NX / LX;           // a warp covers LX x 32 / LX threads
    constexpr int ZS = PT + 4, PS = DT + 4;
    const int k = K ? K : s.k, k2 = k * k, fp = f32_filt_pitch(k2);
    const int L = f32_row_len(PT, s.Wo, k, s.stride), kL = k * L;
    extern __shared__ __align__(16) float sm[];
    float *const zb = sm, *const pb = zb + 2 * KC * ZS, *const fb = pb + 3 * KC * PS, *const xb = fb + 2 * KC * fp;
    long long *const tab = reinterpret_cast<long long *>(xb + 2 * KC * kL);      // per staged position: offset in x (channel 0), -1: outside
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int grp = KS == 1 ? 0 : warp / (WC / KS), gw = KS == 1 ? warp : warp % (WC / KS);
    const bool producer = warp >= WC;
    const int pt = tid - NC, pwarp = warp - WC;
    const int tx = (gw % NXW) * LX + lane % LX, ty = (gw / NXW) * (32 / LX) + lane / LX;
    const long long npix = (long long)s.N * s.Ho * s.Wo;
    const long long p0 = (long long)blockIdx.x * PT;
    const int d0 = (int)blockIdx.y * DT;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    for (int j = tid; j < kL; j += T) tab[j] = -1;
    __syncthreads();
    const int ext = k > s.stride ? k - s.stride : 0;
    const int wo0 = (int)(p0 % s.Wo);
    for (int j = tid; j < PT; j += T) {
        const long long p = p0 + j;
        if (p < npix) {
            const int r = (wo0 + j) / s.Wo, wo = (wo0 + j) - r * s.Wo;
            const long long row = p / s.Wo;
            const int ho = (int)(row % s.Ho), n = (int)(row / s.Ho);
            const int hi = ho * s.stride - s.pad, wi = wo * s.stride - s.pad, q0 = j * s.stride + r * ext;
            const bool last = wo == s.Wo - 1 || j == PT - 1 || p == npix - 1;
            const int nv = last ? k : (k < s.stride ? k : s.stride);      // the positions this window does not share with the next one
            for (int u = 0; u < k; ++u)
                for (int v = 0; v < nv; ++v)
                    if (hi + u >= 0 && hi + u < s.H && wi + v >= 0 && wi + v < s.W)
                        tab[u * L + q0 + v] = n * s.xn + (hi + u) * s.xh + (wi + v) * s.xw;
        }
    }
    constexpr int NI = NP / PT > 0 ? NP / PT : 1, PER = KC / NI;       // producer threads per pixel, each with PER consecutive channels of z
    static_assert((NI * PT == NP || PT == 96) && PER * NI == KC, "z phase covers the chunk");
    const int zpx = pt % PT, zi = pt / PT;
    const int zq = p0 + zpx < npix ? zpx * s.stride + (wo0 + zpx) / s.Wo * ext : 0;
    int zqs[PT >= 32 ? PT / 32 : 1];                 // the same per group of 32 pixels
    if constexpr (PT >= 32)
#pragma unroll
        for (int g = 0; g < PT / 32; ++g) {
            const int j = 32 * g + lane;
            zqs[g] = p0 + j < npix ? j * s.stride + (wo0 + j) / s.Wo * ext : 0;
        }
    const int nq = (s.G + KC - 1) / KC;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    auto chan_of = [&](int q) { const int i = q * KC + lane; return lane < KC && i < s.G ? __ldg(chan + i) : -1; };
    int c_next = chan_of(0);
    __syncthreads();

    // Starts chunk q's copies.  Returns the chunk's channels that begin a new input channel, as a mask: a staged slot each.
    auto stage = [&](int q) -> uint32_t {
        const int c = c_next;
        c_next = q + 1 < nq ? chan_of(q + 1) : -1;
        const int before = __shfl_up_sync(0xffffffffu, c, 1);
        const uint32_t m = __ballot_sync(0xffffffffu, c >= 0 && (lane == 0 || c != before));
        {
            // 8 channels x 4 output channels per warp and step: whole sectors in, 32 different banks out
            const int kk = (pwarp & 1) * 8 + (lane & 7), dl0 = (pwarp >> 1) * 4 + (lane >> 3);
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(pb + (q % 3) * KC * PS + kk * PS + dl0);
            const bool in = q * KC + kk < s.G;
            const float *src = pw + (size_t)(d0 + dl0) * s.G + q * KC + kk;
#pragma unroll
            for (int t = 0; t < (DT + 2 * WP - 1) / (2 * WP); ++t, src += (size_t)2 * WP * s.G) {
                if (DT % (2 * WP) && dl0 + t * 2 * WP >= DT) break;
                const bool ok = in && d0 + dl0 + t * 2 * WP < s.D;
                cp_async4(dst + t * 2 * WP * 4, ok ? src : pw, ok);
            }
        }
        {
            float *dst = fb + (q & 1) * KC * fp;
            const int n = min(KC, s.G - q * KC) * k2;
            for (int t = pt; t < KC * k2; t += NP) {
                const int kk = t / k2;
                cp_async4((uint32_t)__cvta_generic_to_shared(dst + kk * fp + (t - kk * k2)), t < n ? dw + (size_t)q * KC * k2 + t : dw, t < n);
            }
        }
        const uint32_t xs = (uint32_t)__cvta_generic_to_shared(xb + (q & 1) * KC * kL);
        if constexpr (!NHWC) {
            uint32_t slot = xs;
            for (uint32_t mm = m; mm; mm &= mm - 1, slot += (uint32_t)kL * 4) {
                const float *xc = x + __shfl_sync(0xffffffffu, c, __ffs(mm) - 1) * s.xc;
                for (int j = pt; j < kL; j += NP) {
                    const long long o = tab[j];
                    cp_async4(slot + (uint32_t)j * 4, o >= 0 ? xc + o : x, o >= 0);
                }
            }
        } else {
            // neighbouring lanes take neighbouring channels of one position
            const int ns = __popc(m), sl = lane & (KC - 1);
            const int cs = __shfl_sync(0xffffffffu, c, sl < ns ? (int)__fns(m, 0, sl + 1) : 0);
            if (sl < ns)
                for (int j = pwarp * (32 / KC) + lane / KC; j < kL; j += NP / KC) {
                    const long long o = tab[j];
                    cp_async4(xs + (uint32_t)(sl * kL + j) * 4, o >= 0 ? x + o + cs : x, o >= 0);
                }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        return m;
    };
    // z of a chunk.  Tiles of 32 pixels and more: a warp takes PW consecutive channels and all PG groups of 32 pixels, lanes =
    // pixels, so that a filter in registers serves PG pixels and a window all filters of its input channel (both come from
    // shared memory, whose bandwidth the products need: 16 cycles of it per 16 cycles of multiply-adds).
    auto make_z = [&](int q, uint32_t m) {
        const float *fs = fb + (q & 1) * KC * fp;
        if constexpr (PT >= 32 && K != 0 && K <= 3) {
            constexpr int PG = PT / 32, PW = KC / WP > 0 ? KC / WP : 1;
            static_assert(WP * PW == KC, "warps share the chunk");
            const float *xs = xb + (q & 1) * KC * kL;
            float *dst = zb + (q & 1) * KC * ZS + lane;
            float acc[PW][PG];
            float w[PW][f32_filt_pitch(K * K)];
#pragma unroll
            for (int j = 0; j < PW; ++j)
#pragma unroll
                for (int t = 0; t < f32_filt_pitch(K * K) / 4; ++t)
                    *reinterpret_cast<float4 *>(&w[j][4 * t]) = *reinterpret_cast<const float4 *>(fs + (pwarp * PW + j) * fp + 4 * t);
#pragma unroll
            for (int g = 0; g < PG; ++g) {
                float xr[K * K];
#pragma unroll
                for (int j = 0; j < PW; ++j) {
                    const int kk = pwarp * PW + j;
                    if (j == 0 || ((m >> kk) & 1u)) {      // the same for the whole warp
                        const float *xc = xs + max(__popc(m & ((2u << kk) - 1u)) - 1, 0) * kL + zqs[g];
#pragma unroll
                        for (int u = 0; u < K; ++u)
#pragma unroll
                            for (int v = 0; v < K; ++v) xr[u * K + v] = xc[u * L + v];
                    }
                    float a = 0.f;
#pragma unroll
                    for (int t = 0; t < K * K; ++t) a = fmaf(w[j][t], xr[t], a);
                    acc[j][g] = a;
                }
            }
#pragma unroll
            for (int j = 0; j < PW; ++j)
#pragma unroll
                for (int g = 0; g < PG; ++g) dst[(pwarp * PW + j) * ZS + 32 * g] = q * KC + pwarp * PW + j < s.G ? acc[j][g] : 0.f;      // i >= G: not 0 * x, x may be infinite
            return;
        } else {
            if (pt >= NI * PT) return;
            float *dst = zb + (q & 1) * KC * ZS + zpx;
            const float *xs = xb + (q & 1) * KC * kL + zq;
#pragma unroll (PER < 4 ? PER : 4)
            for (int j = 0; j < PER; ++j) {
                const int kk = zi * PER + j;
                const int slot = max(__popc(m & ((2u << kk) - 1u)) - 1, 0);
                const float *xc = xs + slot * kL, *ker = fs + kk * fp;
                float acc = 0.f;
                if constexpr (K != 0) {
#pragma unroll
                    for (int u = 0; u < K; ++u)
#pragma unroll
                        for (int v = 0; v < K; ++v) acc = fmaf(ker[u * K + v], xc[u * L + v], acc);
                } else {
                    for (int u = 0; u < k; ++u)
                        for (int v = 0; v < k; ++v) acc = fmaf(ker[u * k + v], xc[u * L + v], acc);
                }
                dst[kk * ZS] = q * KC + kk < s.G ? acc : 0.f;
            }
        }
    };

    if (producer) {
        uint32_t m1 = stage(0);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        named_bar(1, NP);
        if (nq > 1) {
            const uint32_t m = m1;
            m1 = stage(1);
            make_z(0, m);
        } else {
            make_z(0, m1);
        }
#pragma unroll 1
        for (int q = 0; q < nq; ++q) {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            __syncthreads();     // chunk q + 1 is staged, z of chunk q written, what chunk q - 1 used may be overwritten
            uint32_t m2 = 0;
            if (q + 2 < nq) m2 = stage(q + 2);
            if (q + 1 < nq) make_z(q + 1, m1);
            m1 = m2;
        }
        if constexpr (KS > 1) {
#pragma unroll 1
            for (int half = 0; half < 4; ++half) __syncthreads();
        }
        return;
    }
    float acc[TP][TD];
#pragma unroll
    for (int e = 0; e < TP; ++e)
#pragma unroll
        for (int f = 0; f < TD; ++f) acc[e][f] = 0.f;
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
        __syncthreads();
        const float *zc = zb + (q & 1) * KC * ZS, *pc = pb + (q % 3) * KC * PS;
#pragma unroll 8
        for (int j = 0; j < KC / KS; ++j) {
            const int kk = grp * (KC / KS) + j;
            float zv[TP], pv[TD];
            f32_frag<TP, NX>(zc + kk * ZS, tx, zv);
            f32_frag<TD, NY>(pc + kk * PS, ty, pv);
            if constexpr (TP % 2 == 0) {
#pragma unroll
                for (int f = 0; f < TD; ++f)
#pragma unroll
                    for (int e = 0; e < TP; e += 2) ffma2(acc[e][f], acc[e + 1][f], zv[e], zv[e + 1], pv[f], pv[f]);
            } else {
#pragma unroll
                for (int e = 0; e < TP; ++e)
#pragma unroll
                    for (int f = 0; f < TD; ++f) acc[e][f] = fmaf(zv[e], pv[f], acc[e][f]);
            }
        }
    }
    if constexpr (KS > 1) {      // the other group's sums, through what were the operand buffers
        static_assert(KS == 2 && 2 * KC * ZS + 3 * KC * PS >= (TP * TD / 2) * (NC / KS), "half of a group's sums fit");
        const int lt = tid % (NC / KS);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            __syncthreads();
            if (grp == 1) {
#pragma unroll
                for (int e = half * (TP / 2); e < (half + 1) * (TP / 2); ++e)
#pragma unroll
                    for (int f = 0; f < TD; ++f) sm[((e - half * (TP / 2)) * TD + f) * (NC / KS) + lt] = acc[e][f];
            }
            __syncthreads();
            if (grp == 0) {
#pragma unroll
                for (int e = half * (TP / 2); e < (half + 1) * (TP / 2); ++e)
#pragma unroll
                    for (int f = 0; f < TD; ++f) acc[e][f] += sm[((e - half * (TP / 2)) * TD + f) * (NC / KS) + lt];
            }
        }
        if (grp == 1) return;
    }

    // bias, ReLU, store: 16 bytes at a time where four pixels (NCHW) or four channels (NHWC) lie together and aligned
    const int hw = s.Ho * s.Wo;
    const bool vec = NHWC ? s.D % 4 == 0 : hw % 4 == 0;
#pragma unroll
    for (int f = 0; f < TD; ++f) {
        const int d = d0 + f32_pos<TD, NY>(ty, f);
        const float b = (bias && d < s.D) ? __ldg(bias + d) : 0.f;
#pragma unroll
        for (int e = 0; e < TP; ++e) {
            acc[e][f] += b;
            if (s.relu) acc[e][f] = fmaxf(acc[e][f], 0.f);
        }
    }
    if constexpr (!NHWC) {
#pragma unroll
        for (int e = 0; e < TP; e += TP >= 4 ? 4 : 1) {
            const long long p = p0 + f32_pos<TP, NX>(tx, e);
            if (p >= npix) continue;
#pragma unroll
            for (int f = 0; f < TD; ++f) {
                const int d = d0 + f32_pos<TD, NY>(ty, f);
                if (d >= s.D) continue;
                if constexpr (TP >= 4) {
                    if (vec) {
                        *reinterpret_cast<float4 *>(y + (p / hw) * s.yn + d * s.yc + p % hw) = make_float4(acc[e][f], acc[e + 1][f], acc[e + 2][f], acc[e + 3][f]);
                    } else {
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (p + g < npix) y[((p + g) / hw) * s.yn + d * s.yc + (p + g) % hw] = acc[e + g][f];
                    }
                } else {
                    y[(p / hw) * s.yn + d * s.yc + p % hw] = acc[e][f];
                }
            }
        }
    } else {
#pragma unroll
        for (int e = 0; e < TP; ++e) {
            const long long p = p0 + f32_pos<TP, NX>(tx, e);
            if (p >= npix) continue;
#pragma unroll
            for (int f = 0; f < TD; f += TD >= 4 ? 4 : 1) {
                const int d = d0 + f32_pos<TD, NY>(ty, f);
                if (d >= s.D) continue;
                if constexpr (TD >= 4) {
                    if (vec) {
                        *reinterpret_cast<float4 *>(y + p * s.D + d) = make_float4(acc[e][f], acc[e][f + 1], acc[e][f + 2], acc[e][f + 3]);
                    } else {
#pragma unroll
                        for (int g = 0; g < 4; ++g)
                            if (d + g < s.D) y[p * s.D + d + g] = acc[e][f + g];
                    }
                } else {
                    y[p * s.D + d] = acc[e][f];
                }
            }
        }
    }
}

static int grid_for(const gdws_plan_s *p, long long total, int block)
{
    long long b = (total + block - 1) / block;
    const long long cap = (long long)sm_count_of(p) * 16;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

gdws_status_t f32_depthwise(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, float *z, cudaStream_t st)
{
    const F32Shape s = make_shape(p, x->layout, x->n, x->h, x->w);
    const long long total = (long long)s.N * s.G * s.Ho * s.Wo;
    gdw_f32_kernel<<<grid_for(p, total, 256), 256, 0, st>>>(s, (const float *)x->ptr, dw_w, p->d_chan, z);
    p->launches++;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GDWS_OK : cuda_fail(e, "gdw_f32_kernel launch");
}

gdws_status_t f32_pointwise(gdws_plan_s *p, const float *z, const float *pw_w, const float *bias,
                            gdws_tensor_t *y, cudaStream_t st)
{
    F32Shape s = make_shape(p, y->layout, y->n, 1, 1);
    s.Ho = y->h; s.Wo = y->w;
    // strides of z and y depend only on the output extents
    if (y->layout == GDWS_NCHW) {
        s.zw = 1; s.zh = s.Wo; s.zc = (long long)s.Ho * s.Wo; s.zn = s.zc * s.G;
        s.yw = 1; s.yh = s.Wo; s.yc = (long long)s.Ho * s.Wo; s.yn = s.yc * s.D;
    } else {
        s.zc = 1; s.zw = s.G; s.zh = (long long)s.Wo * s.G; s.zn = s.zh * s.Ho;
        s.yc = 1; s.yw = s.D; s.yh = (long long)s.Wo * s.D; s.yn = s.yh * s.Ho;
    }
    const long long total = (long long)s.N * s.D * s.Ho * s.Wo;
    pw_f32_kernel<<<grid_for(p, total, 256), 256, 0, st>>>(s, z, pw_w, bias, (float *)y->ptr);
    p->launches++;
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? GDWS_OK : cuda_fail(e, "pw_f32_kernel launch");
}

namespace {

size_t f32_smem(int pt, int dt, int Wo, int k, int stride)
{
    const size_t kL = (size_t)k * f32_row_len(pt, Wo, k, stride);
    return sizeof(float) * kF32KC * (2 * (pt + 4) + 3 * (dt + 4) + 2 * f32_filt_pitch(k * k) + 2 * kL) + kL * sizeof(long long);
}

template <int PT, int DT, int TP, int TD, int KS, int NP, int K, bool NHWC>
gdws_status_t f32_launch(const F32Shape &s, const gdws_plan_s *p, const float *x, const float *dw, const float *pw, const float *bias, float *y, cudaStream_t st)
{
    const size_t smem = f32_smem(PT, DT, s.Wo, s.k, s.stride);
    auto kernel = fused_f32_kernel<PT, DT, TP, TD, KS, NP, K, NHWC>;
    static bool attr_set[64] = {};
    if (!attr_set[p->device & 63]) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(fused_f32_kernel)");
        attr_set[p->device & 63] = true;
    }
    const long long npix = (long long)s.N * s.Ho * s.Wo;
    const cudaError_t e = launch_overlapped(kernel, dim3((unsigned)((npix + PT - 1) / PT), (unsigned)((s.D + DT - 1) / DT)),
                                            (unsigned)((PT / TP) * (DT / TD) * KS + NP), smem, st, s, x, dw, pw, bias, (const int32_t *)p->d_chan, y);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "fused_f32_kernel launch"); }
    return GDWS_OK;
}

template <int PT, int DT, int TP, int TD, int KS, int NP, class... A>
gdws_status_t f32_launch_for(bool nhwc, const F32Shape &s, A... a)
{
    if (nhwc) {
        switch (s.k) {
        case 1: return f32_launch<PT, DT, TP, TD, KS, NP, 1, true>(s, a...);
        case 3: return f32_launch<PT, DT, TP, TD, KS, NP, 3, true>(s, a...);
        case 5: return f32_launch<PT, DT, TP, TD, KS, NP, 5, true>(s, a...);
        default: return f32_launch<PT, DT, TP, TD, KS, NP, 0, true>(s, a...);
        }
    }
    switch (s.k) {
    case 1: return f32_launch<PT, DT, TP, TD, KS, NP, 1, false>(s, a...);
    case 3: return f32_launch<PT, DT, TP, TD, KS, NP, 3, false>(s, a...);
    case 5: return f32_launch<PT, DT, TP, TD, KS, NP, 5, false>(s, a...);
    default: return f32_launch<PT, DT, TP, TD, KS, NP, 0, false>(s, a...);
    }
}

// Block tiles of fused_f32_kernel and the share of the multiply-add rate that a busy SM reaches with each: measured in NCHW before
// the z phase got its present form, which made the wide tiles some 8 % faster and left their order as it was.
struct F32Config { int pt, dt; double rate; };
constexpr F32Config kF32Configs[] = {
    {8, 16, 0.025}, {16, 32, 0.08}, {32, 32, 0.11}, {32, 64, 0.19}, {32, 128, 0.24}, {64, 128, 0.24}, {96, 128, 0.34}, {128, 128, 0.36},
};

// The tile whose busiest SM is done first: large tiles reuse more per load, small ones leave no SM idle.
int f32_config(const gdws_plan_s *p, long long npix, int Wo, double *cycles = nullptr)
{
    const int sms = sm_count_of(p);
    int best = 0;
    double best_cost = 1e300;
    for (int c = 0; c < (int)(sizeof(kF32Configs) / sizeof(kF32Configs[0])); ++c) {
        const F32Config &f = kF32Configs[c];
        const long long blocks = ((npix + f.pt - 1) / f.pt) * ((p->D + f.dt - 1) / f.dt);
        if ((npix + f.pt - 1) / f.pt > 0x7fffffffLL || (p->D + f.dt - 1) / f.dt > 65535) continue;
        if (f32_smem(f.pt, f.dt, Wo, p->k, p->stride) > (size_t)kMaxSmem) continue;      // long rows of large filters: narrower tiles
        const double per_block = (double)p->G * f.pt * (f.dt + 1.5 * p->k * p->k) / 128.0;        // cycles at the full rate
        const long long per_sm = (blocks + sms - 1) / sms;
        // a block alone on its SM waits for its own loads: 2500 cycles a chunk of the small tiles,
        // 4000 of the widest
        const double alone = p->G / (double)kF32KC * (2200.0 + 0.12 * f.pt * f.dt) + 3000.0;
        const double cost = std::max(per_sm * per_block / f.rate, std::max(alone, per_block / (0.8 * f.rate)));
        if (cost < best_cost) { best_cost = cost; best = c; }
    }
    if (cycles) *cycles = best_cost;
    return best_cost < 1e300 ? best : -1;
}

}  // namespace

int f32_alu_config(const gdws_plan_s *p, long long npix, int Wo) { return f32_config(p, npix, Wo); }

// Estimate of fused_f32_kernel's time for n images.
double f32_alu_us(const gdws_plan_s *p, int n, int h, int w)
{
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    double cycles = 0;
    f32_config(p, (long long)n * Ho * Wo, Wo, &cycles);
    return 3.0 + cycles / 1850.0;
}

gdws_status_t f32_fused(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, const float *pw_w,
                        const float *bias, gdws_tensor_t *y, cudaStream_t st)
{
    int config = -2;
    // a launch that is refused leaves the layer to the kernel below, which covers it as well
    if (f32_tc_takes(p, x->n, x->h, x->w, &config) && f32_fused_tc(p, x, dw_w, pw_w, bias, y, st) == GDWS_OK) return GDWS_OK;
    const F32Shape s = make_shape(p, x->layout, x->n, x->h, x->w);
    const bool nhwc = x->layout == GDWS_NHWC;
    const float *xp = (const float *)x->ptr;
    float *yp = (float *)y->ptr;
    gdws_status_t rc = GDWS_ERR_UNSUPPORTED;
    const gdws_plan_s *cp = p;
    switch (config == -2 ? f32_config(p, (long long)s.N * s.Ho * s.Wo, s.Wo) : config) {
    case 0: rc = f32_launch_for<8, 16, 1, 1, 1, 128>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 1: rc = f32_launch_for<16, 32, 2, 2, 1, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 2: rc = f32_launch_for<32, 32, 4, 2, 1, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 3: rc = f32_launch_for<32, 64, 4, 4, 1, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 4: rc = f32_launch_for<32, 128, 4, 8, 2, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 5: rc = f32_launch_for<64, 128, 8, 8, 1, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 6: rc = f32_launch_for<96, 128, 8, 8, 2, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    case 7: rc = f32_launch_for<128, 128, 8, 8, 1, 256>(nhwc, s, cp, xp, dw_w, pw_w, bias, yp, st); break;
    default: return fail(GDWS_ERR_UNSUPPORTED, "too many pixels for the fp32 fused kernel");
    }
    if (rc == GDWS_OK) p->launches++;
    return rc;
}

}  // namespace gdws
