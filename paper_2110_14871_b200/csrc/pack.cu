// Weight packing for the bf16 kernels: every form a kernel may read is written by ONE launch, so that a forward that is
// given its weights costs two launches.  (Six small launches before: 3 us each on the GPU, most of a small layer's time.)
// Blocks take pieces of the outputs, in the order of PackParams::first.
#include <algorithm>

#include "sm100.cuh"

namespace gdws {

constexpr int kPackThreads = 256, kPackPiece = 2048;     // elements of a block where the output is a flat array
constexpr int kFoldPackPer = 1, kFoldPackD = 4 * kFoldPackPer, kFoldPackTaps = 9;
enum { kPackImg, kPackTaps, kPackBias, kPackFilt, kPackSlab, kPackFold, kPackParts };

struct PackParams {
    const void *dw, *pw;
    const float *bias;
    int is_bf16;
    int first[kPackParts + 1];       // first block of each output
    int C, D, G, k2, Dpad, Gpad, nchunks, wstride;
    const int32_t *off, *chan, *chunk_meta;
    uint16_t *pw_img;
    float *taps;
    uint32_t *dwpack;
    float *bias_out;
    const TcChunk *tc_chunks;
    int tc_nchunks, tc_nslabs, tc_dloc, tc_nparts, rec_hw;
    uint16_t *tc_filt, *tc_pw;
    int fold_dblocks, fold_dp;
    uint16_t *fold;
};

__device__ __forceinline__ float load_weight(const void *w, size_t idx, int is_bf16)
{
    return is_bf16 ? bf16_bits_to_float(((const uint16_t *)w)[idx]) : ((const float *)w)[idx];
}

// pw_w[D][G] -> one operand image per 64-wide K chunk: rows d (zero rows up to Dpad), 64 bf16
// of K per 128-byte row, 128-byte swizzle; columns beyond G are zero.
__device__ void pack_img(const PackParams &P, int piece)
{
    const long long total = (long long)P.nchunks * P.Dpad * kChunk;
    for (int e = threadIdx.x; e < kPackPiece; e += kPackThreads) {
        const long long t = (long long)piece * kPackPiece + e;
        if (t >= total) return;
        const int kk = (int)(t % kChunk);
        const long long r = t / kChunk;
        const int d = (int)(r % P.Dpad), q = (int)(r / P.Dpad), i = q * kChunk + kk;
        float v = 0.f;
        if (d < P.D && i < P.G) v = load_weight(P.pw, (size_t)d * P.G + i, P.is_bf16);
        const uint32_t off = (uint32_t)(d >> 3) * 1024u + (uint32_t)(d & 7) * 128u + (uint32_t)(((kk >> 3) ^ (d & 7)) << 4) + (uint32_t)(kk & 7) * 2u;
        P.pw_img[(size_t)q * P.Dpad * kChunk + (off >> 1)] = float_to_bf16_bits(v);
    }
}

// dw_w[G][k][k] -> (1) fp32 taps [Gpad][k*k] (zero rows for the padding) for the unfused kernel,
// (2) [Gpad][wstride] words for the fused kernel: the taps, then the index of the channel inside the
// input box staged for its K chunk (chan[i] - first channel of that box).
__device__ void pack_taps(const PackParams &P, int piece)
{
    const int total = P.Gpad * P.wstride;
    for (int e = threadIdx.x; e < kPackPiece; e += kPackThreads) {
        const int t = piece * kPackPiece + e;
        if (t >= total) return;
        const int i = t / P.wstride, j = t - i * P.wstride;
        uint32_t word = 0;
        if (j < P.k2) {
            float v = 0.f;
            if (i < P.G) v = load_weight(P.dw, (size_t)i * P.k2 + j, P.is_bf16);
            v = bf16_bits_to_float(float_to_bf16_bits(v));
            P.taps[(size_t)i * P.k2 + j] = v;
            word = __float_as_uint(v);
        } else if (j == P.k2 && i < P.G) {
            word = (uint32_t)(P.chan[i] - P.chunk_meta[4 * (i / kChunk) + 2]);
        }
        P.dwpack[t] = word;
    }
}

// dw_w[G][k][k] -> one record per intermediate slot of the tensor-core GDW path: the slot's channel inside its 16-channel
// window (0xFFFF for the padding slots of a chunk), then the k*k taps as bf16.  One block per chunk.
__device__ void pack_filt(const PackParams &P, int chunk)
{
    const TcChunk ch = P.tc_chunks[chunk];
    for (int e = threadIdx.x; e < ch.npad * P.rec_hw; e += kPackThreads) {
        const int t = e / P.rec_hw, h = e - t * P.rec_hw;
        uint16_t val = 0;
        if (h == 0) val = t < ch.n ? (uint16_t)(P.chan[ch.i0 + t] - ch.cbase) : (uint16_t)0xFFFFu;
        else if (h <= P.k2 && t < ch.n) val = float_to_bf16_bits(load_weight(P.dw, (size_t)(ch.i0 + t) * P.k2 + (h - 1), P.is_bf16));
        P.tc_filt[((size_t)ch.slab0 * 16 + t) * P.rec_hw + h] = val;
    }
}

// pw_w[D][G] -> [part][slab][output channel][16] bf16: per 16 intermediate slots one K-major operand slab of the
// pointwise product, 32 bytes per output channel, 32-byte swizzle.  One block per slab and part.
__device__ void pack_slab(const PackParams &P, int idx)
{
    const int part = idx / P.tc_nslabs, slab = idx - part * P.tc_nslabs;
    int lo = 0, hi = P.tc_nchunks - 1;           // the chunk whose slabs these are
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (P.tc_chunks[mid].slab0 <= slab) lo = mid; else hi = mid - 1;
    }
    const TcChunk ch = P.tc_chunks[lo];
    const int t0 = (slab - ch.slab0) * 16, per_slab = 16 * P.tc_dloc;
    uint16_t *out = P.tc_pw + (size_t)idx * per_slab;
    for (int e = threadIdx.x; e < per_slab; e += kPackThreads) {
        const int dl = e >> 4, kk = e & 15, t = t0 + kk, d = part * P.tc_dloc + dl;
        float val = 0.f;
        if (t < ch.n && d < P.D) val = load_weight(P.pw, (size_t)d * P.G + ch.i0 + t, P.is_bf16);
        // row dl of the slab: 32 bytes, its two 16-byte halves swapped in rows 4..7 of every 8 (32-byte swizzle)
        out[dl * 16 + ((((kk >> 3) ^ ((dl >> 2) & 1))) << 3) + (kk & 7)] = float_to_bf16_bits(val);
    }
}

// Rounds a filter's taps to bf16, each to one of its two neighbours, so that the taps' sum keeps its value as far as the taps
// with a fraction of at least kFlip of their spacing allow.  Activations have a mean: rounding every tap to its nearest
// neighbour alone lets the errors of a filter add up on it.  (Relative error of y before its own rounding, 64 -> 64 channels:
// inputs with a large mean 1.5e-3 -> 4e-4, half-rectified 1.64e-3 -> 1.5e-3, without a mean 1.66e-3 -> 1.8e-3.)
constexpr float kFlip = 0.25f;
template <int T> __device__ __forceinline__ void round_taps(float (&v)[T])
{
    float q[T], sum = 0.f;
#pragma unroll
    for (int t = 0; t < T; ++t) {
        q[t] = bf16_bits_to_float(float_to_bf16_bits(v[t]));
        sum += v[t] - q[t];
    }
#pragma unroll 1
    for (int it = 0; it < 3; ++it) {
        float best = fabsf(sum), step = 0.f;
        int which = -1;
#pragma unroll
        for (int t = 0; t < T; ++t) {
            const float e = v[t] - q[t];
            const float u = __uint_as_float(__float_as_uint(v[t]) & 0x7F800000u) * 0.0078125f;     // spacing of bf16 values around v
            const float left = fabsf(sum - copysignf(u, e));
            if (e * sum > 0.f && fabsf(e) >= kFlip * u && left < best) { best = left; which = t; step = copysignf(u, e); }
        }
        if (which < 0) break;
        sum -= step;
#pragma unroll
        for (int t = 0; t < T; ++t)
            if (t == which) q[t] += step;
    }
#pragma unroll
    for (int t = 0; t < T; ++t) v[t] = q[t];
}

// Folded filters: W[d,c,tap] = sum_j P[d, off_c+j] K[off_c+j, tap] in fp32, rounded to bf16 once (round_taps).  Rows are (window of 64
// input channels, tap, output channel), 64 input channels each; rows d >= D and channels >= C are zero.  A block takes one
// window and 4 output channels: thread = one channel x one output channel, up to 9 taps at a time in registers.  (Four
// output channels per thread read a tap once for all four, but left a 72 -> 120 layer 16 blocks: 5 us slower.)
__device__ void pack_fold(const PackParams &P, int idx)
{
    const int win = idx / P.fold_dblocks, cl = threadIdx.x & 63, c = win * 64 + cl;
    const int d0 = (idx - win * P.fold_dblocks) * kFoldPackD + (threadIdx.x >> 6) * kFoldPackPer;
    const int i0 = c < P.C ? P.off[c] : 0, i1 = c < P.C ? P.off[c + 1] : 0;
    auto weight = [&](const void *w, size_t i) {          // the two-stage kernels use the weights rounded to bf16 as well
        return P.is_bf16 ? bf16_bits_to_float(((const uint16_t *)w)[i]) : bf16_bits_to_float(float_to_bf16_bits(((const float *)w)[i]));
    };
    for (int t0 = 0; t0 < P.k2; t0 += kFoldPackTaps) {
        float acc[kFoldPackPer][kFoldPackTaps] = {};
#pragma unroll 4
        for (int i = i0; i < i1; ++i) {
            float p[kFoldPackPer];
#pragma unroll
            for (int e = 0; e < kFoldPackPer; ++e) p[e] = d0 + e < P.D ? weight(P.pw, (size_t)(d0 + e) * P.G + i) : 0.f;
#pragma unroll
            for (int t = 0; t < kFoldPackTaps; ++t) {
                const float v = t0 + t < P.k2 ? weight(P.dw, (size_t)i * P.k2 + t0 + t) : 0.f;
#pragma unroll
                for (int e = 0; e < kFoldPackPer; ++e) acc[e][t] = fmaf(p[e], v, acc[e][t]);
            }
        }
#pragma unroll
        for (int e = 0; e < kFoldPackPer; ++e) round_taps(acc[e]);      // taps beyond the filter are zeros and stay so
#pragma unroll
        for (int t = 0; t < kFoldPackTaps; ++t)
            if (t0 + t < P.k2)
#pragma unroll
                for (int e = 0; e < kFoldPackPer; ++e)
                    if (d0 + e < P.fold_dp) P.fold[(((size_t)win * P.k2 + t0 + t) * P.fold_dp + d0 + e) * 64 + cl] = float_to_bf16_bits(acc[e][t]);
    }
}

__global__ void __launch_bounds__(kPackThreads) pack_kernel(const __grid_constant__ PackParams P)
{
    grid_launch_dependents();
    grid_dependency_wait();      // the kernel before may still read what this one overwrites
    const int b = (int)blockIdx.x;
    if (b >= P.first[kPackFold]) pack_fold(P, b - P.first[kPackFold]);
    else if (b >= P.first[kPackSlab]) pack_slab(P, b - P.first[kPackSlab]);
    else if (b >= P.first[kPackFilt]) pack_filt(P, b - P.first[kPackFilt]);
    else if (b >= P.first[kPackBias]) {
        const int t = (b - P.first[kPackBias]) * kPackThreads + (int)threadIdx.x;
        if (t < P.Dpad) P.bias_out[t] = (P.bias && t < P.D) ? P.bias[t] : 0.f;
    }
    else if (b >= P.first[kPackTaps]) pack_taps(P, b - P.first[kPackTaps]);
    else pack_img(P, b);
}

gdws_status_t bf16_pack(gdws_plan_s *p, const void *dw_w, const void *pw_w, const float *bias, gdws_dtype_t dtype, cudaStream_t st)
{
    PackParams P;
    P.dw = dw_w; P.pw = pw_w; P.bias = bias; P.is_bf16 = dtype == GDWS_BF16;
    P.C = p->C; P.D = p->D; P.G = p->G; P.k2 = p->k * p->k; P.Dpad = p->Dpad; P.Gpad = p->Gpad; P.nchunks = p->nchunks; P.wstride = p->wstride;
    P.off = p->d_off; P.chan = p->d_chan; P.chunk_meta = p->d_chunk_meta;
    P.pw_img = p->d_pw_img; P.taps = p->d_dw; P.dwpack = p->d_dwpack; P.bias_out = p->d_bias;
    P.tc_chunks = p->d_tc_chunks; P.tc_nchunks = (int)p->tc_chunks.size(); P.tc_nslabs = p->tc_nslabs; P.tc_dloc = p->tc_dloc;
    P.tc_nparts = p->tc_nparts; P.rec_hw = p->tc_rec_hw; P.tc_filt = p->d_tc_filt; P.tc_pw = p->d_tc_pw;
    P.fold_dblocks = (p->fold_dp + kFoldPackD - 1) / kFoldPackD; P.fold_dp = p->fold_dp; P.fold = p->d_fold;
    const long long blocks[kPackParts] = {
        ((long long)p->nchunks * p->Dpad * kChunk + kPackPiece - 1) / kPackPiece,
        (p->Gpad * (long long)p->wstride + kPackPiece - 1) / kPackPiece,
        (p->Dpad + kPackThreads - 1) / kPackThreads,
        p->tc_ok ? (long long)p->tc_chunks.size() : 0,
        p->tc_ok ? (long long)p->tc_nslabs * p->tc_nparts : 0,
        p->fold_ok ? (long long)p->fold_nwin * P.fold_dblocks : 0,
    };
    long long total = 0;
    for (int i = 0; i < kPackParts; ++i) {
        P.first[i] = (int)total;
        total += blocks[i];
        if (total > 0x7fffffffLL) return fail(GDWS_ERR_UNSUPPORTED, "weights too large to pack");
    }
    P.first[kPackParts] = (int)total;
    const cudaError_t e = launch_overlapped(pack_kernel, (unsigned)total, kPackThreads, 0, st, P);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "weight pack launch"); }
    p->launches++;
    p->packed = true;
    return GDWS_OK;
}

}  // namespace gdws
