// Weight packing for the bf16 kernels: every form a kernel may read is written by ONE launch, so that a forward that is
// given its weights costs two launches.  (Six small launches before: 3 us each on the GPU, most of a small layer's time.)
// Blocks take pieces of the outputs, in the order of PackParams::first.
#include <algorithm>

#include "sm100.cuh"

namespace gdws {

constexpr int kPackThreads = 256, kPackPiece = 2048;     // elements of a block where the output is a flat array
constexpr int kFoldPackStage = 12288;     // bf16 values of filters and weights that a block holds at a time
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
    int fold_dblocks, fold_dp, fold_blocks, fold_sum_step;
    uint16_t *fold;
    float2 *fold_sums;
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

// Folded filters: W[d,c,tap] = sum_j P[d, off_c+j] K[off_c+j, tap] in fp32, as two bf16 terms: W rounded to nearest, and what
// that leaves over rounded to nearest.  Rows are (term, window of 64 input channels, tap, output channel), 64 input channels
// each; rows d >= D and channels >= C are zero.  A block takes one window and 4 PER output channels: thread = one channel x PER
// output channels.  PER = 1 where blocks are few (four output channels per thread left a 72 -> 120 layer 16 blocks: 5 us slower), 4
// where the loads of the taps, which lie far apart for neighbouring channels, take the time (kFoldPackWide).
// Beside them, per block (or every n-th): the sum of the squared taps and of the filters' squared tap sums, from which the
// forward decides whether it takes the second term.

// A weight rounded to bf16: the two-stage kernels use them so as well.
__device__ __forceinline__ float fold_weight(const PackParams &P, const void *w, size_t i)
{
    return P.is_bf16 ? bf16_bits_to_float(((const uint16_t *)w)[i]) : bf16_bits_to_float(float_to_bf16_bits(((const float *)w)[i]));
}

// One tap of a thread's channel and PER output channels.
template <int PER> __device__ __forceinline__ void pack_fold_store(const PackParams &P, int win, int cl, int t, int d0, size_t term, const float (&w)[PER], float &energy, float (&sum)[PER])
{
#pragma unroll
    for (int e = 0; e < PER; ++e) {
        uint16_t *out = P.fold + (((size_t)win * P.k2 + t) * P.fold_dp + d0 + e) * 64 + cl;
        const uint16_t hi = float_to_bf16_bits(w[e]);
        out[0] = hi;
        out[term] = float_to_bf16_bits(w[e] - bf16_bits_to_float(hi));
        energy = fmaf(w[e], w[e], energy);
        sum[e] += w[e];
    }
}

template <int PER> __device__ __forceinline__ void pack_fold_sums(const PackParams &P, int win, int group, float energy, const float (&sum)[PER])
{
    if (group % P.fold_sum_step) return;
    __shared__ float2 part[kPackThreads / 32];
    float2 v = make_float2(energy, 0.f);
#pragma unroll
    for (int e = 0; e < PER; ++e) v.y = fmaf(sum[e], sum[e], v.y);
#pragma unroll
    for (int o = 16; o; o >>= 1) { v.x += __shfl_xor_sync(0xffffffffu, v.x, o); v.y += __shfl_xor_sync(0xffffffffu, v.y, o); }
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        v = part[0];
#pragma unroll
        for (int w = 1; w < kPackThreads / 32; ++w) { v.x += part[w].x; v.y += part[w].y; }
        P.fold_sums[win * ((P.fold_dblocks + P.fold_sum_step - 1) / P.fold_sum_step) + group / P.fold_sum_step] = v;
    }
}

// PER = 4: up to 9 taps of a filter in registers, their loads in flight together.  (Through shared memory as below: 6.3 -> 8.5 us for 352 ->
// 336 channels.)
__device__ __forceinline__ void pack_fold_wide(const PackParams &P, int idx)
{
    constexpr int PER = 4, TAPS = 9;
    const int win = idx / P.fold_dblocks, group = idx - win * P.fold_dblocks, cl = threadIdx.x & 63, c = win * 64 + cl;
    const int d0 = (group * 4 + (threadIdx.x >> 6)) * PER;
    const int i0 = c < P.C ? P.off[c] : 0, i1 = c < P.C && d0 < P.D ? P.off[c + 1] : i0;
    const size_t term = (size_t)P.fold_dp * (P.fold_blocks / P.fold_dblocks) * P.k2 * 64;
    float energy = 0.f, sum[PER] = {};
    for (int t0 = 0; t0 < P.k2; t0 += TAPS) {
        float acc[TAPS][PER] = {};
#pragma unroll 1
        for (int i = i0; i < i1; ++i) {
            float p[PER], v[TAPS];
#pragma unroll
            for (int e = 0; e < PER; ++e) p[e] = d0 + e < P.D ? fold_weight(P, P.pw, (size_t)(d0 + e) * P.G + i) : 0.f;
#pragma unroll
            for (int t = 0; t < TAPS; ++t) v[t] = t0 + t < P.k2 ? fold_weight(P, P.dw, (size_t)i * P.k2 + t0 + t) : 0.f;
#pragma unroll
            for (int e = 0; e < PER; ++e)
#pragma unroll
                for (int t = 0; t < TAPS; ++t) acc[t][e] = fmaf(p[e], v[t], acc[t][e]);
        }
#pragma unroll
        for (int t = 0; t < TAPS; ++t)
            if (t0 + t < P.k2) pack_fold_store<PER>(P, win, cl, t0 + t, d0, term, acc[t], energy, sum);
    }
    pack_fold_sums<PER>(P, win, group, energy, sum);
}

// PER = 1.  A window's filters lie in a row: the block fetches them and their weights to shared memory in wide loads, all in flight
// together, as many filters at a time as fit.  (Each thread fetching its own, 9 taps of 5 filters at a time, left a call that is given
// its weights waiting for load after load: packing alone 80 -> 176 channels,
// 5 x 5 taps 11.6 -> 6.6 us.)
template <int TAPS> __device__ __forceinline__ void pack_fold(const PackParams &P, int idx)
{
    extern __shared__ __align__(16) uint16_t stage[];        // kFoldPackStage
    constexpr int ROWS = 4;
    const int win = idx / P.fold_dblocks, group = idx - win * P.fold_dblocks, cl = threadIdx.x & 63, c = win * 64 + cl;
    const int row = threadIdx.x >> 6, r0 = group * ROWS, d0 = r0 + row;
    const int i0 = c < P.C ? P.off[c] : 0, i1 = c < P.C && d0 < P.D ? P.off[c + 1] : i0;
    const int f0 = P.off[win * 64], f1 = P.off[min(P.C, win * 64 + 64)];        // the window's filters
    const int most = (kFoldPackStage - 32) / (P.k2 + ROWS);
    uint16_t *const pws = stage + (most * P.k2 + 23) / 8 * 8;
    float acc[TAPS][1] = {};
#pragma unroll 1
    for (int f = f0; f < f1; f += most) {
        const int n = min(most, f1 - f);
        const size_t e0 = (size_t)f * P.k2 & ~(size_t)7, e1 = (size_t)(f + n) * P.k2, all = (size_t)P.G * P.k2;
        if (f > f0) __syncthreads();             // what was there has been read
#pragma unroll 4
        for (size_t e = e0 + 8 * threadIdx.x; e < e1; e += 8 * kPackThreads) {
            uint4 v;
            if (P.is_bf16 && e + 8 <= all) {
                v = *reinterpret_cast<const uint4 *>((const uint16_t *)P.dw + e);
            } else {
                uint32_t h[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) h[j] = e + j < all ? float_to_bf16_bits(fold_weight(P, P.dw, e + j)) : 0u;
                v = make_uint4(h[0] | h[1] << 16, h[2] | h[3] << 16, h[4] | h[5] << 16, h[6] | h[7] << 16);
            }
            *reinterpret_cast<uint4 *>(stage + (e - e0)) = v;
        }
#pragma unroll 2
        for (int i = threadIdx.x; i < n; i += kPackThreads) {
            uint16_t v[ROWS];
#pragma unroll
            for (int r = 0; r < ROWS; ++r) v[r] = r0 + r < P.D ? float_to_bf16_bits(fold_weight(P, P.pw, (size_t)(r0 + r) * P.G + f + i)) : 0;
#pragma unroll
            for (int r = 0; r < ROWS; ++r) pws[r * most + i] = v[r];
        }
        __syncthreads();
        const uint16_t *const taps = stage + ((size_t)f * P.k2 - e0);
#pragma unroll 1
        for (int i = max(i0, f); i < min(i1, f + n); ++i) {
            const float p = bf16_bits_to_float(pws[row * most + i - f]);
#pragma unroll
            for (int t = 0; t < TAPS; ++t)
                if (t < P.k2) acc[t][0] = fmaf(p, bf16_bits_to_float(taps[(i - f) * P.k2 + t]), acc[t][0]);
        }
    }
    const size_t term = (size_t)P.fold_dp * (P.fold_blocks / P.fold_dblocks) * P.k2 * 64;
    float energy = 0.f, sum[1] = {};
#pragma unroll
    for (int t = 0; t < TAPS; ++t)
        if (t < P.k2) pack_fold_store<1>(P, win, cl, t, d0, term, acc[t], energy, sum);
    pack_fold_sums<1>(P, win, group, energy, sum);
}

// One kernel per way to fold: with the code of all of them in one, calls that fold nothing took up to 0.8 us longer.
enum { kFoldNot, kFoldWide, kFoldNine, kFoldMore };
template <int FOLD> __global__ void __launch_bounds__(kPackThreads, 3) pack_kernel(const __grid_constant__ PackParams P)
{
    grid_launch_dependents();
    grid_dependency_wait();      // the kernel before may still read what this one overwrites
    const int b = (int)blockIdx.x;
    if (FOLD != kFoldNot && b >= P.first[kPackFold]) {
        const int idx = b - P.first[kPackFold];
        if constexpr (FOLD == kFoldWide) pack_fold_wide(P, idx);
        else pack_fold<FOLD == kFoldNine ? 9 : 25>(P, idx);
    }
    else if (b >= P.first[kPackSlab]) pack_slab(P, b - P.first[kPackSlab]);
    else if (b >= P.first[kPackFilt]) pack_filt(P, b - P.first[kPackFilt]);
    else if (b >= P.first[kPackBias]) {
        const int t = (b - P.first[kPackBias]) * kPackThreads + (int)threadIdx.x;
        if (t < P.Dpad) P.bias_out[t] = (P.bias && t < P.D) ? P.bias[t] : 0.f;
    }
    else if (b >= P.first[kPackTaps]) pack_taps(P, b - P.first[kPackTaps]);
    else pack_img(P, b);
}

gdws_status_t bf16_pack(gdws_plan_s *p, const void *dw_w, const void *pw_w, const float *bias, gdws_dtype_t dtype, bool fold, cudaStream_t st)
{
    fold = p->fold_ok && (fold || p->opt_dw_math == 3 || p->Dpad > 512);      // beyond 512 output channels the two stages may have no kernel
    PackParams P;
    P.dw = dw_w; P.pw = pw_w; P.bias = bias; P.is_bf16 = dtype == GDWS_BF16;
    P.C = p->C; P.D = p->D; P.G = p->G; P.k2 = p->k * p->k; P.Dpad = p->Dpad; P.Gpad = p->Gpad; P.nchunks = p->nchunks; P.wstride = p->wstride;
    P.off = p->d_off; P.chan = p->d_chan; P.chunk_meta = p->d_chunk_meta;
    P.pw_img = p->d_pw_img; P.taps = p->d_dw; P.dwpack = p->d_dwpack; P.bias_out = p->d_bias;
    P.tc_chunks = p->d_tc_chunks; P.tc_nchunks = (int)p->tc_chunks.size(); P.tc_nslabs = p->tc_nslabs; P.tc_dloc = p->tc_dloc;
    P.tc_nparts = p->tc_nparts; P.rec_hw = p->tc_rec_hw; P.tc_filt = p->d_tc_filt; P.tc_pw = p->d_tc_pw;
    P.fold_dblocks = p->fold_dp / (4 * p->fold_per); P.fold_dp = p->fold_dp; P.fold_blocks = p->fold_blocks; P.fold = p->d_fold;
    P.fold_sum_step = p->fold_sum_step; P.fold_sums = p->d_fold_sums;
    const long long blocks[kPackParts] = {
        ((long long)p->nchunks * p->Dpad * kChunk + kPackPiece - 1) / kPackPiece,
        (p->Gpad * (long long)p->wstride + kPackPiece - 1) / kPackPiece,
        (p->Dpad + kPackThreads - 1) / kPackThreads,
        p->tc_ok ? (long long)p->tc_chunks.size() : 0,
        p->tc_ok ? (long long)p->tc_nslabs * p->tc_nparts : 0,
        fold ? (long long)p->fold_blocks : 0,
    };
    long long total = 0;
    for (int i = 0; i < kPackParts; ++i) {
        P.first[i] = (int)total;
        total += blocks[i];
        if (total > 0x7fffffffLL) return fail(GDWS_ERR_UNSUPPORTED, "weights too large to pack");
    }
    P.first[kPackParts] = (int)total;
    const bool staged = fold && p->fold_per == 1;
    const auto kernel = !fold ? pack_kernel<kFoldNot> : (!staged ? pack_kernel<kFoldWide> : (P.k2 <= 9 ? pack_kernel<kFoldNine> : pack_kernel<kFoldMore>));
    const cudaError_t e = launch_overlapped(kernel, (unsigned)total, kPackThreads, staged ? kFoldPackStage * sizeof(uint16_t) : 0, st, P);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "weight pack launch"); }
    p->launches++;
    p->packed = true;
    p->fold_packed = fold;
    return GDWS_OK;
}

}  // namespace gdws
