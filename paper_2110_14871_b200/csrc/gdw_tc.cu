// The GDW stage on its own, on the tensor cores: z[pixel][Gpad] in bf16, NHWC, filters up to 5 x 5, strides 1 and 2.
//
// z = K x is itself a k x k convolution, from C to G channels, whose filters are zero but for one input channel each.  64
// neighbouring intermediate channels read few neighbouring input channels (Property 2 keeps them in order; 24 at a mean multiplier of
// 2.7), so a product of 16 input channels per K step wastes little: per tap and 16 channels one product of M = 256 (a pair of blocks,
// 128 pixels each) and N = 64.  The tensor cores take some 44 cycles for it; 128 pixels x 64 channels on the ALUs cost an SM 1100
// cycles of multiply-adds and loads (2900 in the kernel that does so), here 64 channels at a mean multiplier of 2.7 some 500.
//
// Measured, ALUs | here: 64 -> 191 channels at 64 x 56 x 56 47.6 | 40.3 us, 424 -> 1181 at 38 x 19 x 25, stride 2 57.7 | 21.2, 512 -> 1415
// at 9 x 9 x 9 35.6 | 10.2, 176 -> 2203 at 28 x 28 x 28, 5 x 5 taps 146 | 80.5; nothing in it, 6.7 us against 4.5.
// What bounds it: an item (a pair of tiles x 64 channels) takes some 1.05 us, of which its 18 products at a mean multiplier of 2.7 are
// 0.4; without its stores the first layer takes 33 us, without its products 38.  The layout that follows:
//   * A operand: the input box of a tile, all taps from one box, as in the folded kernel (csrc/fold.cu); 16, 32 or 64
//     channels wide, whatever the widest run of 64 intermediate channels reads (2, 4 or 8 pieces of 16 bytes per pixel, swizzled alike).
//   * B operand: built by four warps from the packed taps, zeros elsewhere.  All of a layer's stay in shared memory where they fit
//     (then items of one tile follow one another and share its box where their channels lie in one); otherwise a block walks through the tiles of one run of 64 channels before the next.
//   * Epilogue: four groups of four warps, an item each; staged and stored by TMA.
// A product of zero and an infinity is NaN, and a filter of zeros meets the neighbours' inputs: a z that is not finite is computed
// again from its own channel.
#include <float.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <new>

#include "sm100.cuh"

namespace gdws {

constexpr int kGdwThreads = 24 * 32, kGdwMmaWarp = 0, kGdwAWarp = 1, kGdwTmemWarp = 2, kGdwBuildWarp = 4, kGdwEpiWarp = 8;
constexpr int kGdwMaxA = 6, kGdwMaxB = 16, kGdwAcc = 8, kGdwGroups = 4, kGdwMaxSteps = 25, kGdwMaxChunks = 1024;

// What a run of 64 channels reads: bits 0-3 its first K step (16 channels) in its box, 4-8 its K steps, 16-31 the box's first channel;
// runs that share a box: whether it is the first / last of them.
constexpr uint32_t kGdwFirst = 1u << 10, kGdwLast = 1u << 11;

struct alignas(64) GdwParams {
    CUtensorMap tmap_x[4];       // x as (C, W, H, N), box (row bytes / 2, IW, rows, TN); stride 2: one dense view per parity
    CUtensorMap tmap_z;          // z as (Gpad, Wo, Ho, N), box (64, PW, PH, TN)
    const uint16_t *x;
    const float *taps;           // [Gpad][k*k]
    const int32_t *chan;
    int *status;
    int k2, nboxes, nchunks, G;
    uint32_t steps[kGdwMaxSteps];        // A offset / 16 within the box, tap << 16
    uint32_t boxes[kGdwMaxSteps];        // first load, loads << 8, first step << 16, steps << 24
    int load_map[kGdwMaxSteps], load_dw[kGdwMaxSteps], load_dh[kGdwMaxSteps];
    int N, C, H, W, k, stride, pad, Ho, Wo;
    int TN, PH, PW, tiles_h, tiles_w, pairs, nitems;
    int rb, maps_used, na, nb, resident, groups;      // rb: bytes of a staged pixel (32, 64, 128)
    uint32_t dv_run[2], dv_thw[2], dv_tw[2];      // divisions by the runs (resident) or the pairs, by tiles of an image, of a row
    uint32_t swizzle, a_sbo, a_bytes, a_load, a_slot, b_tap, b_buf;
    uint32_t off_a, off_b, off_chunk;
    uint32_t info[kGdwMaxB];     // resident: the runs
};

__device__ __forceinline__ void gdw_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (!mbar_try_wait(bar, parity)) mbar_wait_relaxed_slow(bar, parity, 16384u, abort_flag, status, code);
}
// The leader waits for arrivals from both blocks: acquire at cluster scope.  Bounded like the others.
static __device__ __noinline__ void gdw_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    for (uint32_t it = 0; it < kSpinLimit && !*abort_flag; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
        if (ok) return;
        if (it > 4096) __nanosleep(64);
    }
    if (*abort_flag) return;
    *abort_flag = 1;
    atomicOr(status, code);
}

// The values of a warp's 32 pixels that are not finite, once more on the ALUs (0 for the padding channels): odd has a bit for each of
// its pixel's 64 channels.  A lane takes a channel, pixel by pixel: neighbouring channels read the same or neighbouring inputs, and a
// window's loads are in flight together.  (With a pixel per lane and a load at a time 64 x 64 x 56 x 56 infinities took 3580 us;
// here 624, ordinary values 40.)
template <int KM>              // filters up to KM x KM
static __device__ __noinline__ void gdw_plain(const GdwParams *params, uint32_t rows_s, int r0, int n0, int h0, int w0, int i0, uint32_t odd0, uint32_t odd1)
{
    const GdwParams &P = *params;
    const int lane = threadIdx.x & 31, ppi = P.PH * P.PW;
    const long long row = (long long)P.W * P.C;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const uint32_t odd = h ? odd1 : odd0;
        const int j = h * 32 + lane, c = P.chan[i0 + j];
        const uint16_t *const at = P.x + (c < 0 ? 0 : c);
        float tap[KM * KM];
#pragma unroll
        for (int t = 0; t < KM * KM; ++t) tap[t] = c >= 0 && t / KM < P.k && t % KM < P.k ? P.taps[(size_t)(i0 + j) * P.k2 + t / KM * P.k + t % KM] : 0.f;
#pragma unroll 1
        for (uint32_t todo = __ballot_sync(0xffffffffu, odd != 0); todo; todo &= todo - 1) {
            const int px = __ffs(todo) - 1, r = r0 + px, nl = r / ppi, ph = (r - nl * ppi) / P.PW, pw = r - nl * ppi - ph * P.PW;
            const uint32_t mask = __shfl_sync(0xffffffffu, odd, px);
            const int n = n0 + nl, ho = h0 + ph, wo = w0 + pw, hi = ho * P.stride - P.pad, wi = wo * P.stride - P.pad;
            if (n >= P.N || ho >= P.Ho || wo >= P.Wo || !((mask >> lane) & 1u)) continue;
            const uint16_t *x = at + (((long long)n * P.H + hi) * P.W + wi) * P.C;       // the window's first value, inside the image or not
            uint32_t v[KM * KM], cols = 0;       // bits as loaded: zeros outside
#pragma unroll
            for (int w = 0; w < KM; ++w) cols |= w < P.k && (unsigned)(wi + w) < (unsigned)P.W ? 1u << w : 0u;
#pragma unroll
            for (int u = 0; u < KM; ++u, x += row) {
                const bool in = u < P.k && (unsigned)(hi + u) < (unsigned)P.H;
#pragma unroll
                for (int w = 0; w < KM; ++w) v[KM * u + w] = in && ((cols >> w) & 1u) ? __ldg(x + w * P.C) : 0u;
            }
            float z = 0.f;
#pragma unroll
            for (int t = 0; t < KM * KM; ++t)
                if (t / KM < P.k && t % KM < P.k) z = fmaf(tap[t], __uint_as_float(v[t] << 16), z);
            sts16(rows_s + (uint32_t)r * 128u + (((uint32_t)(2 * j) & ~15u) ^ ((uint32_t)(r & 7) << 4)) + ((uint32_t)(2 * j) & 15u), float_to_bf16_bits(c < 0 ? 0.f : z));
        }
        __syncwarp();
    }
}

// The products of NS taps from s0 on, NK K steps each: straight-line code (a loop costs some 30 cycles per product).
template <int NS, int NK>
__device__ __forceinline__ void gdw_issue(const GdwParams &P, int s0, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi, uint32_t tap, uint32_t idesc, uint32_t more)
{
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        const uint32_t st = P.steps[s0 + s], al = a_lo + (st & 0xFFFFu), bl = b_lo + (st >> 16) * tap;
#pragma unroll
        for (int kk = 0; kk < NK; ++kk) umma_pair_words(d, al + 2u * kk, a_hi, bl + 2u * kk, b_hi, idesc, s | kk ? 1u : more);
    }
}

// NINE: 3 x 3 taps from one box per tile.  (As one kernel with the other shapes' code it took 42 us instead of 40 for 64 -> 191 channels.)
template <bool NINE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGdwThreads, 1) gdw_tc_kernel(const __grid_constant__ GdwParams P)
{
    extern __shared__ uint8_t smem_raw[];
    // afull[6] aempty[6] | bfull[16] bempty[16] | accfull[8] accfree[8] | drain
    constexpr int kBars = 2 * kGdwMaxA + 2 * kGdwMaxB + 2 * kGdwAcc + 1;
    __shared__ __align__(8) uint64_t bars[kBars];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    volatile int *const vabort = &abort_flag;
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t o_s = smem_u32(base), a_s = o_s + P.off_a, b_s = o_s + P.off_b;
    int *const chunks = reinterpret_cast<int *>(base + P.off_chunk);       // per run of 64 channels (kGdwFirst)
    const uint32_t bar_afull = smem_u32(&bars[0]), bar_aempty = bar_afull + 8 * kGdwMaxA, bar_bfull = bar_aempty + 8 * kGdwMaxA, bar_bempty = bar_bfull + 8 * kGdwMaxB;
    const uint32_t bar_accfull = bar_bempty + 8 * kGdwMaxB, bar_accfree = bar_accfull + 8 * kGdwAcc, bar_drain = bar_accfree + 8 * kGdwAcc;
    if (tid == 0) abort_flag = 0;
    // Full barriers and accfree are used in the leader only; the "empty" ones and accfull are completed in both blocks by its commits.
    if (tid < kBars) {
        const int b = tid - 2 * kGdwMaxA, acc = b - 2 * kGdwMaxB;
        const bool many = (b >= 0 && b < kGdwMaxB) || (acc >= kGdwAcc && acc < 2 * kGdwAcc);       // four warps of both blocks
        mbar_init(bar_afull + 8 * (uint32_t)tid, many ? 8u : 1u);
        fence_mbar_init();
    }
    grid_launch_dependents();
    if (warp == kGdwAWarp && lane == 0) {
#pragma unroll 1
        for (int l = 0; l < 4; ++l)
            if ((P.maps_used >> l) & 1) prefetch_tensor_map(&P.tmap_x[l]);
    }
    if (warp == kGdwTmemWarp) tmem_alloc_pair(smem_u32(&tmem_slot), 64u * kGdwAcc);
    for (int q = tid; q < P.nchunks; q += kGdwThreads) {         // written when the plan was made
        if (P.resident) {
            chunks[q] = (int)P.info[q];
        } else {
            const int c0 = __ldg(P.chan + q * kChunk) & ~7, last = __ldg(P.chan + min(q * kChunk + kChunk, P.G) - 1);
            chunks[q] = (int)((uint32_t)c0 << 16 | (uint32_t)((last + 1 - c0 + 15) >> 4) << 4 | kGdwFirst | kGdwLast);
        }
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    grid_dependency_wait();
    const uint32_t tmem = tmem_slot;
    const int cluster = (int)blockIdx.x >> 1, nclusters = (int)gridDim.x >> 1;
    const int i0 = (int)((long long)P.nitems * cluster / nclusters), i1 = (int)((long long)P.nitems * (cluster + 1) / nclusters);
    const int cb = P.rb >> 1;                    // channels of a box
    // Item -> run of 64 channels, this block's tile.
    auto run_of = [&](int it) { const int d = div_by(it, P.dv_run); return P.resident ? it - d * P.nchunks : d; };
    auto tile_of = [&](int it, int *n0, int *h0, int *w0) {
        const int d = div_by(it, P.dv_run);
        int tile = 2 * (P.resident ? d : it - d * P.pairs) + (int)rank;
        const int bn = div_by(tile, P.dv_thw);
        tile -= bn * P.tiles_h * P.tiles_w;
        const int bh = div_by(tile, P.dv_tw);
        *n0 = bn * P.TN; *h0 = bh * P.PH; *w0 = (tile - bh * P.tiles_w) * P.PW;
    };

    if (warp == kGdwMmaWarp) {
        if (rank == 0 && elect_one()) {
            // ---------------- products ----------------
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 17) | (16u << 24);   // fp32 += bf16 x bf16, M = 256, N = 64
            const uint32_t a_hi = ((P.a_sbo >> 4) & 0x3FFFu) | (1u << 14) | P.swizzle, b_hi = (((uint32_t)P.rb * 8u) >> 4) | (1u << 14) | P.swizzle;
            const uint32_t tap = P.b_tap >> 4;
            uint32_t slot = 0, par = 0, buf = 0, bpar = 0, known = 0;
            int have = -1;
#pragma unroll 1
            for (int n = 0; n < i1 - i0; ++n) {
                const int q = run_of(i0 + n), acc = n & (kGdwAcc - 1);
                bool fresh;                      // the run's filters have not been waited for
                if (P.resident) {
                    buf = (uint32_t)q;           // written once
                    fresh = !((known >> q) & 1u);
                    known |= 1u << q;
                } else {
                    fresh = q != have;
                    if (fresh && have >= 0) {    // the run before is over
                        umma_commit_pair(bar_bempty + 8 * buf);
                        if (++buf == (uint32_t)P.nb) { buf = 0; bpar ^= 1u; }
                    }
                    have = q;
                }
                if (fresh) gdw_wait_cluster(bar_bfull + 8 * buf, bpar, &abort_flag, P.status, kStatusWaitOperand);
                if (n >= kGdwAcc) gdw_wait_cluster(bar_accfree + 8 * acc, (uint32_t)((n >> 3) - 1) & 1u, &abort_flag, P.status, kStatusWaitStage);
                const uint32_t d = tmem + 64u * (uint32_t)acc, info = (uint32_t)chunks[q];
                uint32_t more = 0, b_lo = (((b_s + buf * P.b_buf) & 0x3FFFFu) >> 4) | (1u << 16);
                const uint32_t k0 = 2u * (info & 15u);       // first K step: 32 bytes each
                const bool take = (info & kGdwFirst) || n == 0, leave = (info & kGdwLast) || n == i1 - i0 - 1;
#pragma unroll 1
                for (int steps = (int)((info >> 4) & 31u); steps > 0; steps -= cb >> 4, b_lo += (uint32_t)P.k2 * tap) {
                    const int nk = min(steps, cb >> 4);
                    uint32_t at = slot, apar = par;      // boxes that several runs share: those of a tile stay until its last run has read them
#pragma unroll 1
                    for (int b = 0; b < (NINE ? 1 : P.nboxes); ++b) {
                        if (take) mbar_wait_call(bar_afull + 8 * at, apar, &abort_flag, P.status, kStatusWaitOperand);
                        tc_fence_after();
                        const uint32_t a_lo = ((((a_s + at * P.a_slot) & 0x3FFFFu) >> 4) | (1u << 16)) + k0;
                        if constexpr (NINE) {
                            if (nk == 1) gdw_issue<9, 1>(P, 0, d, a_lo, a_hi, b_lo + k0, b_hi, tap, idesc, more);
                            else if (nk == 2) gdw_issue<9, 2>(P, 0, d, a_lo, a_hi, b_lo + k0, b_hi, tap, idesc, more);
                            else if (nk == 3) gdw_issue<9, 3>(P, 0, d, a_lo, a_hi, b_lo + k0, b_hi, tap, idesc, more);
                            else gdw_issue<9, 4>(P, 0, d, a_lo, a_hi, b_lo + k0, b_hi, tap, idesc, more);
                            more = 1;
                        } else {
                            const uint32_t box = P.boxes[b];
                            int s = (int)((box >> 16) & 0xFFu);
                            const int s1 = s + (int)(box >> 24);
#pragma unroll 1
                            for (; nk == 1 && s + 5 <= s1; s += 5) {        // 5 x 5 taps: few channels have many filters
                                gdw_issue<5, 1>(P, s, d, a_lo, a_hi, b_lo + k0, b_hi, tap, idesc, more);
                                more = 1;
                            }
#pragma unroll 1
                            for (; s < s1; ++s) {
                                const uint32_t st = P.steps[s], al = a_lo + (st & 0xFFFFu), bl = b_lo + k0 + (st >> 16) * tap;
                                umma_pair_words(d, al, a_hi, bl, b_hi, idesc, more);
                                more = 1;
                                if (nk > 1) umma_pair_words(d, al + 2u, a_hi, bl + 2u, b_hi, idesc, 1u);
                                if (nk > 2) umma_pair_words(d, al + 4u, a_hi, bl + 4u, b_hi, idesc, 1u);
                                if (nk > 3) umma_pair_words(d, al + 6u, a_hi, bl + 6u, b_hi, idesc, 1u);
                            }
                        }
                        if (leave) umma_commit_pair(bar_aempty + 8 * at);
                        if (++at == (uint32_t)P.na) { at = 0; apar ^= 1u; }
                    }
                    if (leave) { slot = at; par = apar; }
                }
                umma_commit_pair(bar_accfull + 8 * acc);
            }
            umma_commit_pair(bar_drain);         // teardown: covers every product issued
        }
        __syncwarp();
    } else if (warp == kGdwAWarp) {
        if (lane == 0) {
            // ---------------- input boxes of this block's tile ----------------
            const uint32_t full0 = map_shared(bar_afull, 0);
            uint32_t slot = 0, par = 1;
            int n = 0;
            bool stop = false;
#pragma unroll 1
            for (int it = i0; it < i1 && !stop; ++it) {
                const uint32_t info = (uint32_t)chunks[run_of(it)];
                if (!(info & kGdwFirst) && it != i0) continue;       // the box is there
                int n0, h0, w0, c = (int)(info >> 16);
                tile_of(it, &n0, &h0, &w0);
#pragma unroll 1
                for (int steps = (int)((info >> 4) & 31u); steps > 0 && !stop; steps -= cb >> 4, c += cb)
#pragma unroll 1
                    for (int b = 0; b < P.nboxes; ++b, ++n) {
                        gdw_wait(bar_aempty + 8 * slot, par, &abort_flag, P.status, kStatusWaitStage);
                        if (*vabort) { stop = true; break; }
                        const int l0 = (int)(P.boxes[b] & 0xFFu), nl = (int)((P.boxes[b] >> 8) & 0xFFu);
                        if (rank == 0) mbar_expect_tx(bar_afull + 8 * slot, 2u * P.a_bytes * (uint32_t)nl);
#pragma unroll 1
                        for (int l = l0; l < l0 + nl; ++l)
                            tma_load_4d_pair(a_s + slot * P.a_slot + (uint32_t)(l - l0) * P.a_load, &P.tmap_x[P.load_map[l]], c, w0 + P.load_dw[l], h0 + P.load_dh[l],
                                             n0, full0 + 8 * slot);
                        if (++slot == (uint32_t)P.na) { slot = 0; par ^= 1u; }
                    }
            }
            // Teardown: the last phase armed on each slot completes when both blocks' copies have landed.
            if (rank == 0)
                for (int i = 0, j = n - 1; i < P.na && j >= 0; ++i, --j) mbar_wait_drain(bar_afull + 8 * (j % P.na), (uint32_t)(j / P.na) & 1u);
        }
    } else if (warp >= kGdwBuildWarp && warp < kGdwEpiWarp) {
        // ---------------- filters: this block's 32 of a run's 64 intermediate channels ----------------
        const int t = tid - kGdwBuildWarp * 32;
        const uint32_t full0 = map_shared(bar_bfull, 0), low = (uint32_t)P.rb / 16u - 1u;       // 16-byte pieces of a row less one: 1, 3, 7
        const int shift = P.rb == 128 ? 0 : (P.rb == 64 ? 1 : 2);                              // rows that share the pieces' order
        // A thread's row and taps of a run, asked for a run ahead: the loads' latency passes beside the stores of the run before.
        constexpr int kTaps = (kGdwMaxSteps + 3) / 4;
        const int r = t & 31, tap0 = t >> 5;
        float tap[kTaps];
        int ch = -1;
        auto fetch = [&](int q) {
            const int i = q * kChunk + (int)rank * 32 + r;       // < Gpad
            ch = __ldg(P.chan + i);
#pragma unroll
            for (int j = 0; j < kTaps; ++j) tap[j] = tap0 + 4 * j < P.k2 ? __ldcg(P.taps + (size_t)i * P.k2 + tap0 + 4 * j) : 0.f;
        };
        auto build = [&](int q, uint32_t buf, int next) {
            const uint32_t info = (uint32_t)chunks[q], dst = b_s + buf * P.b_buf;
            const int c0 = (int)(info >> 16);
            const uint32_t bytes = (((info >> 4) & 31u) * 16u > (uint32_t)cb ? 2u : 1u) * (uint32_t)P.k2 * P.b_tap;
            for (uint32_t o = (uint32_t)t * 16u; o < bytes; o += 2048u) sts128(dst + o, make_uint4(0, 0, 0, 0));
            named_bar_sync(1, 128);
            const int col = ch - c0, w = col >= cb ? 1 : 0, cl = col - w * cb;       // two boxes of 64 at most
            const uint32_t at = dst + (uint32_t)(w * P.k2 + tap0) * P.b_tap + (uint32_t)(r * P.rb) + ((((uint32_t)cl >> 3) ^ (((uint32_t)r >> shift) & low)) << 4) + (uint32_t)(cl & 7) * 2u;
#pragma unroll
            for (int j = 0; j < kTaps; ++j)
                if (ch >= 0 && tap0 + 4 * j < P.k2) sts16(at + 4u * (uint32_t)j * P.b_tap, float_to_bf16_bits(tap[j]));
            fetch(next);
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(full0 + 8 * buf);
        };
        if (P.resident) {
#pragma unroll 1
            for (int j = 0; j < min(P.nchunks, i1 - i0); ++j) {      // in the order in which they are needed
                const int q = (i0 + j) % P.nchunks;
                if (j == 0) fetch(q);
                build(q, (uint32_t)q, q + 1 < P.nchunks ? q + 1 : 0);
            }
        } else {
            uint32_t buf = 0, par = 1;
#pragma unroll 1
            for (int it = i0; it < i1;) {
                const int q = it / P.pairs;
                if (it == i0) fetch(q);
                gdw_wait(bar_bempty + 8 * buf, par, &abort_flag, P.status, kStatusWaitStage);
                build(q, buf, min(q + 1, P.nchunks - 1));
                if (++buf == (uint32_t)P.nb) { buf = 0; par ^= 1u; }
                it = (q + 1) * P.pairs;
            }
        }
    } else if (warp >= kGdwEpiWarp) {
        // ---------------- epilogue: TMEM -> bf16 -> z, 64 channels of 128 pixels at a time ----------------
        const int lg = warp & 3, r = lg * 32 + lane, grp = (warp - kGdwEpiWarp) >> 2;
        const bool issuer = lg == 0 && lane == 0;
        const uint32_t free0 = map_shared(bar_accfree, 0), row_s = o_s + (uint32_t)grp * 16384u + (uint32_t)r * 128u, rx = (uint32_t)(r & 7) << 4;
#pragma unroll 1
        for (int it = i0 + grp; grp < P.groups && it < i1; it += P.groups) {
            const int n = it - i0, acc = n & (kGdwAcc - 1), q = run_of(it);
            int n0, h0, w0;
            tile_of(it, &n0, &h0, &w0);
            if (lane == 0) gdw_wait(bar_accfull + 8 * acc, (uint32_t)(n >> 3) & 1u, &abort_flag, P.status, kStatusWaitMma);
            __syncwarp();
            tc_fence_after();
            if (issuer) bulk_wait_read_all();    // the staging buffer's last box has left it
            named_bar_sync(2 + grp, 128);
            uint32_t odd[2] = {};                // channels that are not finite
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                uint32_t v[32];
                tmem_ld32(tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(acc * 64 + h * 32), v);
                tmem_ld_wait();
                float worst = 0.f;               // NaN where a value is not finite
#pragma unroll
                for (int e = 0; e < 32; ++e) worst = fmaf(__uint_as_float(v[e]), 0.f, worst);
                if (worst != 0.f) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) odd[h] |= fabsf(__uint_as_float(v[e])) <= FLT_MAX ? 0u : 1u << e;
                }
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    uint32_t o[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[e] = pack_bf16x2(__uint_as_float(v[8 * p + 2 * e]), __uint_as_float(v[8 * p + 2 * e + 1]));
                    sts128(row_s + ((uint32_t)(h * 64 + p * 16) ^ rx), make_uint4(o[0], o[1], o[2], o[3]));
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(free0 + 8 * acc);
            if (__any_sync(0xffffffffu, odd[0] | odd[1])) gdw_plain<NINE ? 3 : 5>(&P, o_s + (uint32_t)grp * 16384u, lg * 32, n0, h0, w0, q * kChunk, odd[0], odd[1]);
            fence_proxy_async();
            named_bar_sync(2 + grp, 128);
            if (issuer) {
                tma_store_4d(o_s + (uint32_t)grp * 16384u, &P.tmap_z, q * kChunk, w0, h0, n0);
                bulk_commit();
            }
        }
        if (issuer) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0) mbar_wait_drain(bar_drain, 0);         // bounded, ignores the abort flag
    __syncwarp();
    cluster_sync();              // nothing of this pair is in flight any more: either block may end
    if (warp == kGdwTmemWarp) tmem_dealloc_pair(tmem, 64u * kGdwAcc);
}

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
namespace {

struct GdwLaunch {
    LaunchKey key;
    GdwParams P;
    double us = 0;               // estimate
    int IH = 0, IW = 0, grid = 0;
    size_t smem = 0;
    bool taken = false;
    const void *x = nullptr, *z = nullptr;       // the addresses the tensor maps were encoded for
};

struct GdwGeom {
    int layout = 0, TN = 0, PH = 0, PW = 0, IH = 0, IW = 0, nloads = 0, tiles_h = 0, tiles_w = 0;
    int64_t pairs = 0;
    double cycles = 0;
};

// Input channels that a run of 64 intermediate channels spans, from the last multiple of 8 before it.
int gdw_span(const gdws_plan_s *p, int q)
{
    const int c0 = p->chan[q * kChunk] & ~7, last = p->chan[std::min((q + 1) * kChunk, p->G) - 1];
    return last + 1 - c0;
}

// Everything about a launch but the addresses of x and z; false: not covered.
bool gdw_prepare(const gdws_plan_s *p, int n, int Ho, int Wo, GdwLaunch *L)
{
    const int k = p->k, sd = p->stride;
    if (k > 5 || sd > 2 || p->C % 8 || p->nchunks > kGdwMaxChunks || p->C > 0x7fff) return false;
    int widest = 0;
    double ksteps = 0;
    for (int q = 0; q < p->nchunks; ++q) {
        const int s = gdw_span(p, q);
        widest = std::max(widest, s);
        ksteps += k * k * ((s + 15) / 16);
    }
    if (widest > 128) return false;
    const int cb = widest <= 16 ? 16 : (widest <= 32 ? 32 : 64), nw = (widest + cb - 1) / cb;      // narrow boxes where the runs are narrow
    const TcTaps t = tc_taps(k, sd, p->pad);
    const int nclusters = std::max(1, sm_count_of(p) / 2);
    GdwGeom best;
    auto consider = [&](int layout, int TN, int PH, int PW) {
        GdwGeom g;
        g.layout = layout; g.TN = TN; g.PH = PH; g.PW = PW;
        g.tiles_h = (Ho + PH - 1) / PH; g.tiles_w = (Wo + PW - 1) / PW;
        g.pairs = ((int64_t)((n + TN - 1) / TN) * g.tiles_h * g.tiles_w + 1) / 2;
        g.IW = layout == 3 ? 4 : PW + t.ext;
        g.IH = layout == 1 ? PH + t.ext : PH;
        g.nloads = layout == 1 ? t.npar * t.npar : (layout == 2 ? k * t.npar : k * k);
        const double boxes = (double)g.nloads * TN * g.IH * g.IW * cb * 2 * nw / 45.0;       // one thread's loads: some 45 bytes per clock
        const double item = std::max(std::max(ksteps / p->nchunks * 46.0 + 300.0, boxes), 700.0);
        g.cycles = std::ceil((double)g.pairs * p->nchunks / nclusters) * item;
        if (!best.layout || g.cycles < best.cycles) best = g;
    };
    if (Wo > 4) {
        consider(1, 1, 16, 8);
        for (int PH = 8; PH >= 1; PH >>= 1) consider(2, 16 / PH, PH, 8);
    } else {
        for (int PH = 32; PH >= 2; PH >>= 1) consider(3, 32 / PH, PH, 4);
    }
    const GdwGeom &g = best;
    GdwParams &P = L->P;
    memset(&P, 0, sizeof(P));
    const int64_t nitems = g.pairs * p->nchunks;
    if (nitems > 0x3fffffffLL) return false;
    P.taps = p->d_dw; P.chan = p->d_chan; P.status = p->d_status;
    P.k2 = k * k; P.nchunks = p->nchunks; P.G = p->G;
    P.N = n; P.C = p->C; P.k = k; P.stride = sd; P.pad = p->pad; P.Ho = Ho; P.Wo = Wo;
    P.TN = g.TN; P.PH = g.PH; P.PW = g.PW; P.tiles_h = g.tiles_h; P.tiles_w = g.tiles_w; P.pairs = (int)g.pairs; P.nitems = (int)nitems;
    P.rb = cb * 2;
    P.swizzle = (cb == 64 ? 2u : (cb == 32 ? 4u : 6u)) << 29;    // 128-, 64-, 32-byte swizzle
    P.a_bytes = (uint32_t)(g.TN * g.IH * g.IW * P.rb);
    P.a_load = (P.a_bytes + 1023u) / 1024u * 1024u;
    P.a_sbo = g.layout == 3 ? 8u * (uint32_t)P.rb : (uint32_t)(g.IW * P.rb);
    P.b_tap = 32u * (uint32_t)P.rb;
    P.b_buf = (uint32_t)(nw * k * k) * P.b_tap;
    // All filters stay if they leave room for input boxes and two staging buffers; items then go tile by tile.  The loads of a window
    // share a box (one barrier) where two such boxes fit.
    const size_t fixed = 1024 + (size_t)p->nchunks * 4 + 64;
    bool placed = false;
    for (int resident = 1; resident >= 0 && !placed; --resident) {
        if (resident && p->nchunks > kGdwMaxB) continue;
        for (int groups = kGdwGroups; groups >= 2 && !placed; groups >>= 1)
            for (int per_box = g.nloads; per_box >= 1 && !placed; per_box = per_box > 2 ? (per_box + 1) / 2 : per_box - 1)
                for (int nb = resident ? p->nchunks : 2; nb >= (resident ? p->nchunks : 1) && !placed; --nb) {
                    const size_t used = fixed + (size_t)groups * 16384 + (size_t)nb * P.b_buf;
                    const size_t slot = (size_t)per_box * P.a_load;
                    if (used + 2 * slot > (size_t)kMaxSmem) continue;
                    P.na = (int)std::min<size_t>(kGdwMaxA, ((size_t)kMaxSmem - used) / slot);
                    P.a_slot = (uint32_t)slot; P.nb = nb; P.resident = resident; P.groups = groups;
                    placed = true;
                }
    }
    if (!placed) return false;
    const int per_box = (int)(P.a_slot / P.a_load);
    int nl = 0, ns = 0;
    auto add_load = [&](int hp, int wp, int dh, int dw) {
        P.load_map[nl] = hp * 2 + wp; P.load_dh[nl] = dh; P.load_dw[nl] = dw;
        P.maps_used |= 1 << (hp * 2 + wp);
        if (nl % per_box == 0) P.boxes[P.nboxes++] = (uint32_t)nl | (uint32_t)ns << 16;
        P.boxes[P.nboxes - 1] += 1u << 8;
        ++nl;
    };
    auto add_step = [&](int u, int v, int row, int col) {
        P.steps[ns++] = ((uint32_t)((row * g.IW + col) * P.rb) >> 4) + (P.a_load >> 4) * (uint32_t)((nl - 1) % per_box) | (uint32_t)(u * k + v) << 16;
        P.boxes[P.nboxes - 1] += 1u << 24;
    };
    for (int hp = 0; hp < sd && g.layout == 1; ++hp)
        for (int wp = 0; wp < sd; ++wp) {
            if (!t.used[hp] || !t.used[wp]) continue;
            add_load(hp, wp, t.omin[hp], t.omin[wp]);
            for (int u = 0; u < k; ++u)
                for (int v = 0; v < k; ++v)
                    if (t.par[u] == hp && t.par[v] == wp) add_step(u, v, t.off[u] - t.omin[hp], t.off[v] - t.omin[wp]);
        }
    for (int u = 0; u < k && g.layout == 2; ++u)
        for (int wp = 0; wp < sd; ++wp) {
            if (!t.used[wp]) continue;
            add_load(t.par[u], wp, t.off[u], t.omin[wp]);
            for (int v = 0; v < k; ++v)
                if (t.par[v] == wp) add_step(u, v, 0, t.off[v] - t.omin[wp]);
        }
    for (int u = 0; u < k && g.layout == 3; ++u)
        for (int v = 0; v < k; ++v) {
            add_load(t.par[u], t.par[v], t.off[u], t.off[v]);
            add_step(u, v, 0, 0);
        }
    if (nl != g.nloads || ns != k * k) return false;
    // Runs that share a box: neighbours whose channels lie within its 64 from the first run's first channel on.  A tile's boxes then stay
    // until its last run has read them, which only pays (and with fewer slots than boxes would wait forever) if the next tile's fit beside them.
    const bool share = nw == 1 && P.na >= 2 * P.nboxes;
    for (int q = 0, first = 0; P.resident && q < p->nchunks; ++q) {
        const int lo = p->chan[q * kChunk], hi = p->chan[std::min((q + 1) * kChunk, p->G) - 1] + 1;
        if (q == first) P.info[q] = kGdwFirst | (uint32_t)(lo & ~7) << 16;
        const int c0 = (int)(P.info[first] >> 16);
        if (q > first && (!share || hi - c0 > cb)) {
            P.info[q - 1] |= kGdwLast;
            first = q--;
            continue;
        }
        const int k0 = (lo - c0) / 16;
        P.info[q] |= (uint32_t)c0 << 16 | (uint32_t)k0 | (uint32_t)((hi - c0 + 15) / 16 - k0) << 4;
    }
    if (P.resident) P.info[p->nchunks - 1] |= kGdwLast;
    div_magic(P.resident ? p->nchunks : (int)g.pairs, P.dv_run); div_magic(g.tiles_h * g.tiles_w, P.dv_thw); div_magic(g.tiles_w, P.dv_tw);
    P.off_a = (uint32_t)P.groups * 16384u;
    P.off_b = P.off_a + (uint32_t)P.na * P.a_slot;
    P.off_chunk = P.off_b + (uint32_t)P.nb * P.b_buf;
    L->smem = std::max<size_t>(1024 + (size_t)P.off_chunk + (size_t)p->nchunks * 4, kMaxSmem / 2 + 4096);      // one block per SM: it takes all of the tensor memory
    L->IH = g.IH; L->IW = g.IW;
    // Fitted to 45 layers, within 20 % of most: an item of 3 x 3 taps takes 1.08 us, of 5 x 5 1.95, or what its boxes take to arrive.
    const double item = std::max(k <= 3 ? 1.08 : 1.95, (double)P.a_bytes * g.nloads * nw / 52e3);
    L->us = 6.5 + std::ceil((double)nitems / nclusters) * item + (P.nboxes - 1);      // boxes one after the other: a microsecond each, once
    L->grid = 2 * (int)std::min<int64_t>(nitems, nclusters);
    return true;
}

// The GDW stage on the ALUs: a run of 64 channels of a tile takes 1.43 us (5 x 5: 2.05; 0.55 per tap where no specialised code applies).
double gdw_alu_us(const gdws_plan_s *p, int n, int h, int w)
{
    Tile t;
    if (!choose_tile(p, n, h, w, &t)) return 1e9;
    const double run = t.fast ? (p->k == 5 ? (p->stride == 1 ? 2.05 : 1.4) : 1.43) : 0.55 * p->k * p->k;
    return 2.5 + std::ceil((double)t.tiles() / sm_count_of(p)) * p->nchunks * run;
}

gdws_status_t gdw_maps(const gdws_plan_s *p, const gdws_tensor_t *x, void *z, GdwLaunch *L)
{
    GdwParams &P = L->P;
    tensor_map_encode_fn encode = encode_fn();
    if (!encode) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from this driver");
    const int sd = p->stride;
    const CUtensorMapSwizzle sw = P.rb == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : (P.rb == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const bool anew = L->x != x->ptr;
    if (anew) L->x = nullptr;    // until all of them are of this address
    for (int m = 0; m < 4 && anew; ++m) {
        if (!((P.maps_used >> m) & 1)) continue;
        const int hp = m >> 1, wp = m & 1, Wp = (x->w - wp + sd - 1) / sd, Hp = (x->h - hp + sd - 1) / sd;
        const cuuint64_t dims[4] = {(cuuint64_t)p->C, (cuuint64_t)Wp, (cuuint64_t)Hp, (cuuint64_t)x->n};
        const cuuint64_t strides[3] = {(cuuint64_t)sd * p->C * 2, (cuuint64_t)sd * x->w * p->C * 2, (cuuint64_t)x->h * x->w * p->C * 2};
        const cuuint32_t box[4] = {(cuuint32_t)P.rb / 2, (cuuint32_t)L->IW, (cuuint32_t)L->IH, (cuuint32_t)P.TN};
        const CUresult r = encode(&P.tmap_x[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (uint8_t *)x->ptr + ((size_t)hp * x->w + wp) * p->C * 2, dims, strides, box, estr,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (x) failed with code %d", (int)r);
    }
    L->x = x->ptr;
    P.x = (const uint16_t *)x->ptr;
    if (L->z != z) {
        const cuuint64_t gp = (cuuint64_t)p->Gpad;
        const cuuint64_t dims[4] = {gp, (cuuint64_t)P.Wo, (cuuint64_t)P.Ho, (cuuint64_t)x->n};
        const cuuint64_t strides[3] = {gp * 2, (cuuint64_t)P.Wo * gp * 2, (cuuint64_t)P.Ho * P.Wo * gp * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)P.PW, (cuuint32_t)P.PH, (cuuint32_t)P.TN};
        const CUresult r = encode(&P.tmap_z, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, z, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                  CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (z) failed with code %d", (int)r);
        L->z = z;
    }
    return GDWS_OK;
}

}  // namespace

// The prepared launch of a size; null without host memory for it.
static GdwLaunch *gdw_prepared(gdws_plan_s *p, int n, int h, int w)
{
    const LaunchKey key = {n, h, w, p->opt_dw_math};
    if (GdwLaunch *L = LaunchCache<GdwLaunch>::find(p->launch_cache[kCacheGdw], key)) return L;
    std::unique_ptr<GdwLaunch> e(new (std::nothrow) GdwLaunch);
    if (!e) return nullptr;
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    e->key = key;
    // one row or column and stride 2: the view of the odd ones is empty
    e->taken = p->G > 0 && !(p->stride == 2 && (h < 2 || w < 2) && tc_taps(p->k, 2, p->pad).used[1]) && gdw_prepare(p, n, Ho, Wo, e.get());
    e->P.H = h; e->P.W = w;
    if (e->taken && p->opt_dw_math != 2) e->taken = e->us < gdw_alu_us(p, n, h, w);
    return LaunchCache<GdwLaunch>::add(p->launch_cache[kCacheGdw], std::move(e));
}

bool bf16_depthwise_on_tc(gdws_plan_s *p, int n, int h, int w)
{
    if (p->opt_dw_math == 1 || p->opt_tile || p->opt_a_layout) return false;
    const GdwLaunch *L = gdw_prepared(p, n, h, w);
    return L && L->taken;
}

// GDWS_ERR_UNSUPPORTED: not covered, nothing was launched.
gdws_status_t bf16_depthwise_tc(gdws_plan_s *p, const gdws_tensor_t *x, void *z, cudaStream_t st)
{
    GdwLaunch *L = gdw_prepared(p, x->n, x->h, x->w);
    if (!L) return fail(GDWS_ERR_ALLOC, "out of host memory");
    if (!L->taken) return fail(GDWS_ERR_UNSUPPORTED, "GDW stage on the tensor cores: layer not covered");
    const gdws_status_t rc = gdw_maps(p, x, z, L);
    if (rc != GDWS_OK) return rc;
    const int nine = L->P.k2 == 9 && L->P.nboxes == 1;
    const auto kernel = nine ? gdw_tc_kernel<true> : gdw_tc_kernel<false>;
    static bool attr_set[64][2] = {};
    if (!attr_set[p->device & 63][nine]) {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(gdw_tc_kernel)");
        attr_set[p->device & 63][nine] = true;
    }
    const cudaError_t e = launch_overlapped(kernel, (unsigned)L->grid, kGdwThreads, L->smem, st, L->P);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "gdw_tc_kernel launch"); }
    p->launches++;
    return GDWS_OK;
}

}  // namespace gdws
