// The GDWS forward as ONE k x k convolution with folded filters, bf16 NHWC, on sm_100a.
//
// y = P (K x): the layer is a product of two linear maps, and the products may be taken in either order.  The two-stage
// kernels form z = K x per pixel and then P z; this one forms the k x k filters W[d,c,u,v] = sum_j P[d, off_c+j] K[off_c+j,u,v]
// (Property 1 and 2; the proof of Lemma 1 reads the same identity backwards) when the weights are packed, and runs
//     y[pixel, d] = bias[d] + sum_{u,v,c} x[pixel shifted by (u,v), c] W[d,c,u,v]
// as a tensor-core product with fp32 accumulators over k*k*C.  It takes C k^2 D multiply-adds per pixel where the two
// stages take G (k^2 + D), but all of them run at full tensor-core rate: nothing is rounded, scattered or handed over
// between two stages.  The one bf16 rounding between the stages moves from z to W (measured 1.66e-3 of the result either
// way, before y's own); where filters cut a constant input off W is taken in two terms (kFoldPass).  bf16_form_of below decides per layer and input size.
//
// What bounds it, and the layout that follows:
//   * A operand (x): the input box of a tile is staged once per 64 input channels as [row][column][64 channels] (128 bytes
//     per pixel, 128-byte swizzle, written by TMA).  For every tap it is a valid K-major operand (8 output pixels of a row
//     are 8 consecutive 128-byte rows, groups of 8 are a row pitch apart) that differs from the next tap's only in its
//     start address, so x is fetched once (plus halo) and not once per tap.
//   * B operand (W): 128 x N x 16 products are bound by the tensor pipe from N = 128 on only if the operand traffic keeps
//     up: the L2 delivers some 59 bytes per clock and SM, one block with N = 256 would ask for 64.  Two blocks (a cluster)
//     therefore share one product of M = 256 (cta_group::2): each holds its own 128 pixels and HALF of the filters, which
//     halves the weight traffic and the shared memory they take.  Where all filters of a block's share fit shared memory
//     beside the input boxes they are loaded once and stay.
//   * The accumulators are double buffered (2 x up to 256 TMEM columns): a tile's epilogue overlaps the next tile.
//
// Roles per block of 24 warps: warps 0 and 1 issue the products (leader block only), 2 and 3 load the input boxes, 4 and 5
// the filters (one lane each), warp 6 allocates tensor memory, warps 8-23 run the epilogue.  A work item is a pair of
// tiles of 128 output pixels x a block of up to 256 output channels.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>

#include "sm100.cuh"

namespace gdws {

constexpr int kFoldAWarp = 2, kFoldBWarp = 4, kFoldTmemWarp = 6, kFoldTermWarp = 7;     // two warps each for products, input boxes, filters
constexpr int kFoldEpiWarp0 = 8, kFoldEpiGroups = 4;      // up to four groups of four epilogue warps
constexpr int kFoldMaxSmem = 226 * 1024;                  // dynamic shared memory (227 KB less the barriers)
constexpr int kFoldThreads = (kFoldEpiWarp0 + 4 * kFoldEpiGroups) * 32;
constexpr int kFoldMaxSteps = 25;        // taps
constexpr int kFoldMaxA = 8;             // input box slots
constexpr int kFoldMaxB = 40;            // filter units in shared memory (one tap x 64 input channels each)
constexpr uint32_t kFoldSw128 = 2u << 29;   // descriptor high word: layout type "128-byte swizzle"
constexpr int kFoldMaxAcc = 8;           // accumulators in tensor memory
// A unit is a run of product steps (taps) whose filters share one barrier: bits 0-7 its first step, 8-15 its steps,
// then whether it is the first / last one that reads its input box.
constexpr uint32_t kUnitFirst = 1u << 16, kUnitLast = 1u << 17, kUnitLastBox = 1u << 18;   // LastBox: the first unit of the window's last box

struct alignas(64) FoldParams {
    CUtensorMap tmap_x[4];       // x as (C, W, H, N), box (64, IW, rows, TN), 128-byte swizzle; stride 2: one dense view per parity
    CUtensorMap tmap_w;          // folded filters as rows of 64 input channels, box (64, Npart / 2)
    CUtensorMap tmap_y;          // y as (D, Wo, Ho, N), box (128 bytes of channels, PW, PH, TN)
    const float *bias;
    const float2 *sums;          // of the packing blocks (kFoldPass)
    int nsums;
    int *status;
    int nwin, nk_last, nsteps, nunits, nboxes, mma_warps;
    uint32_t steps[kFoldMaxSteps];       // per product step of a window: A offset / 16, tap << 16
    uint32_t units[kFoldMaxSteps];
    uint32_t boxes[kFoldMaxSteps];       // per input box of a window: its first load, loads << 8
    int load_map[kFoldMaxSteps], load_dw[kFoldMaxSteps], load_dh[kFoldMaxSteps];
    int D, Dp, Npart, nparts, relu, out_f32;
    int TN, PH, PW, tiles_h, tiles_w, nitems;
    uint32_t dv_parts[2], dv_thw[2], dv_tw[2];
    uint32_t a_sbo, a_bytes, a_load, a_slot, b_tap, b_unit;      // b_tap: bytes of one tap's filters, b_unit: of a unit's slot
    int maps_used;
    int na, nb, resident, acc_cols, nacc, nacc_shift;
    uint32_t a_skip, a_flip, b_skip, b_flip;     // ring places and parity changes that an item's boxes / units amount to
    int gi, gb;                                  // epilogue groups: gi take alternate items, gb share an item's column blocks
    uint32_t off_a, off_b, off_bias;
};

__device__ __forceinline__ int fold_div(int n, const uint32_t (&md)[2]) { return (int)(((uint64_t)(uint32_t)n * md[0]) >> md[1]); }

__device__ __forceinline__ void fold_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (!mbar_try_wait(bar, parity)) mbar_wait_relaxed_slow(bar, parity, 16384u, abort_flag, status, code);
}
// The leader waits for arrivals from both blocks: acquire at cluster scope.  Bounded like the others.
__device__ __forceinline__ uint32_t fold_try_wait_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
static __device__ __noinline__ void fold_wait_cluster(uint32_t bar, uint32_t parity, volatile int *abort_flag, int *status, int code)
{
    if (*abort_flag) return;
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        if (fold_try_wait_cluster(bar, parity)) return;
        if (it > 4096) __nanosleep(64);
        if ((it & 1023) == 1023 && *abort_flag) return;
    }
    *abort_flag = 1;
    atomicOr(status, code);
}

// The products of one unit: n steps of nk x (K = 16).  Straight-line code when both are constants (STEPS, NK not 0).
template <int STEPS, int NK>
__device__ __forceinline__ void fold_issue(const FoldParams &P, int s0, int n, int nk, uint32_t d, uint32_t a_lo, uint32_t a_hi, uint32_t b_lo, uint32_t b_hi,
                                           uint32_t b_tap, uint32_t idesc, uint32_t accumulate)
{
    if constexpr (STEPS != 0) {
#pragma unroll
        for (int j = 0; j < STEPS; ++j) {
            const uint32_t al = a_lo + (P.steps[s0 + j] & 0xFFFFu), bl = b_lo + (uint32_t)j * b_tap;
#pragma unroll
            for (int kk = 0; kk < NK; ++kk) umma_pair_words(d, al + 2u * kk, a_hi, bl + 2u * kk, b_hi, idesc, j | kk ? 1u : accumulate);
        }
    } else {
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
            const uint32_t al = a_lo + (P.steps[s0 + j] & 0xFFFFu), bl = b_lo + (uint32_t)j * b_tap;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
                if (NK == 4 || kk < nk) umma_pair_words(d, al + 2u * kk, a_hi, bl + 2u * kk, b_hi, idesc, (uint32_t)j | accumulate | (uint32_t)kk);
        }
    }
}

struct FoldBars { uint32_t afull, aempty, bfull, bempty, accfull, accfree; };

// The rest of the products where the filters need their second term, by the thread that has issued item 0's first term: item 0's
// windows once more, then the other items, twice through their windows each.  The filters pass through their ring, also where
// there is room for all of one term.  (As a variant of the loops of the common case, with a flag in registers, it cost every
// layer 2 to 4 %: what those loops compare with has to stay in the constant bank.)
static __device__ __noinline__ void fold_second(const FoldParams *params, int my_items, uint32_t tmem, uint32_t a_s, uint32_t b_s, FoldBars bar, volatile int *abort_flag)
{
    const FoldParams &P = *params;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.Npart >> 3) << 17) | (16u << 24);
    const uint32_t a_hi = ((P.a_sbo >> 4) & 0x3FFFu) | (1u << 14) | kFoldSw128, b_hi = (1024u >> 4) | (1u << 14) | kFoldSw128;
    const uint32_t a_lo0 = ((a_s & 0x3FFFFu) >> 4) | (1u << 16), b_lo0 = ((b_s & 0x3FFFFu) >> 4) | (1u << 16);
    if (P.resident)              // item 0's first term did not release its filters
        for (int u = 0; u < P.nb; ++u) umma_commit_pair(bar.bempty + 8 * (uint32_t)u);
    // both rings as the first term leaves them
    const int boxes = P.nwin * P.nboxes, units = P.nwin * P.nunits;
    uint32_t aslot = (uint32_t)(boxes % P.na), apar = (uint32_t)(boxes / P.na) & 1u, bslot = (uint32_t)(units % P.nb), bpar = (uint32_t)(units / P.nb) & 1u;
#pragma unroll 1
    for (int it = 0; it < my_items; ++it) {
        const int buf = it & (P.nacc - 1);
        const uint32_t d = tmem + (uint32_t)(buf * P.acc_cols);
        if (it >= P.nacc) fold_wait_cluster(bar.accfree + 8 * buf, (uint32_t)((it >> P.nacc_shift) - 1) & 1u, abort_flag, P.status, kStatusWaitStage);
#pragma unroll 1
        for (int w = it ? 0 : P.nwin; w < 2 * P.nwin; ++w) {
            const int nk = w == P.nwin - 1 || w == 2 * P.nwin - 1 ? P.nk_last : 4;
#pragma unroll 1
            for (int u = 0; u < P.nunits; ++u) {
                const uint32_t un = P.units[u];
                if (un & kUnitFirst) mbar_wait_call(bar.afull + 8 * aslot, apar, abort_flag, P.status, kStatusWaitOperand);
                mbar_wait_call(bar.bfull + 8 * bslot, bpar, abort_flag, P.status, kStatusWaitOperand);
                tc_fence_after();
                fold_issue<0, 0>(P, (int)(un & 0xFFu), (int)((un >> 8) & 0xFFu), nk, d, a_lo0 + aslot * (P.a_slot >> 4), a_hi, b_lo0 + bslot * (P.b_unit >> 4), b_hi, P.b_tap >> 4,
                                 idesc, (uint32_t)(w | u));
                umma_commit_pair(bar.bempty + 8 * bslot);
                if (++bslot == (uint32_t)P.nb) { bslot = 0; bpar ^= 1u; }
                if (un & kUnitLast) {
                    umma_commit_pair(bar.aempty + 8 * aslot);
                    if (++aslot == (uint32_t)P.na) { aslot = 0; apar ^= 1u; }
                }
            }
        }
        if (it != my_items - 1) umma_commit_pair(bar.accfull + 8 * buf);
    }
}

// UNITS x STEPS: the window's units when they are all alike (unrolled: 3 x 3 taps or 9 x 1), 0: table driven.  NK: 1 to 3: the only
// window has so many K steps of 16 channels (up to 48 channels: straight-line code as for whole windows, 16 x 32 -> 16 x 192 x 165 31.3 ->
// 26.6 us); 4: whole windows, and a last one of any number.
template <int UNITS, int STEPS, int NK = 4>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kFoldThreads, 1) fold_kernel(const __grid_constant__ FoldParams P)
{
    extern __shared__ uint8_t smem_raw[];
    // afull[8] aempty[8] | bfull[40] bempty[40] | accfull[8] accfree[8] | turn[2] | drain | terms
    constexpr int kBars = 2 * kFoldMaxA + 2 * kFoldMaxB + 2 * kFoldMaxAcc + 4;
    __shared__ __align__(8) uint64_t bars[kBars];
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag;
    __shared__ int second_term;      // 1: the filters' second term is taken as well (bar_terms: it is known)
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_rank();
    volatile int *const vabort = &abort_flag;
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t o_s = smem_u32(base);
    const uint32_t a_s = o_s + P.off_a, b_s = o_s + P.off_b;
    float *bias_sm = reinterpret_cast<float *>(base + P.off_bias);
    const uint32_t bar_afull = smem_u32(&bars[0]), bar_aempty = bar_afull + 8 * kFoldMaxA;
    const uint32_t bar_bfull = bar_aempty + 8 * kFoldMaxA, bar_bempty = bar_bfull + 8 * kFoldMaxB;
    const uint32_t bar_accfull = bar_bempty + 8 * kFoldMaxB, bar_accfree = bar_accfull + 8 * kFoldMaxAcc, bar_turn = bar_accfree + 8 * kFoldMaxAcc, bar_drain = bar_turn + 16, bar_terms = bar_drain + 8;

    if (tid == 0) abort_flag = second_term = 0;
    // Full barriers are used in the leader only (its own arrive with the bytes of both blocks); "free" barriers are
    // completed in both blocks by the leader's commits; accfree counts the epilogue warps of both blocks.
    if (tid < kBars) {
        static_assert(kBars <= kFoldThreads, "one barrier per thread");
        const int acc = tid - (2 * kFoldMaxA + 2 * kFoldMaxB);
        mbar_init(bar_afull + 8 * (uint32_t)tid, acc >= kFoldMaxAcc && acc < 2 * kFoldMaxAcc ? 8u * (uint32_t)P.gb : (tid == kBars - 2 ? 2u : 1u));
        fence_mbar_init();
    }
    grid_launch_dependents();
    if (warp == kFoldAWarp && lane == 0) {
#pragma unroll 1
        for (int l = 0; l < 4; ++l)
            if ((P.maps_used >> l) & 1) prefetch_tensor_map(&P.tmap_x[l]);
    } else if (warp == kFoldBWarp && lane == 0) {
        prefetch_tensor_map(&P.tmap_w);
    } else if (warp == kFoldEpiWarp0 && lane == 0) {
        prefetch_tensor_map(&P.tmap_y);
    }
    if (warp == kFoldTmemWarp) tmem_alloc_pair(smem_u32(&tmem_slot), (uint32_t)(P.nacc * P.acc_cols));
    tc_fence_before();
    __syncthreads();
    cluster_sync();              // both blocks' barriers are initialised before either signals the other's
    tc_fence_after();
    grid_dependency_wait();      // from here on global memory is touched
    const uint32_t tmem = tmem_slot;
    const int cluster = (int)blockIdx.x >> 1, nclusters = (int)gridDim.x >> 1;
    const int my_items = (P.nitems - cluster + nclusters - 1) / nclusters;
    const int nunits = UNITS ? UNITS : P.nunits;
    // Whether an item takes the windows once more for the filters' second term.  All roles ask after the first item's first
    // term, so that the sums are read beside the first copies and products.
    auto two_terms = [&]() -> int {
        fold_wait(bar_terms, 0, &abort_flag, P.status, kStatusWaitOperand);
        return *(volatile int *)&second_term;
    };

    if (warp < kFoldAWarp) {
        if (rank == 0 && elect_one()) {
            // ---------------- products: one thread, or one in each of two warps that take alternate items ----------------
            // The tensor pipe queues only some two products per thread: what a thread does between its products (waits,
            // commits, some fifty cycles each) would leave the pipe idle if the other thread's were not there.  The warps
            // take turns at WAITING for boxes and filters: a phase parity names a barrier's phase only to a thread that
            // knows the phase before it to be complete, i.e. that everything the rings held for earlier items has landed.
            // The next unit's barriers are polled right after a unit's commits, so that the poll's round trip (a hundred
            // cycles) passes while the tensor pipe works on what was queued.
            const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(P.Npart >> 3) << 17) | (16u << 24);   // fp32 += bf16 x bf16, M = 256
            const uint32_t a_hi = ((P.a_sbo >> 4) & 0x3FFFu) | (1u << 14) | kFoldSw128;
            const uint32_t b_hi = (1024u >> 4) | (1u << 14) | kFoldSw128;
            const uint32_t a_lo0 = ((a_s & 0x3FFFFu) >> 4) | (1u << 16), b_lo0 = ((b_s & 0x3FFFFu) >> 4) | (1u << 16);
            const uint32_t a_step = P.a_slot >> 4, b_step = P.b_unit >> 4;
            const uint32_t b_tap = P.b_tap >> 4;
            uint32_t aslot = 0, apar = 0, bslot = 0, bpar = 0, a_lo = a_lo0, b_lo = b_lo0;
            uint32_t seen_a = 0, seen_b = 0;
            auto skip_item = [&]() {             // past the boxes and filters of the other warp's item
                aslot += P.a_skip; apar ^= P.a_flip;
                if (aslot >= (uint32_t)P.na) { aslot -= (uint32_t)P.na; apar ^= 1u; }
                a_lo = a_lo0 + aslot * a_step;
                if (!P.resident) {
                    bslot += P.b_skip; bpar ^= P.b_flip;
                    if (bslot >= (uint32_t)P.nb) { bslot -= (uint32_t)P.nb; bpar ^= 1u; }
                    b_lo = b_lo0 + bslot * b_step;
                }
            };
            const bool two = P.mma_warps == 2;
            if (warp == 1) skip_item();
            int it = two || warp == 0 ? warp : my_items;
            if (two && warp == 1 && two_terms()) it = my_items;      // fold_second takes all items
#pragma unroll 1
            for (; it < my_items; it += P.mma_warps) {
                const int buf = it & (P.nacc - 1);
                const uint32_t d = tmem + (uint32_t)(buf * P.acc_cols);
                if (it >= P.nacc) {
                    const uint32_t par = (uint32_t)((it >> P.nacc_shift) - 1) & 1u;
                    if (!fold_try_wait_cluster(bar_accfree + 8 * buf, par)) fold_wait_cluster(bar_accfree + 8 * buf, par, &abort_flag, P.status, kStatusWaitStage);
                }
                if (two && it > 0)  // the other warp has waited for all of item it - 1
                    mbar_wait_call(bar_turn + 8 * (uint32_t)(warp ^ 1), (uint32_t)((it - 1) >> 1) & 1u, &abort_flag, P.status, kStatusWaitStage);
                const bool wait_b = !P.resident || it < P.mma_warps;
                if (two) seen_a = seen_b = 0;
                if (P.resident) { bslot = 0; b_lo = b_lo0; }
#pragma unroll 1
                for (int w = 0; w < P.nwin; ++w) {
                    const int nk = w == P.nwin - 1 ? P.nk_last : 4;
#pragma unroll (UNITS ? UNITS : 1)
                    for (int u = 0; u < nunits; ++u) {
                        const uint32_t un = P.units[u];
                        const bool first = un & kUnitFirst, last = un & kUnitLast;
                        if (first && !seen_a) mbar_wait_call(bar_afull + 8 * aslot, apar, &abort_flag, P.status, kStatusWaitOperand);
                        if (wait_b && !seen_b) mbar_wait_call(bar_bfull + 8 * bslot, bpar, &abort_flag, P.status, kStatusWaitOperand);
                        if (two && w == P.nwin - 1 && (wait_b ? u == nunits - 1 : (un & kUnitLastBox) != 0)) mbar_arrive(bar_turn + 8 * (uint32_t)warp);
                        tc_fence_after();
                        const int s0 = STEPS ? u * STEPS : (int)(un & 0xFFu), n = (int)((un >> 8) & 0xFFu);
                        if constexpr (NK != 4) fold_issue<STEPS, NK>(P, s0, n, NK, d, a_lo, a_hi, b_lo, b_hi, b_tap, idesc, (uint32_t)u);
                        else if (nk == 4) fold_issue<STEPS, 4>(P, s0, n, 4, d, a_lo, a_hi, b_lo, b_hi, b_tap, idesc, (uint32_t)(w | u));
                        else fold_issue<0, 0>(P, s0, n, nk, d, a_lo, a_hi, b_lo, b_hi, b_tap, idesc, (uint32_t)(w | u));
                        if (!P.resident) umma_commit_pair(bar_bempty + 8 * bslot);
                        if (last) umma_commit_pair(bar_aempty + 8 * aslot);
                        b_lo += b_step;
                        if (++bslot == (uint32_t)P.nb) { bslot = 0; b_lo = b_lo0; bpar ^= (uint32_t)!P.resident; }
                        if (last) {
                            a_lo += a_step;
                            if (++aslot == (uint32_t)P.na) { aslot = 0; a_lo = a_lo0; apar ^= 1u; }
                        }
                        if (w == P.nwin - 1 && u == nunits - 1) {
                            if (it == 0 && two_terms()) {
                                fold_second(&P, my_items, tmem, a_s, b_s, {bar_afull, bar_aempty, bar_bfull, bar_bempty, bar_accfull, bar_accfree}, &abort_flag);
                                goto issued;
                            }
                            if (it != my_items - 1) umma_commit_pair(bar_accfull + 8 * buf);
                            if (two) skip_item();
                        }
                        if (!two || w != P.nwin - 1 || u != nunits - 1) {
                            if (wait_b) seen_b = mbar_try_wait(bar_bfull + 8 * bslot, bpar);
                            if (last) seen_a = mbar_try_wait(bar_afull + 8 * aslot, apar);
                        }
                    }
                }
            }
        issued:
            // Teardown: one more commit covers every product issued and every earlier commit's arrival in both blocks.
            umma_commit_pair(bar_drain);
        }
        __syncwarp();
    } else if (warp < kFoldBWarp) {
        if (lane == 0) {
            // ---------------- input boxes of this block's tile ----------------
            // Two warps take alternate boxes (a box costs a thread some 400 cycles of waits and set-up).  With an odd number of
            // slots one warp takes all: a thread may only wait for phases of slots whose every earlier phase it waited for.
            const int me = warp - kFoldAWarp, step = P.na & 1 ? 1 : 2;
            uint32_t slot = (uint32_t)me, par = 1;           // na >= 2
            int n = 0;                                       // boxes up to here, both warps' together
            const uint32_t full0 = map_shared(bar_afull, 0);
            int terms = 1;                                   // of the filters: the windows are taken once for each
            bool stop = false;
#pragma unroll 1
            for (int it = 0; it < my_items && !stop; ++it) {
                int tile = 2 * fold_div(cluster + it * nclusters, P.dv_parts) + (int)rank;
                const int bn = fold_div(tile, P.dv_thw);
                tile -= bn * P.tiles_h * P.tiles_w;
                const int bh = fold_div(tile, P.dv_tw), bw = tile - bh * P.tiles_w;
                const int n0 = bn * P.TN, h0 = bh * P.PH, w0 = bw * P.PW;
#pragma unroll 1
                for (int t = 0; t < terms; ++t) {
#pragma unroll 1
                    for (int w = 0; w < P.nwin && !stop; ++w)
#pragma unroll 1
                        for (int b = 0; b < P.nboxes; ++b, ++n) {
                            if ((n & (step - 1)) != me) continue;
                            if (n >= P.na) fold_wait(bar_aempty + 8 * slot, par, &abort_flag, P.status, kStatusWaitStage);
                            if (*vabort) { stop = true; break; }
                            const int l0 = (int)(P.boxes[b] & 0xFFu), nl = (int)(P.boxes[b] >> 8);
                            if (rank == 0) mbar_expect_tx(bar_afull + 8 * slot, 2u * P.a_bytes * (uint32_t)nl);
#pragma unroll 1
                            for (int j = 0; j < nl; ++j) {
                                const int l = l0 + j;
                                tma_load_4d_pair(a_s + slot * P.a_slot + (uint32_t)j * P.a_load, &P.tmap_x[P.load_map[l]], w * 64, w0 + P.load_dw[l], h0 + P.load_dh[l],
                                                 n0, full0 + 8 * slot);
                            }
                            slot += (uint32_t)step;
                            if (slot >= (uint32_t)P.na) { slot -= (uint32_t)P.na; par ^= 1u; }
                        }
                    if (it + t == 0) terms += two_terms();
                }
            }
            // Teardown: the last phase armed on each slot completes when both blocks' copies have landed (box j and those
            // of the same parity are this warp's; a warp that stopped early armed box n - 2 or n - 1 last).
            if (rank == 0)
                for (int i = 0, j = n - 1; i < P.na && j >= 0; ++i, --j)
                    if ((j & (step - 1)) == me) mbar_wait_drain(bar_afull + 8 * (j % P.na), (uint32_t)(j / P.na) & 1u);
        }
    } else if (warp < kFoldTmemWarp) {
        if (lane == 0) {
            // ---------------- filters: this block's half of the work item's output channels ----------------
            const int me = warp - kFoldBWarp, step = P.nb & 1 ? 1 : 2;     // as the boxes
            uint32_t slot = (uint32_t)me, par = 1;           // nb >= 2
            int n = 0;
            const uint32_t full0 = map_shared(bar_bfull, 0);
            int terms = 1;
            bool stop = false;
#pragma unroll 1
            for (int it = 0; it < my_items && !stop; ++it) {
                const int item = cluster + it * nclusters;
                const int part = item - fold_div(item, P.dv_parts) * P.nparts;
                const int d0 = part * P.Npart + (int)rank * (P.Npart >> 1);
#pragma unroll 1
                for (int t = 0; t < terms; ++t) {
                    const int row0 = t * P.nwin * P.nsteps * P.Dp + d0;
#pragma unroll 1
                    for (int w = 0; w < P.nwin && !stop; ++w)
#pragma unroll 1
                        for (int u = 0; u < nunits; ++u, ++n) {
                            if ((n & (step - 1)) != me) continue;
                            if (n >= P.nb) fold_wait(bar_bempty + 8 * slot, par, &abort_flag, P.status, kStatusWaitStage);
                            if (*vabort) { stop = true; break; }
                            const int s0 = (int)(P.units[u] & 0xFFu), ns = (int)((P.units[u] >> 8) & 0xFFu);
                            if (rank == 0) mbar_expect_tx(bar_bfull + 8 * slot, 2u * P.b_tap * (uint32_t)ns);
#pragma unroll 1
                            for (int j = 0; j < ns; ++j) {
                                const int tap = (int)((P.steps[s0 + j] >> 16) & 0xFFu);
                                tma_load_2d_pair(b_s + slot * P.b_unit + (uint32_t)j * P.b_tap, &P.tmap_w, 0, (w * P.nsteps + tap) * P.Dp + row0, full0 + 8 * slot);
                            }
                            slot += (uint32_t)step;
                            if (slot >= (uint32_t)P.nb) { slot -= (uint32_t)P.nb; par ^= 1u; }
                        }
                    if (it + t == 0) terms += two_terms();
                }
                if (P.resident && terms == 1) break;       // they stay
            }
            if (rank == 0)
                for (int i = 0, j = n - 1; i < P.nb && j >= 0; ++i, --j)
                    if ((j & (step - 1)) == me) mbar_wait_drain(bar_bfull + 8 * (j % P.nb), (uint32_t)(j / P.nb) & 1u);
        }
    } else if (warp == kFoldTermWarp) {
        // ---------------- one term of the filters or two ----------------
        const bool second = fold_second_term(P.sums, P.nsums, lane);
        if (lane == 0) {
            second_term = second;
            mbar_arrive(bar_terms);
        }
        __syncwarp();
    } else if (warp >= kFoldEpiWarp0) {
        // ---------------- epilogue: TMEM -> bias / ReLU -> y, 128 bytes of channels per pixel at a time ----------------
        // A block of rows (row r = pixel r of the tile) is staged with its 16-byte pieces swizzled by row, and stored by
        // TMA, which clips the box to the tensor.  gi groups of four warps take alternate items, gb share the column blocks
        // of one.  The block's last item, whose epilogue nothing hides, is shared by all four groups: its products are done,
        // so the input boxes' memory serves as staging for the groups that have none.
        const int lg = warp & 3, r = lg * 32 + lane, grp = (warp - kFoldEpiWarp0) >> 2;
        const bool issuer = (warp & 3) == 0 && lane == 0;
        const uint32_t bias_s = smem_u32(bias_sm);
        const uint32_t free0 = map_shared(bar_accfree, 0);
        for (int d = r + 128 * grp; d < P.nparts * P.Npart; d += 128 * kFoldEpiGroups) bias_sm[d] = d < P.D ? __ldg(P.bias + d) : 0.f;
        named_bar_sync(5, 128 * kFoldEpiGroups);
        const int blk = P.out_f32 ? 32 : 64;                 // channels per staged block
        const int gi = P.gb == 1 ? grp : (P.gb == 2 ? grp >> 1 : 0), groups = P.gi * P.gb;
        const uint32_t stage_s = grp < groups ? o_s + (uint32_t)grp * 16384u : a_s + (uint32_t)(grp - groups) * 16384u;
        const int last_it = my_items - 1;
        int it = grp < groups ? gi : last_it;
#pragma unroll 1
        while (true) {
            it = min(it, last_it);
            const bool last = it == last_it;
            const int cb0 = (last ? grp : grp & (P.gb - 1)) * blk, cb_step = (last ? kFoldEpiGroups : P.gb) * blk;
            const int item = cluster + it * nclusters;
            int tile = fold_div(item, P.dv_parts);
            const int part = item - tile * P.nparts;
            tile = 2 * tile + (int)rank;
            const int bn = fold_div(tile, P.dv_thw);
            tile -= bn * P.tiles_h * P.tiles_w;
            const int bh = fold_div(tile, P.dv_tw), bw = tile - bh * P.tiles_w;
            const int buf = it & (P.nacc - 1);
            if (lane == 0) {      // the last item waits for the end of all products: their operands' memory is used again
                if (last) fold_wait(bar_drain, 0, &abort_flag, P.status, kStatusWaitMma);
                else fold_wait(bar_accfull + 8 * buf, (uint32_t)(it >> P.nacc_shift) & 1u, &abort_flag, P.status, kStatusWaitMma);
            }
            __syncwarp();
            tc_fence_after();
            const uint32_t t_base = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)(buf * P.acc_cols);
            const int d0 = part * P.Npart;
            const int nd = min(P.Npart, P.D - d0);           // channels of this item that exist
            const uint32_t rx = (uint32_t)(r & 7) << 4;
            bool read = false;
#pragma unroll 1
            for (int cb = cb0; cb < nd; cb += cb_step) {
                const uint32_t row_s = stage_s + (uint32_t)r * 128u;
                if (issuer) bulk_wait_read_all();            // the staging buffer's last box has left it
                named_bar_sync(1 + grp, 128);
#pragma unroll 1
                for (int h = 0; h < blk && cb + h < P.Npart; h += 32) {
                    uint32_t acc[32];
                    tmem_ld32(t_base + (uint32_t)(cb + h), acc);
                    const uint32_t bias_h = bias_s + (uint32_t)(d0 + cb + h) * 4u;
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 8; ++q) {            // bias, ReLU on four channels
                        float bv[4];
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(bv[0]), "=f"(bv[1]), "=f"(bv[2]), "=f"(bv[3]) : "r"(bias_h + 16u * q));
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            float f = __uint_as_float(acc[4 * q + e]) + bv[e];
                            if (P.relu) f = fmaxf(f, 0.f);
                            acc[4 * q + e] = __float_as_uint(f);
                        }
                    }
                    if (!P.out_f32) {
                        const uint32_t c = (uint32_t)h * 2u;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            uint32_t o[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) o[e] = pack_bf16x2(__uint_as_float(acc[8 * q + 2 * e]), __uint_as_float(acc[8 * q + 2 * e + 1]));
                            sts128(row_s + ((c + 16u * q) ^ rx), make_uint4(o[0], o[1], o[2], o[3]));
                        }
                    } else {
#pragma unroll
                        for (int q = 0; q < 8; ++q) sts128(row_s + ((16u * q) ^ rx), make_uint4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]));
                    }
                }
                if (!last && cb + cb_step >= nd) {           // this group has read its columns of the accumulator
                    read = true;
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(free0 + 8 * buf);
                }
                fence_proxy_async();
                named_bar_sync(1 + grp, 128);
                if (issuer) {
                    tma_store_4d(stage_s, &P.tmap_y, d0 + cb, bw * P.PW, bh * P.PH, bn * P.TN);
                    bulk_commit();
                }
            }
            if (last) break;
            if (!read && lane == 0) mbar_arrive_cluster(free0 + 8 * buf);     // an item narrower than the group's first block
            it += P.gi;
        }
        if (issuer) bulk_wait_all();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0 && lane == 0) mbar_wait_drain(bar_drain, 0);      // bounded, ignores the abort flag
    __syncwarp();
    cluster_sync();              // nothing of this pair is in flight any more: either block may end
    __syncwarp();
    if (warp == kFoldTmemWarp) tmem_dealloc_pair(tmem, (uint32_t)(P.nacc * P.acc_cols));
}

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
namespace {

struct FoldGeom {
    int layout = 0;              // 1: boxes with halo rows (16 x 8 pixels of one image; one box per parity pair), 2: one copy per
                                 // filter row and column parity (several images per tile), 3: one copy per tap (maps at most 4 wide)
    int TN = 0, PH = 0, PW = 0, IH = 0, IW = 0, nloads = 0;
    int tiles_n = 0, tiles_h = 0, tiles_w = 0;
    int Npart = 0, nparts = 0;   // output channels per work item (a multiple of 32)
    double cycles = 0;           // estimate of the products' time on the busiest pair (picks the geometry)
    double us = 0;               // estimate of the whole launch
    int64_t pairs() const { return ((int64_t)tiles_n * tiles_h * tiles_w + 1) / 2; }
};

// Cycles of one product of M = 256, K = 16 and n output channels: the tensor pipe takes n / 2, fetching 128 rows of A and
// n / 2 rows of B per block at 128 bytes per clock 32 + n / 8.
double fold_mma_cycles(int n) { return std::max(n / 2.0, 32.0 + n / 8.0); }

// Tile shape and output-channel split with the fewest cycles on the busiest pair of blocks: whole waves of work items count.
bool fold_geometry(const gdws_plan_s *p, int n, int Ho, int Wo, bool out_f32, FoldGeom *out)
{
    const int k = p->k;
    const TcTaps t = tc_taps(k, p->stride, p->pad);
    const int nclusters = std::max(1, sm_count_of(p) / 2);
    const double ksteps = k * k * (p->C / 16.0);
    bool found = false;
    auto consider = [&](int layout, int TN, int PH, int PW) {
        FoldGeom g;
        g.layout = layout; g.TN = TN; g.PH = PH; g.PW = PW;
        g.tiles_n = (n + TN - 1) / TN; g.tiles_h = (Ho + PH - 1) / PH; g.tiles_w = (Wo + PW - 1) / PW;
        g.IW = layout == 3 ? 4 : PW + t.ext;
        g.IH = layout == 1 ? PH + t.ext : PH;
        g.nloads = layout == 1 ? t.npar * t.npar : (layout == 2 ? k * t.npar : k * k);
        // bytes of x per product step and block, at the rate the L2 delivers beside the filters
        const double a_bytes = (double)g.nloads * TN * g.IH * g.IW * 32.0 / (k * k);
        for (int parts = 1; parts <= 16; ++parts) {
            const int unit = out_f32 ? 32 : 64;          // a part holds whole staged blocks unless it is the only one
            int np = (p->D + parts - 1) / parts;
            np = (np + (parts > 1 ? unit : 32) - 1) / (parts > 1 ? unit : 32) * (parts > 1 ? unit : 32);
            if (np > 256) continue;
            g.Npart = np; g.nparts = (p->D + np - 1) / np;
            if (parts > 1 && g.nparts < parts) continue;
            const int64_t items = g.pairs() * g.nparts;
            const double waves = (double)((items + nclusters - 1) / nclusters);
            // per product: the tensor pipe, the L2, or the issuing thread (some 30 cycles each, 620 per unit of taps)
            const double issue = 30.0 + 620.0 / (4.0 * (layout == 3 ? 2 : (np > 128 ? std::min(k, 3) : k)));
            const double step = std::max(std::max(fold_mma_cycles(np), (a_bytes + np * 16.0) / 56.0), issue);
            // a wave's products, a little per item for its epilogue and hand-overs, the last epilogue in full
            g.cycles = waves * (ksteps * step + 300.0) + 1500.0 + 6.0 * np;
            if (!found || g.cycles < out->cycles) {
                // A work item takes what its slowest role takes: the products, the input boxes (cycles per staged pixel
                // measured: 2.6, of the strided views 3.6) or the epilogue (1700 + 1100 per 64 channels).
                const double boxes = p->fold_nwin * (double)g.nloads * TN * g.IH * g.IW * (p->stride == 1 ? 2.6 : 3.6);
                const double nblk = (np + 63) / 64;
                const double mma = std::max(std::max(1.08 * fold_mma_cycles(np), issue), np * 16.0 / 60.0);
                const double item = std::max(std::max(ksteps * mma, boxes), 1700.0 + 1100.0 * nblk) + 450.0;
                g.us = (2.0 + (waves * item + 4000.0 + 900.0 * std::min(nblk, 2.0)) / 1850.0) * (p->stride == 1 ? 1.0 : 1.15);      // the strided views' loads: 1.09 to 1.26
                *out = g;
                found = true;
            }
        }
    };
    if (Wo > 4) {
        consider(1, 1, 16, 8);
        for (int PH = 8; PH >= 1; PH >>= 1) consider(2, 16 / PH, PH, 8);
    } else {
        for (int PH = 32; PH >= 2; PH >>= 1) consider(3, 32 / PH, PH, 4);
    }
    return found;
}

}  // namespace

namespace {

struct FoldLaunch {
    LaunchKey key;
    FoldParams P;
    FoldGeom g;
    void (*kernel)(FoldParams) = nullptr;
    int grid = 0;
    size_t smem = 0;
    bool sliced = false;                         // runs in fold_split.cu, nothing else here is set
    const void *x = nullptr, *y = nullptr;       // the addresses the tensor maps were encoded for
};

// Everything about a launch but the addresses of x and y.
gdws_status_t fold_prepare(gdws_plan_s *p, int n, int Ho, int Wo, bool out_f32, FoldLaunch *L)
{
    const int k = p->k, sd = p->stride;
    FoldGeom &g = L->g;
    if (!fold_geometry(p, n, Ho, Wo, out_f32, &g)) return fail(GDWS_ERR_UNSUPPORTED, "folded path: no tile");
    const int64_t nitems = g.pairs() * g.nparts;
    if (nitems > 0x3fffffffLL) return fail(GDWS_ERR_UNSUPPORTED, "too many tiles");
    const int nclusters = (int)std::min<int64_t>(nitems, std::max(1, sm_count_of(p) / 2));
    FoldParams &P = L->P;
    memset(&P, 0, sizeof(P));
    P.nwin = p->fold_nwin; P.nk_last = (p->C - (p->fold_nwin - 1) * 64 + 15) / 16; P.nsteps = k * k;
    P.D = p->D; P.Dp = p->fold_dp; P.Npart = g.Npart; P.nparts = g.nparts;
    P.relu = p->opt_relu; P.out_f32 = out_f32 ? 1 : 0;
    P.TN = g.TN; P.PH = g.PH; P.PW = g.PW; P.tiles_h = g.tiles_h; P.tiles_w = g.tiles_w; P.nitems = (int)nitems;
    P.bias = p->d_bias; P.status = p->d_status; P.sums = p->d_fold_sums; P.nsums = p->fold_nsums;
    P.a_bytes = (uint32_t)(g.TN * g.IH * g.IW * 128);
    P.a_load = (P.a_bytes + 1023u) / 1024u * 1024u;
    P.a_sbo = g.layout == 3 ? 1024u : (uint32_t)g.IW * 128u;
    P.b_tap = (uint32_t)g.Npart / 2u * 128u;
    P.acc_cols = 32;
    while (P.acc_cols < g.Npart) P.acc_cols <<= 1;
    // As many accumulators as fit the 512 columns: with narrow items the way from a tile's last product through the epilogue
    // back to the issuing thread takes as long as two tiles' products.
    P.nacc = std::min(kFoldMaxAcc, 512 / P.acc_cols);
    while ((1 << P.nacc_shift) < P.nacc) ++P.nacc_shift;
    // Input boxes and product steps; run[s]: how many steps, from s on, read the same box (0 inside a run).  A box is one load;
    // with one load per tap two of them, so that the taps can share a unit, and with stride 2 the loads of both column
    // parities: filter rows are then whole (k taps each, the unrolled kernels) where they would be 1, 2, 2 and 4 taps.
    const int per_box = g.layout == 3 || sd == 2 ? 2 : 1;
    P.a_slot = P.a_load * (uint32_t)per_box;
    const TcTaps taps = tc_taps(k, sd, p->pad);
    int nl = 0, ns = 0, run[kFoldMaxSteps] = {}, run0 = 0;
    auto add_load = [&](int hp, int wp, int dh, int dw) {
        P.load_map[nl] = hp * 2 + wp; P.load_dh[nl] = dh; P.load_dw[nl] = dw;
        P.maps_used |= 1 << (hp * 2 + wp);
        if (nl % per_box == 0) { run0 = ns; P.boxes[P.nboxes++] = (uint32_t)nl; }
        P.boxes[P.nboxes - 1] += 1u << 8;
        ++nl;
    };
    auto add_step = [&](int u, int v, int row, int col) {
        // 128 bytes per staged pixel
        P.steps[ns++] = ((uint32_t)(row * g.IW + col) * 8u + (P.a_load >> 4) * (uint32_t)((nl - 1) % per_box)) | (uint32_t)(u * k + v) << 16;
        ++run[run0];
    };
    for (int hp = 0; hp < sd && g.layout == 1; ++hp)
        for (int wp = 0; wp < sd; ++wp) {
            if (!taps.used[hp] || !taps.used[wp]) continue;
            add_load(hp, wp, taps.omin[hp], taps.omin[wp]);
            for (int u = 0; u < k; ++u)
                for (int v = 0; v < k; ++v)
                    if (taps.par[u] == hp && taps.par[v] == wp) add_step(u, v, taps.off[u] - taps.omin[hp], taps.off[v] - taps.omin[wp]);
        }
    for (int u = 0; u < k && g.layout == 2; ++u)
        for (int wp = 0; wp < sd; ++wp) {
            if (!taps.used[wp]) continue;
            add_load(taps.par[u], wp, taps.off[u], taps.omin[wp]);
            for (int v = 0; v < k; ++v)
                if (taps.par[v] == wp) add_step(u, v, 0, taps.off[v] - taps.omin[wp]);
        }
    for (int u = 0; u < k && g.layout == 3; ++u)
        for (int v = 0; v < k; ++v) {
            add_load(taps.par[u], taps.par[v], taps.off[u], taps.off[v]);
            add_step(u, v, 0, 0);
        }
    if (nl != g.nloads || ns != k * k) return fail(GDWS_ERR_UNSUPPORTED, "folded path: internal error in the box plan");
    // Units: what the issuing thread does around a unit's products takes some 700 cycles, a step's four products of 256 output
    // channels 520, of 64 180: a filter row's taps share one barrier (three of them at most where a unit is large).
    const int per_unit = g.layout == 3 ? 2 : (g.Npart > 128 ? std::min(k, 3) : k);
    int unit_steps = 0;
    for (int s0 = 0; s0 < ns; s0 += run[s0])
        for (int j = 0; j < run[s0]; j += per_unit) {
            const int n = std::min(per_unit, run[s0] - j);
            P.units[P.nunits++] = (uint32_t)(s0 + j) | (uint32_t)n << 8 | (j == 0 ? kUnitFirst : 0u) | (j + n == run[s0] ? kUnitLast : 0u) |
                                   (j == 0 && s0 + run[s0] == ns ? kUnitLastBox : 0u);
            unit_steps = std::max(unit_steps, n);
        }
    bool alike = true;
    for (int u = 0; u < P.nunits; ++u) alike = alike && (int)((P.units[u] >> 8) & 0xFFu) == unit_steps;
    P.b_unit = P.b_tap * (uint32_t)unit_steps;
    // Shared memory: output staging | input boxes | filters | bias.  All of a block's filters stay resident if they fit
    // beside two input boxes (three where a window takes several) and it keeps to one block of output channels.
    const size_t bias_bytes = (size_t)g.nparts * g.Npart * 4;
    const int units = P.nwin * P.nunits;
    // Epilogue groups with staging of their own: a tile's way through the epilogue takes some 1400 cycles per column block
    // (128 bytes of channels per pixel); as many groups as keep it below the tile's products, the remaining shared memory
    // goes to filters and boxes.
    const int nblk = (g.Npart + (out_f32 ? 31 : 63)) / (out_f32 ? 32 : 64);
    bool placed = false;
    auto place = [&](bool res, int groups, int na_min, int na_max, int nb_min) {
        const size_t fixed = 1024 + (size_t)groups * 16384 + bias_bytes;
        const size_t b_min = (size_t)(res ? units : nb_min) * P.b_unit;
        for (int na = na_max; na >= na_min; --na) {
            if (fixed + b_min + (size_t)na * P.a_slot > (size_t)kFoldMaxSmem) continue;
            P.resident = res; P.na = na;
            P.nb = res ? units : (int)std::min<size_t>(16, ((size_t)kFoldMaxSmem - fixed - (size_t)na * P.a_slot) / P.b_unit);
            if (!res && P.nb > 4) P.nb &= ~1;      // an even ring is filled by two warps
            P.gb = nblk == 1 || groups == 1 ? 1 : (groups == 4 && nblk > 2 ? 4 : 2);
            P.gi = groups / P.gb;
            return true;
        }
        return false;
    };
    const bool can_stay = units >= 2 && units <= kFoldMaxB && (g.nparts == 1 || nitems <= nclusters);
    const bool several = P.nboxes > 1;       // boxes per window: more in flight to cover their latency
    const double products = k * k * (p->C / 16.0) * fold_mma_cycles(g.Npart), epilogue = 1400.0 * nblk;
    // Filters that stay leave memory for staging: four groups where an item's epilogue is not well below its products
    // (64 -> 64 channels at 32 x 32: 53 us with two groups, 38 with four).  A ring of filters needs it more.
    const int stay_groups = epilogue > 0.75 * products ? 4 : (epilogue > 0.35 * products ? 2 : 1);
    const int groups = epilogue > 1.4 * products ? 4 : (epilogue > 0.8 * products ? 2 : 1);
    for (int gr = stay_groups; can_stay && gr >= 1 && !placed; gr >>= 1) placed = place(true, gr, several ? (gr == 4 ? 4 : 3) : (gr == 4 ? 3 : 2), kFoldMaxA, 0);
    // ring: three units of filters (one being read, two on their way), then boxes, then more of both
    if (!placed) placed = place(false, groups, several ? 4 : 3, several ? 4 : 3, 4) || place(false, groups, 3, 3, 3) || place(false, std::min(groups, 2), 2, 3, 3) || place(false, 1, 2, 3, 3) ||
                          place(false, 1, 2, 3, 2);
    if (!placed) return fail(GDWS_ERR_UNSUPPORTED, "folded path: shared memory does not fit this layer");
    // the last item's epilogue stages in the memory of the boxes and filters
    if ((size_t)P.na * P.a_slot + (size_t)P.nb * P.b_unit < (size_t)(kFoldEpiGroups - P.gi * P.gb) * 16384)
        return fail(GDWS_ERR_UNSUPPORTED, "folded path: no room for the epilogue's staging");
    const uint32_t item_boxes = (uint32_t)(P.nwin * P.nboxes);
    // Items of one box: a second issuing warp fills the gaps that a warp leaves between its items.  (Of several: two items in
    // progress at once hold their boxes twice as long, which costs more than the gaps.)
    P.mma_warps = item_boxes == 1 ? 2 : 1;
    P.a_skip = item_boxes % (uint32_t)P.na; P.a_flip = (item_boxes / (uint32_t)P.na) & 1u;
    P.b_skip = (uint32_t)units % (uint32_t)P.nb; P.b_flip = ((uint32_t)units / (uint32_t)P.nb) & 1u;
    P.off_a = (uint32_t)(P.gi * P.gb) * 16384u;
    P.off_b = P.off_a + (uint32_t)P.na * P.a_slot;
    P.off_bias = P.off_b + (uint32_t)P.nb * P.b_unit;
    size_t smem = 1024 + (size_t)P.off_bias + bias_bytes;
    if (smem < (size_t)kFoldMaxSmem / 2 + 4096) smem = (size_t)kFoldMaxSmem / 2 + 4096;     // one block per SM: tensor memory is never oversubscribed

    div_magic(g.nparts, P.dv_parts); div_magic(g.tiles_h * g.tiles_w, P.dv_thw); div_magic(g.tiles_w, P.dv_tw);

    void (*kernel)(FoldParams) = nullptr;
    int which = 0;
    const int nk = P.nwin == 1 ? P.nk_last : 4;
    if (alike && unit_steps == 3 && P.nunits == 3) {
        kernel = nk == 1 ? fold_kernel<3, 3, 1> : (nk == 2 ? fold_kernel<3, 3, 2> : (nk == 3 ? fold_kernel<3, 3, 3> : fold_kernel<3, 3>));
        which = nk == 4 ? 0 : 3 + nk;
    }
    else if (alike && unit_steps == 5 && P.nunits == 5) {
        kernel = nk == 1 ? fold_kernel<5, 5, 1> : (nk == 2 ? fold_kernel<5, 5, 2> : (nk == 3 ? fold_kernel<5, 5, 3> : fold_kernel<5, 5>));
        which = nk == 4 ? 1 : 6 + nk;
    }
    else if (alike && unit_steps == 1) { kernel = fold_kernel<0, 1>; which = 2; }
    else { kernel = fold_kernel<0, 0>; which = 3; }
    static bool attr_set[64][10] = {};
    if (!attr_set[p->device & 63][which]) {
        cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFoldMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(fold_kernel)");
        attr_set[p->device & 63][which] = true;
    }
    tensor_map_encode_fn encode = encode_fn();
    if (!encode) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from this driver");
    const cuuint64_t dims[2] = {64, (cuuint64_t)2 * P.nwin * P.nsteps * p->fold_dp};
    const cuuint64_t strides[1] = {128};
    const cuuint32_t box[2] = {64, (cuuint32_t)g.Npart / 2}, estr[2] = {1, 1};
    const CUresult r = encode(&P.tmap_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p->d_fold, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (filters) failed with code %d", (int)r);
    L->kernel = kernel; L->grid = 2 * nclusters; L->smem = smem;
    return GDWS_OK;
}

// x as a rank-4 tensor, innermost first: channels, width, height, batch; with stride 2 one view per parity of row and column.
gdws_status_t fold_map_x(const gdws_plan_s *p, const gdws_tensor_t *x, FoldLaunch *L)
{
    tensor_map_encode_fn encode = encode_fn();
    const int sd = p->stride;
    L->x = nullptr;              // until all of them are of this address
    for (int m = 0; m < 4; ++m) {
        if (!((L->P.maps_used >> m) & 1)) continue;
        const int hp = m >> 1, wp = m & 1;
        const int Wp = (x->w - wp + sd - 1) / sd, Hp = (x->h - hp + sd - 1) / sd;
        if (Wp <= 0 || Hp <= 0) return fail(GDWS_ERR_UNSUPPORTED, "folded path: input too small for stride %d", sd);
        const cuuint64_t dims[4] = {(cuuint64_t)p->C, (cuuint64_t)Wp, (cuuint64_t)Hp, (cuuint64_t)x->n};
        const cuuint64_t strides[3] = {(cuuint64_t)sd * p->C * 2, (cuuint64_t)sd * x->w * p->C * 2, (cuuint64_t)x->h * x->w * p->C * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)L->g.IW, (cuuint32_t)L->g.IH, (cuuint32_t)L->g.TN}, estr[4] = {1, 1, 1, 1};
        void *base = (uint8_t *)x->ptr + ((size_t)hp * x->w + wp) * p->C * 2;
        const CUresult r = encode(&L->P.tmap_x[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (x) failed with code %d", (int)r);
    }
    L->x = x->ptr;
    return GDWS_OK;
}

gdws_status_t fold_map_y(const gdws_plan_s *p, const gdws_tensor_t *y, FoldLaunch *L)
{
    const bool out_f32 = y->dtype == GDWS_F32;
    const cuuint64_t es = out_f32 ? 4 : 2;
    const cuuint64_t dims[4] = {(cuuint64_t)p->D, (cuuint64_t)y->w, (cuuint64_t)y->h, (cuuint64_t)y->n};
    const cuuint64_t strides[3] = {p->D * es, (cuuint64_t)y->w * p->D * es, (cuuint64_t)y->h * y->w * p->D * es};
    const cuuint32_t box[4] = {(cuuint32_t)(128 / es), (cuuint32_t)L->g.PW, (cuuint32_t)L->g.PH, (cuuint32_t)L->g.TN}, estr[4] = {1, 1, 1, 1};
    const CUresult r = encode_fn()(&L->P.tmap_y, out_f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, y->ptr, dims, strides,
                                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                   CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (y) failed with code %d", (int)r);
    L->y = y->ptr;
    return GDWS_OK;
}

}  // namespace

// ------------------------------------------------------------------------------------------
// Which form a bf16 layer takes.  The folded form costs C k^2 D multiply-adds per pixel at full tensor-core rate, the
// two-stage forms G (k^2 + D) at what their hand-overs allow.  The constants are fits to timings on B200.  On 200 random layers
// (k = 3 and 5, strides 1 and 2, half of them maps below 10 x 10) the chosen form is 2.9 % slower than the fastest in the mean,
// mostly calls of 5 to 10 us where the three are close; against the two stages alone the choice loses on two of them, 4 and 6 %.
// ------------------------------------------------------------------------------------------
namespace {

double two_stage_us(const gdws_plan_s *p, int n, int h, int w, int Ho, int Wo, int stage)
{
    const double sms = sm_count_of(p);
    auto waves = [&](double items) { return std::ceil(items / sms); };
    if (stage == 1) {
        Tile t;
        if (p->D > 512 || !choose_tile(p, n, h, w, &t)) return 1e9;
        // with stride 2 a chunk's time follows the pixels that a tile has (0.6 to 0.85 us with a few, 1.3 with all; k = 5: 1.2 to 1.9)
        const double fill = std::min(1.0, (double)n * Ho * Wo / (128.0 * (double)t.tiles()));
        const double chunk = (p->stride == 1 ? 0.95 * (p->k == 3 ? 1.0 : 2.1) : 1.25 * (p->k == 3 ? 1.0 : 1.35) * (0.6 + 0.4 * fill)) *
                             (p->D > 256 ? 1.3 : (p->D > 128 ? 1.12 : 1.0));
        return (p->stride == 1 ? 0.9 : 1.0) * (3.5 + waves((double)t.tiles()) * (p->nchunks * chunk + 0.5) + p->D / 128.0);
    }
    double tiles = 1e18;
    auto shape = [&](int TN, int PH, int PW) {
        tiles = std::min(tiles, std::ceil((double)n / TN) * std::ceil((double)Ho / PH) * std::ceil((double)Wo / PW));
    };
    if (Wo > 4) {
        shape(1, 16, 8);
        for (int PH = 8; PH >= 1; PH >>= 1) shape(16 / PH, PH, 8);
    } else {
        for (int PH = 32; PH >= 2; PH >>= 1) shape(32 / PH, PH, 4);
    }
    const double chunks = (double)p->tc_chunks.size() * (p->k == 3 ? 0.72 : 1.2) + p->tc_nslabs * 0.012 * p->tc_dloc / 64.0 + 0.4;
    return (p->stride == 1 ? 0.93 : 1.25) * (4.0 + waves(tiles * p->tc_nparts) * chunks);
}

struct FormChoice {
    LaunchKey key;
    int form = 1;
    bool sliced = false;         // the folded form would run in slices
};

}  // namespace

int bf16_form_of(gdws_plan_s *p, int n, int h, int w, bool out_f32)
{
    const int stage = gdw_stage_of(p);
    if (p->opt_dw_math) return p->opt_dw_math;
    // one row or column and stride 2: the view of the odd ones is empty, and the kernels that read it refuse the input
    if (p->stride == 2 && p->k <= 5 && (h < 2 || w < 2) && tc_taps(p->k, 2, p->pad).used[1]) return 1;
    if (!p->fold_ok || p->opt_tile || p->opt_a_layout) return stage;
    // A channel with g_c = 0 is not part of the layer: the folded form would multiply it by zero filters, and an infinity or
    // NaN in it would reach y.  (Beyond 512 output channels there is no ALU kernel to keep to.)
    if (p->unused && !(stage == 1 && p->Dpad > 512)) return stage;
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    if (n < 1 || Ho < 1 || Wo < 1) return stage;
    const LaunchKey key = {n, h, w, out_f32 ? 2 : 0};
    if (const FormChoice *c = LaunchCache<FormChoice>::find(p->launch_cache[kCacheForm], key)) return c->form;
    FoldGeom g;
    double us = fold_geometry(p, n, Ho, Wo, out_f32, &g) ? g.us : 1e9;
    const double slices = fold_split_us(p, n, Ho, Wo);
    const bool sliced = slices < us;
    // Slices (fold_split.cu) count where a channel has more than two filters in the mean: the estimates were compared with timings there.
    // Below it the choice is the one without them, and a layer that they would win keeps the two stages (384 -> 104 channels, stride 2,
    // 8 x 8, g_c = 2: 12.5 us, in slices 7.3).
    if (p->G > 2 * p->C) us = std::min(us, slices);
    const bool fold = us < two_stage_us(p, n, h, w, Ho, Wo, stage);
    const int form = fold ? 3 : stage;
    if (std::unique_ptr<FormChoice> c{new (std::nothrow) FormChoice}) {
        c->key = key;
        c->form = form;
        c->sliced = sliced;
        LaunchCache<FormChoice>::add(p->launch_cache[kCacheForm], std::move(c));      // kept if there is memory for it
    }
    return form;
}

// Estimate of a bf16 forward of n images, for gdws_forward_host: the form's own, with the generic depthwise code of the ALU
// kernel at 0.55 us per tap and chunk of 64 (measured 0.3 to 0.8).
double bf16_forward_us(gdws_plan_s *p, int n, int h, int w, bool out_f32)
{
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    const int form = p->opt_path == GDWS_PATH_UNFUSED ? 1 : bf16_form_of(p, n, h, w, out_f32);
    if (form == 3) {                     // either kernel may be the only one that covers the layer
        FoldGeom g;
        const double us = std::min(fold_geometry(p, n, Ho, Wo, out_f32, &g) ? g.us : 1e9, fold_split_us(p, n, Ho, Wo));
        if (us < 1e9) return us;
    }
    if (form == 2) return two_stage_us(p, n, h, w, Ho, Wo, 2);
    Tile t;
    if (!choose_tile(p, n, h, w, &t)) return 1e9;
    if (t.fast) return two_stage_us(p, n, h, w, Ho, Wo, 1);
    return 4.0 + std::ceil((double)t.tiles() / sm_count_of(p)) * p->nchunks * 0.55 * p->k * p->k;
}

bool fold_in_slices(gdws_plan_s *p, int n, int h, int w, bool out_f32)
{
    if (const FormChoice *c = LaunchCache<FormChoice>::find(p->launch_cache[kCacheForm], {n, h, w, out_f32 ? 2 : 0})) return c->sliced;
    const int Ho = gdws_out_dim(h, p->k, p->stride, p->pad), Wo = gdws_out_dim(w, p->k, p->stride, p->pad);
    FoldGeom g;
    return !(fold_geometry(p, n, Ho, Wo, out_f32, &g) && g.us <= fold_split_us(p, n, Ho, Wo));
}

gdws_status_t bf16_folded(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, bool given, cudaStream_t st)
{
    if (!p->fold_ok) return fail(GDWS_ERR_UNSUPPORTED, "folded path: layer not covered (stride 1 or 2, k <= 5, C and D multiples of 8)");
    const bool out_f32 = y->dtype == GDWS_F32;
    const LaunchKey key = {x->n, x->h, x->w, (p->opt_relu ? 1 : 0) | (out_f32 ? 2 : 0)};
    gdws_status_t rc;
    FoldLaunch *L = LaunchCache<FoldLaunch>::find(p->launch_cache[kCacheFold], key);
    if (!L) {
        std::unique_ptr<FoldLaunch> e(new (std::nothrow) FoldLaunch);
        if (!e) return fail(GDWS_ERR_ALLOC, "out of host memory");
        e->key = key;
        e->sliced = fold_in_slices(p, x->n, x->h, x->w, out_f32);
        rc = e->sliced ? GDWS_OK : fold_prepare(p, x->n, y->h, y->w, out_f32, e.get());
        if (rc != GDWS_OK) return rc;
        L = LaunchCache<FoldLaunch>::add(p->launch_cache[kCacheFold], std::move(e));
        if (!L) return fail(GDWS_ERR_ALLOC, "out of host memory");
    }
    if (L->sliced) {
        rc = bf16_folded_split(p, x, y, given, st);
        if (rc == GDWS_OK) return rc;
        // refused: pairs cover all but layers of very many output channels
        if (fold_prepare(p, x->n, y->h, y->w, out_f32, L) != GDWS_OK) return rc;
        L->sliced = false;
    }
    if (L->x != x->ptr && (rc = fold_map_x(p, x, L)) != GDWS_OK) return rc;
    if (L->y != y->ptr && (rc = fold_map_y(p, y, L)) != GDWS_OK) return rc;
    const cudaError_t e = launch_overlapped(L->kernel, (unsigned)L->grid, kFoldThreads, L->smem, st, L->P);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "fold_kernel launch"); }
    p->launches++;
    return GDWS_OK;
}

}  // namespace gdws
