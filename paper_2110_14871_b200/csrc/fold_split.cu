// The folded form (csrc/fold.cu) for layers that leave most of the chip idle: the k x k convolution's sum over channels and filter
// rows is cut into up to eight slices, one per block of a cluster.
//
// What bounds such a layer is a chain, not a rate: on pairs of SMs 256 -> 256 channels at 14 x 14 are 144 K steps of some 50 cycles,
// one after the other in each of 4 pairs (140 SMs idle), after launch, prologue and the first loads.  Here a unit of work is one
// filter row of a window of 64 input channels (k taps); a block takes 1 to a few units of a tile of 128 pixels x up to 256 output
// channels, asks for all their operands at once where they fit, and adds them up in tensor memory.  The blocks of a cluster then put
// their sums into shared memory, and each finishes a share of the output channels (bias, ReLU, y) from all of them, read through
// distributed shared memory in the order of the slices.
// Measured, pairs of SMs | slices: 1 x 256 -> 256 x 14 x 14 9.4 | 6.9 us, 1 x 512 -> 512 x 7 x 7 14.0 | 8.0, 4 x 512 -> 512 x 4 x 4 26.7 |
// 8.3, 1 x 64 -> 64 x 56 x 56 (one slice: the shorter way through prologue and epilogue) 6.4 | 4.9, 43 x 48 -> 280 x 16 x 18, 5 x 5 taps,
// stride 2 23.8 (two stages) | 9.5.
// One block per product (M = 128): these layers are not bound by the tensor pipe, and pairs would double the smallest item.
#include <string.h>

#include <algorithm>
#include <mutex>
#include <new>

#include "sm100.cuh"

namespace gdws {

constexpr int kSplitThreads = 8 * 32, kSplitMmaWarp = 0, kSplitAWarp = 1, kSplitBWarp = 2, kSplitTermWarp = 3;
constexpr int kSplitMaxSlots = 8, kSplitMaxSteps = 25;
constexpr uint32_t kSplitSw128 = 2u << 29;   // descriptor high word: layout type "128-byte swizzle"

struct alignas(64) FoldSplitParams {
    CUtensorMap tmap_x[4];       // x as (C, W, H, N), box (64, IW, PH, TN); stride 2: one dense view per parity
    CUtensorMap tmap_w;          // folded filters as rows of 64 input channels, box (64, Npart)
    const float *bias;
    const float2 *sums;          // of the packing blocks, for the filters' second term
    void *y;
    int *status;
    int nsums, k, nwin, nk_last, nl, Dp, D, Npart, nparts, relu, out_f32;
    int N, Ho, Wo, TN, PH, PW, tiles_h, tiles_w, units, split, na, acc_cols, maps_used;
    uint32_t a_sbo, a_bytes, a_load, b_tap, b_off, slot;         // a slot: nl boxes, then k taps of filters from b_off on
    uint32_t step[kSplitMaxSteps];                               // per tap: its operand's offset in the slot / 16
    int load_map[kSplitMaxSteps], load_dw[kSplitMaxSteps], load_dh[kSplitMaxSteps];      // per filter row, nl each
};

// The products of a filter row over 64 input channels, straight-line.
template <int TAPS>
__device__ __forceinline__ void split_issue(const uint32_t *step, uint32_t d, uint32_t lo, uint32_t a_hi, uint32_t bl, uint32_t b_hi, uint32_t b_tap, uint32_t idesc, uint32_t more)
{
#pragma unroll
    for (int v = 0; v < TAPS; ++v)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) umma_bf16_words(d, lo + step[v] + 2u * kk, a_hi, bl + (uint32_t)v * b_tap + 2u * kk, b_hi, idesc, v | kk ? 1u : more);
}

__global__ void __launch_bounds__(kSplitThreads, 1) fold_split_kernel(const __grid_constant__ FoldSplitParams P)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kSplitMaxSlots + 2];       // full[8] empty[8] | all products done | terms known
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_flag, second_term;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    volatile int *const vabort = &abort_flag;
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t s_s = smem_u32(base);
    const uint32_t bar_full = smem_u32(&bars[0]), bar_empty = bar_full + 8 * kSplitMaxSlots, bar_done = bar_empty + 8 * kSplitMaxSlots, bar_terms = bar_done + 8;
    if (tid == 0) abort_flag = second_term = 0;
    if (tid < 2 * kSplitMaxSlots + 2) {
        mbar_init(bar_full + 8 * (uint32_t)tid, 1);
        fence_mbar_init();
    }
    grid_launch_dependents();
    if (warp == kSplitAWarp && lane < 4 && ((P.maps_used >> lane) & 1)) prefetch_tensor_map(&P.tmap_x[lane]);
    if (warp == kSplitBWarp && lane == 0) prefetch_tensor_map(&P.tmap_w);
    if (warp == kSplitTermWarp) tmem_alloc(smem_u32(&tmem_slot), (uint32_t)P.acc_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    grid_dependency_wait();
    const uint32_t tmem = tmem_slot;
    const int group = (int)blockIdx.x / P.split, rank = (int)blockIdx.x - group * P.split;      // a cluster's blocks are neighbours
    int tile = group / P.nparts;
    const int d0 = (group - tile * P.nparts) * P.Npart;
    const int bn = tile / (P.tiles_h * P.tiles_w);
    tile -= bn * P.tiles_h * P.tiles_w;
    const int bh = tile / P.tiles_w, bw = tile - bh * P.tiles_w;
    const int u0 = rank * P.units / P.split, u1 = (rank + 1) * P.units / P.split;
    auto terms = [&]() -> int {          // passes over the units: a second one for the filters' second term
        mbar_wait_call(bar_terms, 0, &abort_flag, P.status, kStatusWaitOperand);
        return 1 + *(volatile int *)&second_term;
    };

    if (warp == kSplitMmaWarp) {
        if (elect_one()) {
            const uint32_t idesc = make_idesc(P.Npart, false);
            const uint32_t a_hi = ((P.a_sbo >> 4) & 0x3FFFu) | (1u << 14) | kSplitSw128, b_hi = (1024u >> 4) | (1u << 14) | kSplitSw128;
            uint32_t slot = 0, par = 0, more = 0;
            int nt = 1;
#pragma unroll 1
            for (int t = 0; t < nt; ++t) {
#pragma unroll 1
                for (int u = u0; u < u1; ++u) {
                    const int w = u / P.k, row = u - w * P.k, nk = w == P.nwin - 1 ? P.nk_last : 4;
                    mbar_wait_call(bar_full + 8 * slot, par, &abort_flag, P.status, kStatusWaitOperand);
                    tc_fence_after();
                    const uint32_t lo = (((s_s + slot * P.slot) & 0x3FFFFu) >> 4) | (1u << 16);
                    uint32_t bl = lo + (P.b_off >> 4);
                    const uint32_t *step = P.step + row * P.k;
                    if (nk == 4 && P.k == 3) split_issue<3>(step, tmem, lo, a_hi, bl, b_hi, P.b_tap >> 4, idesc, more), more = 1;
                    else if (nk == 4 && P.k == 5) split_issue<5>(step, tmem, lo, a_hi, bl, b_hi, P.b_tap >> 4, idesc, more), more = 1;
                    else
#pragma unroll 1
                    for (int v = 0; v < P.k; ++v, bl += P.b_tap >> 4) {
                        const uint32_t al = lo + step[v];
                        umma_bf16_words(tmem, al, a_hi, bl, b_hi, idesc, more);
                        more = 1;
                        if (nk > 1) umma_bf16_words(tmem, al + 2u, a_hi, bl + 2u, b_hi, idesc, 1u);
                        if (nk > 2) umma_bf16_words(tmem, al + 4u, a_hi, bl + 4u, b_hi, idesc, 1u);
                        if (nk > 3) umma_bf16_words(tmem, al + 6u, a_hi, bl + 6u, b_hi, idesc, 1u);
                    }
                    umma_commit(bar_empty + 8 * slot);
                    if (++slot == (uint32_t)P.na) { slot = 0; par ^= 1u; }
                }
                if (t == 0) nt = terms();
            }
            umma_commit(bar_done);
        }
        __syncwarp();
    } else if (warp == kSplitAWarp || warp == kSplitBWarp) {
        if (lane == 0) {
            // One thread asks for the input boxes, one for the filters; the first announces the bytes of both.
            const bool boxes = warp == kSplitAWarp;
            uint32_t slot = 0, par = 1;
            int nt = 1, n = 0;
            bool stop = false;
#pragma unroll 1
            for (int t = 0; t < nt && !stop; ++t) {
#pragma unroll 1
                for (int u = u0; u < u1; ++u, ++n) {
                    const int w = u / P.k, row = u - w * P.k;
                    mbar_wait_call(bar_empty + 8 * slot, par, &abort_flag, P.status, kStatusWaitStage);
                    if (*vabort) { stop = true; break; }
                    const uint32_t dst = s_s + slot * P.slot, bar = bar_full + 8 * slot;
                    if (boxes) {
                        mbar_expect_tx(bar, (uint32_t)P.nl * P.a_bytes + (uint32_t)P.k * P.b_tap);
#pragma unroll 1
                        for (int j = 0, l = row * P.nl; j < P.nl; ++j, ++l)
                            tma_load_4d(dst + (uint32_t)j * P.a_load, &P.tmap_x[P.load_map[l]], w * 64, bw * P.PW + P.load_dw[l], bh * P.PH + P.load_dh[l], bn * P.TN, bar);
                    } else {
                        const int r0 = ((t * P.nwin + w) * P.k + row) * P.k * P.Dp + d0;
#pragma unroll 1
                        for (int v = 0; v < P.k; ++v) tma_load_2d(dst + P.b_off + (uint32_t)v * P.b_tap, &P.tmap_w, 0, r0 + v * P.Dp, bar);
                    }
                    if (++slot == (uint32_t)P.na) { slot = 0; par ^= 1u; }
                }
                if (t == 0) nt = terms();
            }
            // Teardown: the last phase armed on each slot completes when its copies have landed.
            if (boxes)
                for (int i = 0, j = n - 1; i < P.na && j >= 0; ++i, --j) mbar_wait_drain(bar_full + 8 * (j % P.na), (uint32_t)(j / P.na) & 1u);
        }
        __syncwarp();
    } else if (warp == kSplitTermWarp) {
        const bool second = fold_second_term(P.sums, P.nsums, lane);
        if (lane == 0) {
            second_term = second;
            mbar_arrive(bar_terms);
        }
        __syncwarp();
    }

    // ---------------- epilogue, all warps: a lane quarter of tensor memory and every other 16 columns each ----------------
    const int lg = warp & 3, r = lg * 32 + lane;
    if (lane == 0) mbar_wait_call(bar_done, 0, &abort_flag, P.status, kStatusWaitMma);
    __syncwarp();
    tc_fence_after();
    auto pixel = [&](int px, size_t *at) {       // the element of y where a pixel's channels begin; false: outside
        const int ppi = P.PH * P.PW, nl = px / ppi, ph = (px - nl * ppi) / P.PW, pw = px - nl * ppi - ph * P.PW;
        const int n = bn * P.TN + nl, ho = bh * P.PH + ph, wo = bw * P.PW + pw;
        *at = (((size_t)n * P.Ho + ho) * P.Wo + wo) * P.D;
        return n < P.N && ho < P.Ho && wo < P.Wo;
    };
    const uint32_t t_base = tmem + ((uint32_t)(lg * 32) << 16);
    if (P.split == 1) {
        size_t at;
        const bool live = pixel(r, &at);
        for (int c = (warp >> 2) * 16; c < P.Npart; c += 32) {
            uint32_t acc[16];
            tmem_ld16(t_base + (uint32_t)c, acc);
            tmem_ld_wait();
            if (live && d0 + c < P.D) store_row16(acc, P.bias, d0 + c, P.D, (P.relu ? kOutRelu : 0) | (P.out_f32 ? kOutF32 : 0), P.y, at);
        }
    } else {
        // [column][pixel] sums; the operands' memory is free: every copy has landed and every product is done
        __syncthreads();
        float *part = reinterpret_cast<float *>(base);
        for (int c = (warp >> 2) * 16; c < P.Npart; c += 32) {
            uint32_t acc[16];
            tmem_ld16(t_base + (uint32_t)c, acc);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 16; ++e) part[(c + e) * 128 + r] = __uint_as_float(acc[e]);
        }
        cluster_sync();
        const int px = tid & 127;
        size_t at;
        const bool live = pixel(px, &at);
        // 8 output channels of a pixel per thread and step
        for (int g = rank + P.split * (tid >> 7); live && g < P.Npart / 8 && d0 + 8 * g < P.D; g += 2 * P.split) {
            float v[8] = {};
#pragma unroll 1
            for (int o0 = 0; o0 < P.split; o0 += 4) {            // four slices' reads in flight at a time
                float w[4][8];
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                    if (o0 + o >= P.split) break;
                    const uint32_t src = map_shared(s_s + (uint32_t)(8 * g * 128 + px) * 4u, (uint32_t)(o0 + o));
#pragma unroll
                    for (int e = 0; e < 8; ++e) asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(w[o][e]) : "r"(src + (uint32_t)e * 512u));
                }
#pragma unroll
                for (int o = 0; o < 4; ++o)
#pragma unroll
                    for (int e = 0; e < 8; ++e)
                        if (o0 + o < P.split) v[e] += w[o][e];
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                v[e] += __ldg(P.bias + d0 + 8 * g + e);
                if (P.relu) v[e] = fmaxf(v[e], 0.f);
            }
            if (P.out_f32) {
                float4 *dst = reinterpret_cast<float4 *>((float *)P.y + at + d0 + 8 * g);
                dst[0] = make_float4(v[0], v[1], v[2], v[3]);
                dst[1] = make_float4(v[4], v[5], v[6], v[7]);
            } else {
                *reinterpret_cast<uint4 *>((uint16_t *)P.y + at + d0 + 8 * g) =
                    make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
            }
        }
        cluster_sync();          // every block's sums have been read
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kSplitTermWarp) tmem_dealloc(tmem, (uint32_t)P.acc_cols);
}

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
// Clusters of 1 to 8 blocks, one block per SM, that a device runs at the same time: clusters do not cross the chip's groups of SMs, so
// some SMs are left over.  `device` is the current one; it is asked once.
void cluster_capacities(int device, int sms, int (&most)[kMostSlices + 1])
{
    static std::mutex lock;
    static struct { bool known; int most[kMostSlices + 1]; } kept[64];
    std::lock_guard<std::mutex> hold(lock);
    auto &k = kept[device & 63];
    if (!k.known || device > 63) {
        k.known = true;
        k.most[1] = sms;
        cudaFuncSetAttribute(fold_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        for (int split = 2; split <= kMostSlices; ++split) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3((unsigned)(split * 64)); cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = kMaxSmem / 2 + 2048;
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = (unsigned)split; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr; cfg.numAttrs = 1;
            int got = 0;
            if (cudaOccupancyMaxActiveClusters(&got, fold_split_kernel, &cfg) != cudaSuccess) got = 0;      // no clusters: layers keep to the other kernels
            k.most[split] = got;
        }
        cudaGetLastError();
    }
    std::copy(k.most, k.most + kMostSlices + 1, most);
}

int cluster_capacity(const gdws_plan_s *p, int split)
{
    static constexpr int b200[kMostSlices + 1] = {0, kB200Sms, 74, 45, 33, 26, 22, 15, 15};      // as a B200 answers: for queries on a host without a GPU
    return p->device >= 0 ? p->clusters[split] : b200[split];
}

namespace {

struct SplitGeom {
    int layout = 0, TN = 0, PH = 0, PW = 0, IW = 0, nl = 0, tiles_n = 0, tiles_h = 0, tiles_w = 0, Npart = 0, nparts = 0, split = 0, na = 0;
    uint32_t a_bytes = 0, a_load = 0, b_off = 0, slot = 0;
    double us = 0;
    int64_t tiles() const { return (int64_t)tiles_n * tiles_h * tiles_w; }
};

struct SplitLaunch {
    LaunchKey key;
    FoldSplitParams P;
    SplitGeom g;
    size_t smem = 0;
    const void *x = nullptr;     // the address the tensor maps were encoded for
};

// Tile, output channels of a block and slices with the shortest estimated time, one wave of blocks; false where a layer does not fit that.
bool split_geometry(const gdws_plan_s *p, int n, int Ho, int Wo, SplitGeom *out)
{
    const int k = p->k, sms = sm_count_of(p);
    const TcTaps t = tc_taps(k, p->stride, p->pad);
    const int units = p->fold_nwin * k;
    bool found = false;
    auto consider = [&](int layout, int TN, int PH, int PW) {
        SplitGeom g;
        g.layout = layout; g.TN = TN; g.PH = PH; g.PW = PW;
        g.tiles_n = (n + TN - 1) / TN; g.tiles_h = (Ho + PH - 1) / PH; g.tiles_w = (Wo + PW - 1) / PW;
        if (g.tiles() > sms) return;
        g.IW = layout == 3 ? 4 : PW + t.ext;
        g.nl = layout == 3 ? k : t.npar;
        g.a_bytes = (uint32_t)(TN * PH * g.IW * 128);
        g.a_load = (g.a_bytes + 1023u) / 1024u * 1024u;
        g.b_off = (uint32_t)g.nl * g.a_load;
        for (int np = 32; np <= 128; np *= 2) {       // more never were the fastest
            g.Npart = std::min(np, (p->D + 15) / 16 * 16);
            g.nparts = (p->D + g.Npart - 1) / g.Npart;
            g.slot = g.b_off + (uint32_t)(k * g.Npart) * 128u;
            const size_t room = kMaxSmem - 1024;
            for (int split = 1; split <= std::min(kMostSlices, units); ++split) {
                if (g.tiles() * g.nparts > cluster_capacity(p, split)) continue;
                const int upc = (units + split - 1) / split;
                g.split = split;
                g.na = (int)std::min<size_t>(std::min(upc, kSplitMaxSlots), room / g.slot);
                if (g.na < std::min(upc, 2) || (size_t)128 * g.Npart * 4 > room) continue;
                // Fitted to 150 timings of ten layers (within 0.4 us but for 128 channels and five or more slices): a unit takes 0.155 us per
                // tap or what its copies take at 60 bytes per clock; the blocks' sums cost 1.6 to 3 us to add up.
                const double unit = std::max(0.155 * k, (g.nl * (double)g.a_bytes + k * g.Npart * 128.0) / 115e3);
                g.us = 3.35 + 0.0095 * g.Npart + upc * unit + (split > 1 ? 1.1 + 0.0115 * g.Npart + 0.11 * split : 0.0);
                if (!found || g.us < out->us) { *out = g; found = true; }
            }
            if (np >= p->D) break;
        }
    };
    if (Wo > 4) {
        for (int PH = 16; PH >= 1; PH >>= 1) consider(2, 16 / PH, PH, 8);
    } else {
        for (int PH = 32; PH >= 2; PH >>= 1) consider(3, 32 / PH, PH, 4);
    }
    return found;
}

// Everything about a launch but the addresses of x and y.
gdws_status_t split_prepare(gdws_plan_s *p, int n, int Ho, int Wo, bool out_f32, SplitLaunch *L)
{
    const int k = p->k, sd = p->stride;
    SplitGeom &g = L->g;
    if (!split_geometry(p, n, Ho, Wo, &g)) return fail(GDWS_ERR_UNSUPPORTED, "folded path in slices: layer not covered");
    FoldSplitParams &P = L->P;
    memset(&P, 0, sizeof(P));
    P.bias = p->d_bias; P.sums = p->d_fold_sums; P.nsums = p->fold_nsums; P.status = p->d_status;
    P.k = k; P.nwin = p->fold_nwin; P.nk_last = (p->C - (p->fold_nwin - 1) * 64 + 15) / 16; P.nl = g.nl; P.Dp = p->fold_dp; P.D = p->D;
    P.Npart = g.Npart; P.nparts = g.nparts; P.relu = p->opt_relu; P.out_f32 = out_f32 ? 1 : 0;
    P.N = n; P.Ho = Ho; P.Wo = Wo; P.TN = g.TN; P.PH = g.PH; P.PW = g.PW; P.tiles_h = g.tiles_h; P.tiles_w = g.tiles_w;
    P.units = p->fold_nwin * k; P.split = g.split; P.na = g.na;
    P.acc_cols = 32;
    while (P.acc_cols < g.Npart) P.acc_cols <<= 1;
    P.a_bytes = g.a_bytes; P.a_load = g.a_load; P.b_tap = (uint32_t)g.Npart * 128u; P.b_off = g.b_off; P.slot = g.slot;
    P.a_sbo = g.layout == 3 ? 1024u : (uint32_t)g.IW * 128u;
    const TcTaps t = tc_taps(k, sd, p->pad);
    for (int u = 0; u < k; ++u) {
        int j = 0;
        for (int wp = 0; wp < sd && g.layout == 2; ++wp) {
            if (!t.used[wp]) continue;
            const int l = u * g.nl + j;
            P.load_map[l] = t.par[u] * 2 + wp; P.load_dh[l] = t.off[u]; P.load_dw[l] = t.omin[wp];
            for (int v = 0; v < k; ++v)
                if (t.par[v] == wp) P.step[u * k + v] = (uint32_t)(t.off[v] - t.omin[wp]) * 8u + (uint32_t)j * (g.a_load >> 4);
            ++j;
        }
        for (int v = 0; v < k && g.layout == 3; ++v, ++j) {
            const int l = u * g.nl + j;
            P.load_map[l] = t.par[u] * 2 + t.par[v]; P.load_dh[l] = t.off[u]; P.load_dw[l] = t.off[v];
            P.step[u * k + v] = (uint32_t)j * (g.a_load >> 4);
        }
        if (j != g.nl) return fail(GDWS_ERR_UNSUPPORTED, "folded path in slices: internal error in the box plan");
    }
    for (int l = 0; l < k * g.nl; ++l) P.maps_used |= 1 << P.load_map[l];
    L->smem = 1024 + std::max((size_t)g.na * g.slot, g.split > 1 ? (size_t)128 * g.Npart * 4 : 0);
    if (L->smem < (size_t)kMaxSmem / 2 + 2048) L->smem = (size_t)kMaxSmem / 2 + 2048;       // one block per SM: tensor memory is never oversubscribed
    tensor_map_encode_fn encode = encode_fn();
    if (!encode) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled is not available from this driver");
    const cuuint64_t dims[2] = {64, (cuuint64_t)2 * P.nwin * k * k * p->fold_dp};
    const cuuint64_t strides[1] = {128};
    const cuuint32_t box[2] = {64, (cuuint32_t)g.Npart}, estr[2] = {1, 1};
    const CUresult r = encode(&P.tmap_w, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, p->d_fold, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (filters) failed with code %d", (int)r);
    return GDWS_OK;
}

gdws_status_t split_map_x(const gdws_plan_s *p, const gdws_tensor_t *x, SplitLaunch *L)
{
    const int sd = p->stride;
    L->x = nullptr;              // until all of them are of this address
    for (int m = 0; m < 4; ++m) {
        if (!((L->P.maps_used >> m) & 1)) continue;
        const int hp = m >> 1, wp = m & 1, Wp = (x->w - wp + sd - 1) / sd, Hp = (x->h - hp + sd - 1) / sd;
        if (Wp <= 0 || Hp <= 0) return fail(GDWS_ERR_UNSUPPORTED, "folded path: input too small for stride %d", sd);
        const cuuint64_t dims[4] = {(cuuint64_t)p->C, (cuuint64_t)Wp, (cuuint64_t)Hp, (cuuint64_t)x->n};
        const cuuint64_t strides[3] = {(cuuint64_t)sd * p->C * 2, (cuuint64_t)sd * x->w * p->C * 2, (cuuint64_t)x->h * x->w * p->C * 2};
        const cuuint32_t box[4] = {64, (cuuint32_t)L->g.IW, (cuuint32_t)L->g.PH, (cuuint32_t)L->g.TN}, estr[4] = {1, 1, 1, 1};
        const CUresult r = encode_fn()(&L->P.tmap_x[m], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (uint8_t *)x->ptr + ((size_t)hp * x->w + wp) * p->C * 2, dims, strides, box, estr,
                                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(GDWS_ERR_CUDA, "cuTensorMapEncodeTiled (x) failed with code %d", (int)r);
    }
    L->x = x->ptr;
    return GDWS_OK;
}

}  // namespace

double fold_split_us(const gdws_plan_s *p, int n, int Ho, int Wo)
{
    SplitGeom g;
    return split_geometry(p, n, Ho, Wo, &g) ? g.us : 1e9;
}

gdws_status_t bf16_folded_split(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, bool given, cudaStream_t st)
{
    const bool out_f32 = y->dtype == GDWS_F32;
    const LaunchKey key = {x->n, x->h, x->w, (p->opt_relu ? 1 : 0) | (out_f32 ? 2 : 0)};
    gdws_status_t rc;
    SplitLaunch *L = LaunchCache<SplitLaunch>::find(p->launch_cache[kCacheSplit], key);
    if (!L) {
        std::unique_ptr<SplitLaunch> e(new (std::nothrow) SplitLaunch);
        if (!e) return fail(GDWS_ERR_ALLOC, "out of host memory");
        e->key = key;
        rc = split_prepare(p, x->n, y->h, y->w, out_f32, e.get());
        if (rc != GDWS_OK) return rc;
        L = LaunchCache<SplitLaunch>::add(p->launch_cache[kCacheSplit], std::move(e));
        if (!L) return fail(GDWS_ERR_ALLOC, "out of host memory");
    }
    if (L->x != x->ptr && (rc = split_map_x(p, x, L)) != GDWS_OK) return rc;
    L->P.y = y->ptr;
    static bool attr_set[64] = {};
    if (!attr_set[p->device & 63]) {
        const cudaError_t e = cudaFuncSetAttribute(fold_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
        if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(fold_split_kernel)");
        attr_set[p->device & 63] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L->g.tiles() * L->g.nparts * L->g.split));
    cfg.blockDim = dim3(kSplitThreads); cfg.dynamicSmemBytes = L->smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    // All 45 clusters of three fit an idle chip, but not one that the packing kernel leaves SM by SM: with overlapped launches a call that is
    // given its weights waited 3 to 8 us for the last ones (448 -> 264 channels at 4 x 20 x 20: 27 us, 23 without; overlap gains 1 elsewhere;
    // other cluster sizes and forwards before it showed nothing of the kind on 250 layers).
    const bool full = L->g.split == 3 && L->g.tiles() * L->g.nparts == cluster_capacity(p, 3);
    attr[0].val.programmaticStreamSerializationAllowed = given && full ? 0 : 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)L->g.split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = L->g.split > 1 ? 2 : 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fold_split_kernel, L->P);
    if (e != cudaSuccess) { cudaGetLastError(); return cuda_fail(e, "fold_split_kernel launch"); }
    p->launches++;
    return GDWS_OK;
}

}  // namespace gdws
