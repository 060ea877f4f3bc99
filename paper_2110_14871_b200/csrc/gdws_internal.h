// Internal declarations shared by the translation units of libgdws.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <memory>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "gdws.h"

namespace gdws {

constexpr int kChunk = 64;          // intermediate channels per tensor-core K chunk (one 128-byte swizzle row of bf16)
constexpr int kTileRows = 128;      // output pixels per tensor-core tile (UMMA M)
constexpr int kMaxK = 7;
constexpr int kHostPieces = 5;      // pieces that gdws_forward_host overlaps
constexpr int kMostSlices = 8;      // blocks of a cluster that share a tile's sum
constexpr int kMaxSmem = 225 * 1024;      // dynamic shared memory a block may ask for (227 KB minus static use)

// What a plan keeps per input size: launches of fused_bf16_kernel, fused_tc_kernel and fold_kernel, the form of a bf16 forward, the pieces
// of a host call, launches of f32_tc_kernel, gdw_tc_kernel and fold_split_kernel.
enum { kCacheAlu, kCacheTc, kCacheFold, kCacheForm, kCachePieces, kCacheF32, kCacheGdw, kCacheSplit, kCaches };

// Bits of the device status word.
enum : int {
    kStatusWaitStage = 1,   // wait for a free shared-memory stage ran out
    kStatusWaitOperand = 2, // wait for an operand (bulk copy / producer warps) ran out
    kStatusWaitMma = 4,     // wait for the tensor-core commit ran out
};

// One unit of work of the tensor-core GDW path: the intermediate channels i0 .. i0+n-1, all fed by the
// 16 input channels cbase .. cbase+15 (a "window"; cbase is a multiple of 16).  Windows whose channels
// produce more than the path's limit of intermediate channels are cut into several chunks.
struct TcChunk {
    int32_t cbase;       // first input channel of the window
    int32_t i0;          // first intermediate channel (canonical order, Property 2)
    int32_t n;           // intermediate channels of the chunk
    int32_t npad;        // n rounded up to a multiple of 16 (columns of the GDW product, K of the PW product)
    int32_t slab0;       // index of the chunk's first 16-channel slab in the packed arrays
    int32_t flags;       // 1: first chunk of its window (its input box is fetched), 2: last chunk of its window
    int32_t reserved0, reserved1;
};

// Most intermediate channels one chunk of the tensor-core GDW path holds: its B operands (32 bytes per channel and
// tap; up to 9 taps per buffer) must fit shared memory twice, and two GDW
// accumulators must fit beside the PW accumulator in TMEM.
inline int tc_nmax(int k, int dloc) { (void)k; return dloc > 128 ? 96 : 128; }

struct Tile {
    int TN = 0, PH = 0, PW = 0;      // images x rows x columns of output pixels per 128-row tile
    int tiles_n = 0, tiles_h = 0, tiles_w = 0;
    int IH = 0, IW = 0;              // input patch rows / columns per image (with halo)
    int cbox = 0;                    // channels per staged box (32, 64 or 128)
    int box_bytes = 0;               // TN*IH*IW*cbox*2: one TMA box
    int slot_bytes = 0;              // box rounded up to 128
    int nslots = 0;                  // staged-input slots (boxes in flight)
    int nwslots = 0;                 // filter blocks in flight (one per chunk)
    int nsb = 0;                     // pointwise-weight units in the ring
    int spg = 2;                     // operand stages per depthwise group (1 or 2)
    int ostage = 0;                  // bytes of output staging for the TMA-store epilogue (0: direct stores)
    int fast = 0;                    // 1: row-run depthwise path, 2: 4-wide-patch path, 0: generic
    size_t smem = 0;                 // dynamic shared memory of the fused kernel
    int64_t tiles() const { return (int64_t)tiles_n * tiles_h * tiles_w; }
};

}  // namespace gdws

struct gdws_plan_s {
    int C = 0, D = 0, k = 0, stride = 0, pad = 0;
    int G = 0, Gpad = 0, Dpad = 0, nchunks = 0;
    int wstride = 0;                 // 32-bit words per intermediate channel in d_dwpack (multiple of 4)
    std::vector<int32_t> g, off, chan;
    bool unused = false;             // some g_c is 0
    std::vector<int32_t> chunk_c0;   // first input channel read by K chunk q (intermediate channels 64q..64q+63)
    std::vector<int32_t> chunk_c1;   // last input channel read by K chunk q
    int span_max = 0;                // widest channel range of one K chunk, counted from the chunk's first
                                     // channel rounded down to a multiple of 8 (a staged box starts there)
    // Input boxes of the fused kernel: consecutive chunks whose channels fit into one box of `cbox`
    // channels share it.  chunk_meta[q] = {box index within the tile, flags, first channel of the box, 0};
    // flags: 1 = this chunk releases the box when done (last or second-to-last chunk using it),
    // 2 = it is the only chunk of its box (releases twice), 4 = first chunk of its box (the loader fetches it),
    // 8 = first or second chunk of its box (must wait for the box to land).
    int cbox = 0, nboxes = 0;
    std::vector<int32_t> chunk_meta; // 4 ints per chunk

    // Tensor-core GDW path (fused_tc.cu): chunk list, output-channel split, packed sizes.
    bool tc_ok = false;              // the layer is one the path covers (stride 1, k <= 5, ...)
    std::vector<gdws::TcChunk> tc_chunks;
    int tc_nslabs = 0;               // sum of npad / 16 over the chunks
    int tc_maxslabs = 0;             // largest npad / 16 of one chunk
    int tc_nparts = 1, tc_dloc = 0;  // blocks per tile along D, output channels per block (multiple of 16, <= 256)
    int tc_rec_hw = 0;               // 16-bit words per filter record (channel slot, then k*k taps; multiple of 8)

    // Folded path (fold.cu): the layer as one k x k convolution.
    bool fold_ok = false;            // the layer is one the path covers
    int fold_nwin = 0, fold_dp = 0;  // windows of 64 input channels; output channels rounded up to 32
    int fold_per = 1;                // output channels per thread that packs them (1 or 4)
    int fold_blocks = 0;             // packing blocks of the folded filters (windows x groups of 4 fold_per output channels)
    int fold_sum_step = 1, fold_nsums = 0;   // every fold_sum_step-th group of a window writes its sums, fold_nsums in all

    int opt_path = GDWS_PATH_AUTO;
    int opt_relu = 0;
    int opt_tile = 0;
    int opt_a_layout = 0;
    int opt_dw_math = 0;
    int opt_out_f32 = 0;           // bf16 plans: y is fp32

    // device side: one allocation (ensure_device), the pointers below lie in it
    void *d_arena = nullptr;
    size_t arena_bytes = 0;
    int device = -1;
    int sm_count = 0;              // SMs of the plan's device (grid size of the persistent kernel)
    int clusters[gdws::kMostSlices + 1] = {};      // clusters of so many blocks, one per SM, that the device runs at the same time
    bool arch_ok = false;          // the plan's device was checked to be compute capability 10.x
    int32_t *d_off = nullptr;      // [C+1]
    int32_t *d_chan = nullptr;     // [Gpad], -1 for padding
    int32_t *d_chunk_meta = nullptr; // [nchunks][4]
    float *d_dw = nullptr;         // [Gpad][k*k] fp32 depthwise filters, zero rows for padding
    uint32_t *d_dwpack = nullptr;  // [Gpad][wstride]: k*k fp32 filter taps, then the channel's index within its K chunk's slot
    uint16_t *d_pw_img = nullptr;  // [nchunks][Dpad*64] bf16, 128-byte-swizzled K-major operand images
    float *d_bias = nullptr;       // [Dpad]
    gdws::TcChunk *d_tc_chunks = nullptr;
    uint16_t *d_tc_filt = nullptr; // [tc_nslabs * 16][tc_rec_hw]: per intermediate slot, channel index inside the window and the taps (bf16)
    uint16_t *d_tc_pw = nullptr;   // [tc_nparts][tc_nslabs][2][tc_dloc][8] bf16: pointwise weights, one K = 16 operand slab per 16 slots
    uint16_t *d_fold = nullptr;    // [2][fold_nwin][k*k][fold_dp][64] bf16: folded filters, then what their rounding left over
    float2 *d_fold_sums = nullptr; // [fold_nsums]: sums that decide whether a forward takes both terms
    int *d_status = nullptr;       // device status word
    bool packed = false, fold_packed = false;      // the forms of the two stages; the folded filters

    void *ws = nullptr;
    size_t ws_bytes = 0;

    void *stage_x = nullptr, *stage_y = nullptr;  // gdws_forward_host staging
    size_t stage_x_bytes = 0, stage_y_bytes = 0;

    // Prepared launches and choices (LaunchCache below; each file knows its own types).
    std::shared_ptr<void> launch_cache[gdws::kCaches];

    int64_t launches = 0;
};

namespace gdws {

void set_error(const char *fmt, ...);
gdws_status_t fail(gdws_status_t st, const char *fmt, ...);
gdws_status_t cuda_fail(cudaError_t e, const char *what);
gdws_status_t ensure_device(gdws_plan_s *p);   // allocate device tables on the current device
gdws_status_t check_arch();
// plan_mem.cu: memory of a plan's tables, on the current device
cudaError_t plan_mem_alloc(int device, size_t bytes, void **out);
void plan_mem_free(int device, void *ptr, size_t bytes);
void plan_count(int device, int change);       // plans that hold memory of the device; the last one gives the shared things back

// Launch with programmatic stream serialisation: the kernel may be scheduled while the kernel before it in the stream
// is still running (once all blocks of that one have executed griddepcontrol.launch_dependents, which the library's
// kernels do first thing).  Such a kernel touches global memory only after its own griddepcontrol.wait.
template <class... KArgs, class... Args>
inline cudaError_t launch_overlapped(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t smem, cudaStream_t st, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(block); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
// What a launch needs besides the tensors' addresses depends on the input size and a few options only: tile shape, work
// split, shared-memory layout, kernel.  Working it out takes longer than a small layer runs, so a plan keeps the last few;
// a call with the same key encodes tensor maps anew only for the addresses that differ from the last call's.
struct LaunchKey {
    int n, h, w, flags;          // input extents; flags: relu, output type, forced options
    bool operator==(const LaunchKey &o) const { return n == o.n && h == o.h && w == o.w && flags == o.flags; }
};
template <class Entry> struct LaunchCache {
    static constexpr size_t kKeep = 8;
    std::vector<std::unique_ptr<Entry>> entries;      // the most recently used one last
    // The entry of `key`, or null.
    static Entry *find(std::shared_ptr<void> &slot, const LaunchKey &key)
    {
        if (!slot) return nullptr;
        auto &v = static_cast<LaunchCache *>(slot.get())->entries;
        for (size_t i = v.size(); i-- > 0;)
            if (v[i]->key == key) {
                if (i + 1 != v.size()) std::rotate(v.begin() + i, v.begin() + i + 1, v.end());
                return v.back().get();
            }
        return nullptr;
    }
    // Keeps `e`; null without host memory for it (nothing is thrown across the C interface).
    static Entry *add(std::shared_ptr<void> &slot, std::unique_ptr<Entry> e)
    {
        try {
            if (!slot) slot = std::shared_ptr<void>(new LaunchCache, [](void *c) { delete static_cast<LaunchCache *>(c); });
            auto &v = static_cast<LaunchCache *>(slot.get())->entries;
            v.reserve(kKeep);
            if (v.size() >= kKeep) v.erase(v.begin());
            v.push_back(std::move(e));
            return v.back().get();
        } catch (const std::bad_alloc &) {
            return nullptr;
        }
    }
};
// Two streams and the events that order the pieces of a gdws_forward_host call.  Creating them takes milliseconds: a call
// borrows a set and gives it back (one more set per device for each call that runs at the same time, at most two kept).
struct HostPipe {
    int device = 0;
    cudaStream_t in = nullptr, out = nullptr;
    cudaEvent_t begin = nullptr, copied[kHostPieces] = {}, computed[kHostPieces] = {};
};
HostPipe *host_pipe_take(int device);       // null if it cannot be made; the device is current
void host_pipe_give(HostPipe *p);           // its streams are idle
// x and y of a forward call against the plan: pointers, alignment, extents, dtype/layout pair, no overlap
gdws_status_t check_pair(const gdws_plan_s *p, const gdws_tensor_t *x, const gdws_tensor_t *y);
// static_ws.cu: looks up (once per device, the device being current) the address of the built-in scratch array
gdws_status_t static_scratch_prepare(int device);
bool choose_tile(const gdws_plan_s *p, int n, int h, int w, Tile *t);

inline size_t dtype_size(gdws_dtype_t d) { return d == GDWS_F32 ? 4 : 2; }

// Where the fused bf16 kernel runs the GDW stage: 1 = ALUs, 2 = tensor cores.  With the option left at 0 the
// tensor cores are taken where they measured faster on B200: their cost is k*k products per 16-channel window
// whatever the multipliers, the ALU kernel's is proportional to G (and its stride-2 code reuses less of each input
// row), and beyond 256 output channels the tensor-core kernel computes the GDW stage once per 256 of them.
inline int gdw_stage_of(const gdws_plan_s *p)
{
    if (p->opt_dw_math == 1 || p->opt_dw_math == 2) return p->opt_dw_math;
    if (!(p->tc_ok && (p->k == 3 || p->k == 5) && p->stride <= 2)) return 1;
    if (p->stride == 1 && p->Dpad > 256) return 1;     // measured equal or slower there; with stride 2 faster at D = 512 too
    // average multiplier of at least 4, or of at least 2.7 when the PW products are small (at most 128 output channels)
    return (p->G >= 4 * p->C || (p->Dpad <= 128 && 10 * (long long)p->G >= 27 * (long long)p->C)) ? 2 : 1;
}

// SMs of the plan's device; a plan built without a device (host-side queries only) assumes a B200's 148.
constexpr int kB200Sms = 148;
inline int sm_count_of(const gdws_plan_s *p) { return p->sm_count > 0 ? p->sm_count : kB200Sms; }

// f32.cu
gdws_status_t f32_depthwise(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, float *z, cudaStream_t s);
gdws_status_t f32_pointwise(gdws_plan_s *p, const float *z, const float *pw_w, const float *bias,
                            gdws_tensor_t *y, cudaStream_t s);
int f32_alu_config(const gdws_plan_s *p, long long npix, int Wo);     // tile of fused_f32_kernel, -1: none
double f32_alu_us(const gdws_plan_s *p, int n, int h, int w);
gdws_status_t f32_fused(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, const float *pw_w,
                        const float *bias, gdws_tensor_t *y, cudaStream_t s);

// f32_tc.cu
double f32_forward_us(gdws_plan_s *p, int n, int h, int w);
// Whether a forward of this size runs there; if not *alu is the ALU kernel's tile (left as it is if there is no memory to keep the answer).
bool f32_tc_takes(gdws_plan_s *p, int n, int h, int w, int *alu);
gdws_status_t f32_fused_tc(gdws_plan_s *p, const gdws_tensor_t *x, const float *dw_w, const float *pw_w,
                           const float *bias, gdws_tensor_t *y, cudaStream_t s);

// pack.cu
constexpr int kFoldPackWide = 256;   // packing blocks of 4 output channels from which on a thread takes four of them
gdws_status_t bf16_pack(gdws_plan_s *p, const void *dw_w, const void *pw_w, const float *bias,
                        gdws_dtype_t dtype, bool fold, cudaStream_t s);

// bf16.cu
gdws_status_t bf16_depthwise(gdws_plan_s *p, const gdws_tensor_t *x, void *z, cudaStream_t s);
gdws_status_t bf16_pointwise(gdws_plan_s *p, const void *z, gdws_tensor_t *y, cudaStream_t s);
// given: the weights came with the call, the kernel before is the one that packs them
gdws_status_t bf16_fused(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, bool given, cudaStream_t s);
gdws_status_t bf16_depthwise_tiled(gdws_plan_s *p, const gdws_tensor_t *x, void *z, cudaStream_t s);

// gdw_tc.cu
gdws_status_t bf16_depthwise_tc(gdws_plan_s *p, const gdws_tensor_t *x, void *z, cudaStream_t s);
bool bf16_depthwise_on_tc(gdws_plan_s *p, int n, int h, int w);        // whether gdws_depthwise runs there

// fused_tc.cu
gdws_status_t bf16_fused_tc(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, cudaStream_t s);

// fold.cu
gdws_status_t bf16_folded(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, bool given, cudaStream_t s);
// fold_split.cu: the folded form in slices, for layers that leave SMs idle
void cluster_capacities(int device, int sms, int (&most)[kMostSlices + 1]);
int cluster_capacity(const gdws_plan_s *p, int split);     // clusters of `split` blocks, one per SM, that run at the same time
double fold_split_us(const gdws_plan_s *p, int n, int Ho, int Wo);      // estimate; 1e9 where it does not cover the layer
gdws_status_t bf16_folded_split(gdws_plan_s *p, const gdws_tensor_t *x, gdws_tensor_t *y, bool given, cudaStream_t s);
bool fold_in_slices(gdws_plan_s *p, int n, int h, int w, bool out_f32);      // whether a folded forward runs there
double bf16_forward_us(gdws_plan_s *p, int n, int h, int w, bool out_f32);
int bf16_form_of(gdws_plan_s *p, int n, int h, int w, bool out_f32);   // 1 / 2: two stages, GDW on the ALUs / the tensor cores; 3: folded

// Input row h = stride * ho + u - pad of filter row u (columns alike).  With stride 2 the input is read through four
// dense views, one per parity of row and column (every other row, every other column): in the view of parity par
// filter row u reads row ho + off of the view, which turns the strided access into a unit-stride one.
struct TcTaps {
    int par[5] = {}, off[5] = {};          // per filter row (the filter is square and padded alike: same for columns)
    int omin[2] = {}, omax[2] = {};        // per parity: smallest and largest offset
    bool used[2] = {};
    int ext = 0;                           // halo of a copy: the largest omax - omin
    int npar = 0;
};

inline TcTaps tc_taps(int k, int stride, int pad)
{
    TcTaps t;
    for (int par = 0; par < 2; ++par) { t.omin[par] = 1 << 20; t.omax[par] = -(1 << 20); }
    for (int u = 0; u < k; ++u) {
        const int i = u - pad;
        const int par = ((i % stride) + stride) % stride;
        t.par[u] = par; t.off[u] = (i - par) / stride;
        t.used[par] = true;
        t.omin[par] = std::min(t.omin[par], t.off[u]); t.omax[par] = std::max(t.omax[par], t.off[u]);
    }
    for (int par = 0; par < 2; ++par)
        if (t.used[par]) { t.ext = std::max(t.ext, t.omax[par] - t.omin[par]); ++t.npar; }
    return t;
}

}  // namespace gdws
