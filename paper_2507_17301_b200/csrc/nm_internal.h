// Library-internal declarations shared by the host API and the kernel translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/nm.h"

constexpr uint32_t NM_MAGIC = 0x4E4D5754u;  // "NMWT"
constexpr uint32_t NM_TAP_PAD = 0xFFFFFFFFu;  // tap-table entry of a padding column: gathers zero
constexpr int NM_KCHUNK = 32;               // kept columns per shared-memory operand chunk (128 B of TF32)

// Least dynamic shared memory of the kernels that allocate all of an SM's tensor memory, and of the cluster kernel, whose
// CTAs wait for CTAs on other SMs: together more than an SM has, so that the two kinds are never resident on one SM and a
// waiting CTA never stands between a cluster's CTA and its tensor memory.
constexpr size_t NM_EXCLUSIVE_SMEM = 204 * 1024;
constexpr size_t NM_BESIDE_EXCLUSIVE = 24 * 1024;

// Compressed weights of one layer.  `values` / `indices` are the canonical, exportable form;
// `wt` and `taps` are what the convolution kernels read.
struct nm_weights {
    uint32_t magic;
    int device;
    uint8_t* block;      // the handle's device memory: one allocation that every array below except `splitk` lies in
    size_t block_bytes, block_used, zero_from;   // size of the block, bytes of it in use, first byte of the part that is cleared
    bool clear_layouts;  // there are layouts in that part
    double* mass;        // device double[2] + int: L1 sums of the pruning pass, validity of imported indices
    int c_out, kh, kw, c_in, k, kk, n_keep, m_group, tile_t, n_tiles;
    int kk_pad;          // kk rounded up to a multiple of NM_KCHUNK
    double l1_total, l1_kept;   // L1 mass of the dense weights / of the retained ones (l1_total < 0: not known)
    float* values;       // [c_out][kk]     exact fp32 copies of the retained weights
    uint16_t* indices;   // [n_tiles][kk]   retained column positions, ascending
    float* wt;           // [n_tiles][kk_pad / 32][rows of the tile][32] retained weights rounded to TF32 (nearest), rows swizzled, zero padded
    uint32_t* taps;      // [n_tiles][kk_pad] kh << 24 | kw << 16 | c per retained column, NM_TAP_PAD in the padding
    int* status;         // device int[4]: [0] error code, [1] where, [2] block, [3] spare
    // Slab layout (variant 2); v2_ok = 0 when the N:M pattern does not fit it.
    // The reduction axis is cut into chunks of v2_g whole groups: v2_s = g * M source columns, of
    // which every tile keeps v2_kc = g * N (a multiple of 8, at most 32).
    int v2_ok, v2_g, v2_kc, v2_s, v2_chunks;
    float* wt2;          // [c_out][v2_chunks * 32] TF32 weights, chunk-major, first v2_kc of each 32 used
    uint8_t* rel2;       // [n_tiles][v2_chunks * 32] source column of each kept column, relative to its chunk
    // Expanded layout (variant 4): the pruned matrix back in dense shape, zeros in the pruned columns.
    float* splitk;       // scratch for split-K partial sums (variant 4), allocated by nm_autotune; may be NULL
    size_t splitk_bytes;
    float* wx;           // [ceil(k / 32)][wx_rows][32] TF32, rows swizzled (see k_compress); NULL when the shape rules the variant out
    int wx_rows;         // c_out rounded up to a multiple of 32 (the rows past c_out are zero)
    // Select layout (variant 8): steps of sel_s source columns of which every tile keeps sel_kc, chunks of as many steps as fit 32
    // retained columns; NULL when the pattern or the shape rules the variant out.
    float* w3;           // [sel_chunks][c_out][32] TF32, rows swizzled (see k_compress)
    uint8_t* sel3;       // [sel_chunks][n_tiles][32 words] column tables (see k_compress)
    int sel_s, sel_kc, sel_chunks;
    // Plane layout (variant 9): per kernel row a [c_out][32] tile of (kw, c) slots; NULL when the shape rules it out.
    float* ws;           // [kh][c_out][32] TF32, rows swizzled (see k_compress)
};

// Division of n < 2^31 by a divisor known to the host, without the hardware's long sequence (Granlund and Montgomery, "Division by
// invariant integers using multiplication", 1994): the eight
// divisions of an item of the select kernel took 2000 cycles of every warp, as long as three chunks.
struct Divisor {
    uint32_t mul, shift;
};
#ifdef __CUDACC__
__device__ __forceinline__ int div_by(int n, const Divisor& d)
{
    return static_cast<int>((__umulhi(static_cast<uint32_t>(n), d.mul) + static_cast<uint32_t>(n)) >> d.shift);
}
#endif
inline Divisor divisor(int d)
{
    Divisor r = {0u, 0u};
    while ((1ll << r.shift) < d) ++r.shift;
    r.mul = static_cast<uint32_t>(((1ull << 32) * ((1ull << r.shift) - static_cast<uint64_t>(d))) / static_cast<uint64_t>(d) + 1);
    return r;
}

// Geometry handed to the convolution kernels.
struct ConvParams {
    const float* x;
    const float* wt;
    const uint32_t* taps;
    const float* bias;
    const float* residual;   // shortcut input added before the activation: the output's shape, or NULL
    float* y;
    int* status;
    int batch, h, w, c_in, ho, wo, c_out;
    int stride_h, stride_w, pad_h, pad_w, dil_h, dil_w;
    int kh, kw;
    int kk, kk_pad, tile_t, n_tiles, relu;
    int n_keep, m_group;
    long long pixels;  // batch * ho * wo
    int k;
    // slab layout (variant 2)
    const float* wt2;
    const uint8_t* rel2;
    int v2_kc, v2_s, v2_chunks;
    // expanded layout (variant 4)
    const float* wx;
    int wx_rows;
    // split-K scratch of the handle (variant 4 with plan.split > 1, variant 8 with plan.ksplit > 1)
    float* splitk;
    size_t splitk_bytes;
    // select layout (variant 8)
    const float* w3;
    const uint8_t* sel3;
    int sel_s, sel_kc;
    // plane layout (variant 9)
    const float* ws;
};

// Pointwise layers (no padding): a stride passes pixels by, so what is read is what is computed from.
inline bool nm_pointwise_reads_more(const ConvParams& p) { return p.pixels * p.c_in > p.pixels * p.c_out; }

#ifdef __CUDACC__
// Shortcut input of one output pixel from channel `channel` on, as float4s (NULL without a residual or past the end).
__device__ __forceinline__ const float4* nm_residual_row(const ConvParams& p, long long pixel, int channel)
{
    if (!p.residual || pixel >= p.pixels) return nullptr;
    return reinterpret_cast<const float4*>(p.residual + pixel * p.c_out + channel);
}
__device__ __forceinline__ void nm_add4(float4& a, const float4& b)
{
    a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
}
#endif

// What the self-checking build checks: a tap-table entry names a tap and a channel of the layer; `bytes` bytes at `at` lie in [lo, hi).
#ifdef __CUDACC__
#define NM_HOST_DEVICE __host__ __device__
#else
#define NM_HOST_DEVICE
#endif
NM_HOST_DEVICE constexpr bool nm_tap_in_layer(uint32_t tap, int kh, int kw, int c_in)
{
    return static_cast<int>(tap >> 24) < kh && static_cast<int>((tap >> 16) & 0xFFu) < kw && static_cast<int>(tap & 0xFFFFu) < c_in;
}
NM_HOST_DEVICE constexpr bool nm_bytes_in_span(uint64_t at, uint64_t bytes, uint64_t lo, uint64_t hi) { return at >= lo && at + bytes <= hi; }

#ifdef __CUDACC__
// Self-checking build (-DNM_DEBUG_BOUNDS): the kernels that compute addresses from index data range-check
// every such address; a violation is recorded in the handle's status word (error code NM_ERR_INTERNAL, the
// site, the block, the offending value) and the access is skipped.  Nothing traps; nm_weights_check reports it.
#ifdef NM_DEBUG_BOUNDS
__device__ __forceinline__ void nm_debug_violation(int* status, int site, uint32_t value)
{
    if (atomicCAS(status + 0, 0, static_cast<int>(NM_ERR_INTERNAL)) == 0) {
        atomicExch(status + 1, site);
        atomicExch(status + 2, static_cast<int>(blockIdx.x));
        atomicExch(status + 3, static_cast<int>(value));
    }
}
#define NM_CHECKED(cond, status, site, value) \
    if (!(cond)) nm_debug_violation((status), (site), static_cast<uint32_t>(value)); else
// `cond` where it decides whether an access is made: false, and recorded, on a violation.
#define NM_ALLOWED(cond, status, site, value) ((cond) || (nm_debug_violation((status), (site), static_cast<uint32_t>(value)), false))
constexpr bool NM_SELF_CHECKING = true;
#else
#define NM_CHECKED(cond, status, site, value)
#define NM_ALLOWED(cond, status, site, value) true
constexpr bool NM_SELF_CHECKING = false;
#endif
#endif

namespace nmhost {
int sm_count();   // of the device that is current at the first call

// Rounds of `ctas` CTAs, two per SM: the last one counts in full while there are few, half where they drift apart.
inline double cta_rounds(long long ctas, int sms)
{
    const double x = static_cast<double>(ctas) / (2.0 * sms);
    return x < 4.0 ? static_cast<double>((ctas + 2 * sms - 1) / (2 * sms)) : x + 0.5;
}

// Launches `kernel` so that it may begin while the previous kernel of the stream drains
// (programmatic dependent launch); the kernel orders itself with griddepcontrol.wait.
// NM_NO_PDL=1 in the environment falls back to a plain launch.
bool pdl_enabled();
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl_enabled() ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Raises a kernel's dynamic shared-memory limit on the current device, calling the runtime only when a launch
// needs more than the limit already in force (the call would otherwise sit between every two launches).
cudaError_t ensure_dynamic_smem(const void* kernel, size_t bytes);

// Sets the calling thread's error text and returns `s`.
nm_status_t fail(nm_status_t s, const char* fmt, ...);
void count_launch(int n = 1);

// Whether a kernel of device `current` may read or write memory of this kind and owner.  Everything else (another device's
// memory without a peer mapping, pageable host memory) is left to cudaMemcpyAsync, which copies it or refuses it.
constexpr bool kernel_may_touch(cudaMemoryType type, int owner, int current)
{
    return type == cudaMemoryTypeManaged || (type == cudaMemoryTypeDevice && owner == current);
}
bool kernel_may_touch(const void* a, const void* b, int device);   // both of them; false unless `device` is the current one

// nm_layout.cu: the handles' device memory, and the kernel-side copies of the compressed form
void* device_block_alloc(size_t bytes, int device, size_t* got);   // NULL when there is no memory; reuses blocks of freed handles
void device_block_free(void* ptr, size_t bytes, int device, bool idle);   // idle: nothing on the device uses it any more
void device_blocks_trim();                                 // gives back every block kept for later handles
cudaError_t device_malloc(void** ptr, size_t bytes);       // cudaMalloc, tried again after a trim
nm_status_t alloc_handle_memory(nm_weights* h, const char* who);
nm_status_t clear_handle_memory(nm_weights* h, cudaStream_t st);   // the part of the block that is not written in full
// Values and layouts from the index array `idx` and the dense weights (import = false) or the retained values (true).
nm_status_t build_layouts(nm_weights* h, const float* src, const uint16_t* idx, bool import, cudaStream_t st);
nm_status_t finish_handle(nm_weights* h, cudaStream_t st, double* mass2, int* bad);   // synchronises `st`
// Groups that fit a block: selection (`idx` NULL, `src` dense) or check of given indices (`src`: retained values) and all layouts in one
// kernel; synchronises `st`.
bool compressed_in_one(const nm_weights* h);
nm_status_t compress_in_one(nm_weights* h, const float* src, const uint16_t* idx, cudaStream_t st, double* mass2, int* bad);

// nm_prune.cu
nm_status_t prune_on_device(const float* w_dense, nm_weights* h, cudaStream_t st);
nm_status_t build_from_compressed(const float* values, const uint16_t* indices, nm_weights* h, cudaStream_t st);

// nm_conv_gather.cu — variant 1
// MMA width of a tile: the channels it can have, in sixteens
inline int gather_width(int tile_t, int c_out) { return ((tile_t < c_out ? tile_t : c_out) + 15) / 16 * 16; }
nm_status_t launch_conv_gather(const ConvParams& p, cudaStream_t st);
double gather_time_us(const ConvParams& p);   // estimate, one range of the chunks
double gather_estimate_us(const ConvParams& p);   // the same where the stream kernel takes the layer, over all sizes

// nm_conv_slab.cu — variant 2
bool slab_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_slab(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);
// Whether the library default takes this kernel rather than the gather kernel: many CTAs of few chunks, tiles narrow enough that
// several share a pixel block (see the estimates).
bool slab_beats_gather(const ConvParams& p);

// nm_conv_expand.cu — variant 4
bool expand_plan_ok(const ConvParams& p, const nm_plan_t* plan);
size_t expand_splitk_bytes(const ConvParams& p, int splits);   // scratch a split-K plan of this layer needs
size_t expand_balanced_bytes(int bn);                          // scratch a balanced plan (split = -1) with this bn needs
nm_status_t launch_conv_expand(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// second pass of a plan that splits the reduction axis: y = act(sum of the `splits` partial sums
// [split][p_pad pixels][c_out] in p.splitk + bias + shortcut)
nm_status_t launch_splitk_reduce(const ConvParams& p, int splits, int p_pad, cudaStream_t st);

// nm_conv_rowrun.cu — variant 5
bool rowrun_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_rowrun(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_window.cu — variant 6
bool window_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_window(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_pair.cu — variant 7
bool pair_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_pair(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_stream.cu — variant 3
int stream_width(const ConvParams& p, const nm_plan_t* plan);   // channels per work item, 0: the kernel does not take the layer / plan
bool stream_beats_gather(const ConvParams& p);   // (and takes the layer)
nm_status_t launch_conv_stream(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_select.cu — variant 8
bool select_layout_dims(const nm_weights* h, int* s, int* kc);   // false: the pattern or shape rules the kernel out
bool select_plan_ok(const ConvParams& p, const nm_plan_t* plan);
int select_ranges(const ConvParams& p, const nm_plan_t* plan);   // of the reduction axis, 0: the plan does not fit
size_t select_splitk_bytes(const ConvParams& p, int splits);
nm_status_t launch_conv_select(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_planes.cu — variant 9
bool planes_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_planes(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);

// nm_conv_cluster.cu — variant 10
bool cluster_plan_ok(const ConvParams& p, const nm_plan_t* plan);
nm_status_t launch_conv_cluster(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st);
}  // namespace nmhost
