// Host side of the C ABI declared in include/nm.h: argument checks, handle life cycle, plan
// resolution, launches, auto-tuning.  No tensor type other than raw pointers crosses this file.
#include <algorithm>
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <mutex>
#include <unordered_map>
#include <vector>

#include "nm_internal.h"

namespace {
thread_local char g_err[512] = "";
std::atomic<uint64_t> g_launches{0};

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Two byte ranges (16-byte aligned at both ends) copied side by side.
__global__ void k_export(const char* src_a, char* dst_a, size_t bytes_a, const char* src_b, char* dst_b, size_t bytes_b)
{
    const size_t a16 = bytes_a / 16, b16 = bytes_b / 16, step = static_cast<size_t>(gridDim.x) * blockDim.x;
    const size_t first = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
    for (size_t i = first; i < a16 + b16; i += step) {
        if (i < a16) reinterpret_cast<uint4*>(dst_a)[i] = __ldg(reinterpret_cast<const uint4*>(src_a) + i);
        else reinterpret_cast<uint4*>(dst_b)[i - a16] = __ldg(reinterpret_cast<const uint4*>(src_b) + (i - a16));
    }
    if (first < bytes_a % 16) dst_a[a16 * 16 + first] = src_a[a16 * 16 + first];
    if (first < bytes_b % 16) dst_b[b16 * 16 + first] = src_b[b16 * 16 + first];
}

int kept_count(int k, int n_keep, int m_group)
{
    const int full = k / m_group, tail = k % m_group;
    return full * n_keep + std::min(tail, n_keep);
}

// `idle`: the device has been synchronised, so the block may serve the next handle.
void free_handle_memory(nm_weights* h, bool idle)
{
    if (!h) return;
    nmhost::device_block_free(h->block, h->block_bytes, h->device, idle);
    cudaFree(h->splitk);
    h->magic = 0;
    delete h;
}

// Validates the layer description and allocates an empty handle.
nm_status_t make_handle(const char* who, int c_out, int kh, int kw, int c_in, int n_keep, int m_group, int tile_t,
                        nm_weights** out)
{
    if (!out) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: out is NULL", who);
    *out = nullptr;
    if (c_out < 1 || kh < 1 || kw < 1 || c_in < 1)
        return nmhost::fail(NM_ERR_INVALID_ARG, "%s: c_out, kh, kw, c_in must be >= 1", who);
    if (n_keep < 1 || m_group < 1 || n_keep > m_group)
        return nmhost::fail(NM_ERR_INVALID_ARG, "%s: need 1 <= n_keep <= m_group (got %d:%d)", who, n_keep, m_group);
    if (tile_t < 1) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: tile_t must be >= 1", who);
    const long long k = static_cast<long long>(kh) * kw * c_in;
    if (k > 65535) return nmhost::fail(NM_ERR_UNSUPPORTED, "%s: K = %lld exceeds the uint16 index range", who, k);
    if (kh > 255 || kw > 255) return nmhost::fail(NM_ERR_UNSUPPORTED, "%s: kernel extent above 255", who);
    if (tile_t > 256) return nmhost::fail(NM_ERR_UNSUPPORTED, "%s: tile_t above 256", who);

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "%s: cudaGetDevice: %s", who, cudaGetErrorString(e));

    nm_weights* h = new (std::nothrow) nm_weights();
    if (!h) return nmhost::fail(NM_ERR_ALLOC, "%s: out of host memory", who);
    std::memset(h, 0, sizeof(*h));
    h->magic = NM_MAGIC;
    h->l1_total = -1.0;
    h->l1_kept = -1.0;
    h->device = dev;
    h->c_out = c_out; h->kh = kh; h->kw = kw; h->c_in = c_in;
    h->k = static_cast<int>(k);
    h->n_keep = n_keep; h->m_group = m_group; h->tile_t = tile_t;
    h->kk = kept_count(h->k, n_keep, m_group);
    h->n_tiles = (c_out + tile_t - 1) / tile_t;
    h->kk_pad = ((h->kk + NM_KCHUNK - 1) / NM_KCHUNK) * NM_KCHUNK;
    const nm_status_t s = nmhost::alloc_handle_memory(h, who);
    if (s != NM_OK) {
        delete h;
        return s;
    }
    *out = h;
    return NM_OK;
}

// Makes a handle's device the current one, where it is not, for as long as the object lives.
struct OnDevice {
    int before = -1;
    explicit OnDevice(int device)
    {
        int dev = device;
        if (cudaGetDevice(&dev) == cudaSuccess && dev != device && cudaSetDevice(device) == cudaSuccess) before = dev;
    }
    ~OnDevice()
    {
        if (before >= 0) cudaSetDevice(before);
    }
    OnDevice(const OnDevice&) = delete;
    OnDevice& operator=(const OnDevice&) = delete;
};

bool valid(const nm_weights* w) { return w && w->magic == NM_MAGIC; }

// Checks a conv call and fills the kernel parameters.
nm_status_t make_params(const char* who, const nm_weights* w, const float* x, int batch, int h, int wd, int stride_h,
                        int stride_w, int pad_h, int pad_w, int dil_h, int dil_w, const float* bias, int relu,
                        float* y, ConvParams* p)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: bad weights handle", who);
    if (!x || !y) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: x or y is NULL", who);
    if (batch < 1 || h < 1 || wd < 1) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: batch, h, w must be >= 1", who);
    if (stride_h < 1 || stride_w < 1 || dil_h < 1 || dil_w < 1 || pad_h < 0 || pad_w < 0)
        return nmhost::fail(NM_ERR_INVALID_ARG, "%s: stride and dilation must be >= 1, padding >= 0", who);
    if (!aligned16(x) || !aligned16(y) || (bias && !aligned16(bias)))
        return nmhost::fail(NM_ERR_INVALID_ARG, "%s: x, y and bias must be 16-byte aligned", who);
    const long long eh = static_cast<long long>(h) + 2ll * pad_h - static_cast<long long>(dil_h) * (w->kh - 1) - 1;
    const long long ew = static_cast<long long>(wd) + 2ll * pad_w - static_cast<long long>(dil_w) * (w->kw - 1) - 1;
    if (eh < 0 || ew < 0) return nmhost::fail(NM_ERR_INVALID_ARG, "%s: the kernel does not fit the padded image", who);
    const long long ho = eh / stride_h + 1, wo = ew / stride_w + 1;
    const long long pixels = static_cast<long long>(batch) * ho * wo;
    if (ho > 0x7FFFFFFF || wo > 0x7FFFFFFF || pixels > (1ll << 40))
        return nmhost::fail(NM_ERR_UNSUPPORTED, "%s: output too large", who);
    p->x = x; p->wt = w->wt; p->taps = w->taps; p->bias = bias; p->residual = nullptr; p->y = y; p->status = w->status;
    p->batch = batch; p->h = h; p->w = wd; p->c_in = w->c_in;
    p->ho = static_cast<int>(ho); p->wo = static_cast<int>(wo); p->c_out = w->c_out;
    p->stride_h = stride_h; p->stride_w = stride_w; p->pad_h = pad_h; p->pad_w = pad_w;
    p->dil_h = dil_h; p->dil_w = dil_w; p->kh = w->kh; p->kw = w->kw;
    p->kk = w->kk; p->kk_pad = w->kk_pad; p->tile_t = w->tile_t; p->n_tiles = w->n_tiles; p->relu = relu ? 1 : 0;
    p->n_keep = w->n_keep; p->m_group = w->m_group;
    p->pixels = pixels;
    p->k = w->k;
    p->wt2 = w->v2_ok ? w->wt2 : nullptr;
    p->rel2 = w->v2_ok ? w->rel2 : nullptr;
    p->v2_kc = w->v2_kc; p->v2_s = w->v2_s; p->v2_chunks = w->v2_chunks;
    p->wx = w->wx;
    p->wx_rows = w->wx_rows;
    p->splitk = w->splitk;
    p->splitk_bytes = w->splitk_bytes;
    p->w3 = w->w3;
    p->sel3 = w->sel3;
    p->sel_s = w->sel_s; p->sel_kc = w->sel_kc;
    p->ws = w->ws;
    return NM_OK;
}

nm_status_t run_plan(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st)
{
    const int variant = plan ? plan->variant : 0;
    switch (variant) {
        case 0:
            // (the row-run and plane kernels truncate activations and multiply zeros for pruned columns, the others do neither)
            if (nmhost::stream_beats_gather(p)) return nmhost::launch_conv_stream(p, nullptr, st);
            if (nmhost::planes_plan_ok(p, nullptr)) return nmhost::launch_conv_planes(p, nullptr, st);
            // Channel counts that are no multiple of 32: runs of rows where there is enough work for their set-up.  Units of a pixel
            // block, tile and chunk, and us against the gather's: 2352 (8x112x112, 16->32) 18.4 / 20.6, 1568 (32x56x56, 8->64 by
            // 2) 14.4 / 16.4; 1176 (4x56x56, 24->96) 10.1 / 8.3, 784 (2x112x112, 5->32, 7x7 by 2) 6.9 / 5.5.
            if (p.c_in % 32 != 0 && (p.pixels + 127) / 128 * p.n_tiles * (p.kk_pad / NM_KCHUNK) >= 1400 && nmhost::rowrun_plan_ok(p, nullptr))
                return nmhost::launch_conv_rowrun(p, nullptr, st);
            if (nmhost::slab_beats_gather(p)) return nmhost::launch_conv_slab(p, nullptr, st);
            return nmhost::launch_conv_gather(p, st);
        case 1:
            return nmhost::launch_conv_gather(p, st);
        case 2:
            return nmhost::launch_conv_slab(p, plan, st);
        case 3:
            return nmhost::launch_conv_stream(p, plan, st);
        case 4:
            return nmhost::launch_conv_expand(p, plan, st);
        case 5:
            return nmhost::launch_conv_rowrun(p, plan, st);
        case 6:
            return nmhost::launch_conv_window(p, plan, st);
        case 7:
            return nmhost::launch_conv_pair(p, plan, st);
        case 8:
            return nmhost::launch_conv_select(p, plan, st);
        case 9:
            return nmhost::launch_conv_planes(p, plan, st);
        case 10:
            return nmhost::launch_conv_cluster(p, plan, st);
        default:
            return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_conv2d: unknown plan variant %d", variant);
    }
}

// Candidate plans for a layer, most promising first: of two that time alike the earlier is kept.  The expanded-operand kernel
// stands before the select and stream kernels because it adds a shortcut input at less cost (64 -> 256 at 56x56, batch 64: 45
// against 47 us without one, 83 against 113 us with one), which the tuner cannot see.
std::vector<nm_plan_t> candidate_plans(const nm_weights* /*w*/, const ConvParams& p)
{
    std::vector<nm_plan_t> out;
    nm_plan_t a;
    std::memset(&a, 0, sizeof(a));
    // cluster kernel (short launches)
    for (int ksplit : {8, 4, 2, 1}) {
        for (int bn : {32, 64, 128}) {
            a.variant = 10; a.bn = bn; a.ksplit = ksplit;
            if (nmhost::cluster_plan_ok(p, &a)) out.push_back(a);
        }
    }
    std::memset(&a, 0, sizeof(a));
    for (int mt : {2, 3, 4, 1}) {           // window kernel (stride-1 spatial kernels)
        for (int bn : {64, 128, 256}) {
            a.variant = 6; a.bn = bn; a.split = mt; a.stages = 0;
            if (nmhost::window_plan_ok(p, &a)) out.push_back(a);
        }
    }
    std::memset(&a, 0, sizeof(a));
    for (int rows : {0, 2}) {               // plane kernel (at most four input channels, stride 1 or 2)
        a.variant = 9; a.split = rows;
        if (nmhost::planes_plan_ok(p, &a)) out.push_back(a);
    }
    std::memset(&a, 0, sizeof(a));
    a.variant = 5;                          // row-run kernel (few input channels)
    if (p.c_in % 32 != 0 && nmhost::rowrun_plan_ok(p, &a)) out.push_back(a);
    std::memset(&a, 0, sizeof(a));
    // channel widths of a work item for the expanded-operand kernel: the usual three, plus the whole (padded)
    // channel count and 32 for layers whose channel count is not a multiple of 64
    std::vector<int> widths = {64, 128, 256};
    if (p.wx_rows % 64 != 0) {
        if (p.wx_rows <= 256) widths.push_back(p.wx_rows);
        if (p.wx_rows != 32) widths.push_back(32);
    }
    for (int split : {0, 1}) {              // expanded-operand kernel: weights resident where they fit / streamed,
        for (int bn : widths) {             // one or two 32-column blocks per pipeline stage
            for (int kblk : {1, 2}) {
                a.variant = 4; a.bn = bn; a.stages = 0; a.split = split; a.kblk = kblk;
                if (nmhost::expand_plan_ok(p, &a)) out.push_back(a);
            }
        }
    }
    a.kblk = 0;
    for (int bn : {256, 128}) {             // ... run by pairs of CTAs (half the weight traffic per SM)
        a.variant = 7; a.bn = bn; a.stages = 0; a.split = 0;
        if (nmhost::pair_plan_ok(p, &a)) out.push_back(a);
    }
    for (int bn : {256, 128}) {             // ... with (item, stage) ranges balanced over the SMs (needs the handle's scratch)
        for (int kblk : {1, 2}) {
            a.variant = 4; a.bn = bn; a.stages = 0; a.split = -1; a.kblk = kblk;
            if (nmhost::expand_plan_ok(p, &a)) out.push_back(a);
        }
    }
    a.kblk = 0;
    for (int splits : {2, 3, 4}) {          // ... with the reduction axis split (needs the handle's scratch)
        for (int bn : {128, 256}) {
            for (int kblk : {1, 2}) {
                a.variant = 4; a.bn = bn; a.stages = 0; a.split = splits; a.kblk = kblk;
                if (nmhost::expand_plan_ok(p, &a)) out.push_back(a);
            }
        }
    }
    std::memset(&a, 0, sizeof(a));
    // select kernel (contracts over the retained columns only): all of a tile group's channels per CTA down to one
    // tile, with the activation loads it prefers for the shape, and with the reduction axis split where few work
    // items exist (the split plans need the handle's scratch)
    for (int ksplit : {1, 2, 3, 4}) {
        for (int bn : {128, 256, 64, 32}) {
            a.variant = 8; a.bn = bn; a.ksplit = ksplit;
            if (bn % p.tile_t == 0 && nmhost::select_ranges(p, &a) == ksplit) out.push_back(a);
        }
    }
    std::memset(&a, 0, sizeof(a));
    std::vector<int> listed;
    for (int bn : {0, 256, p.tile_t, nmhost::stream_width(p, nullptr)}) {   // stream kernel: default width, widest, one tile per CTA, and the one
        a.variant = 3; a.bn = bn; a.stages = 0;                             // that a call without a plan takes
        const int width = nmhost::stream_width(p, &a);
        if (width == 0 || std::find(listed.begin(), listed.end(), width) != listed.end()) continue;
        listed.push_back(width);
        out.push_back(a);
    }
    std::memset(&a, 0, sizeof(a));
    for (int bn : {0, p.tile_t}) {          // default (as many tiles as fit) and one tile per CTA
        for (int stages : {2, 3}) {
            a.variant = 2; a.bn = bn; a.stages = stages;
            if (nmhost::slab_plan_ok(p, &a)) out.push_back(a);
        }
    }
    std::memset(&a, 0, sizeof(a));
    a.variant = 1;
    out.push_back(a);
    // NM_AUTOTUNE_VARIANTS="1,2,3" restricts the search (e.g. to the kernels that gather only the
    // retained columns); unset = every variant
    if (const char* allow = std::getenv("NM_AUTOTUNE_VARIANTS")) {
        std::vector<nm_plan_t> kept;
        for (const nm_plan_t& c : out)
            if (c.variant < 10 && std::strchr(allow, '0' + c.variant)) kept.push_back(c);
        if (!kept.empty()) out.swap(kept);
    }
    return out;
}

}  // namespace

namespace nmhost {
nm_status_t fail(nm_status_t s, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return s;
}
int sm_count()
{
    static const int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
            return v;
        return 148;
    }();
    return n;
}
bool pdl_enabled()
{
    static const bool on = [] {
        const char* v = std::getenv("NM_NO_PDL");
        return !(v && v[0] == '1');
    }();
    return on;
}
void count_launch(int n) { g_launches.fetch_add(static_cast<uint64_t>(n), std::memory_order_relaxed); }
cudaError_t ensure_dynamic_smem(const void* kernel, size_t bytes)
{
    static std::mutex mu;
    static std::unordered_map<uint64_t, size_t> in_force;   // (device, kernel) -> limit set so far
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t key = (static_cast<uint64_t>(reinterpret_cast<uintptr_t>(kernel)) << 6) ^ static_cast<uint64_t>(dev & 63);
    std::lock_guard<std::mutex> lock(mu);
    const auto it = in_force.find(key);
    if (it != in_force.end() && it->second >= bytes) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    if (e == cudaSuccess) in_force[key] = bytes;
    return e;
}
}  // namespace nmhost

extern "C" {

nm_status_t nm_prune(const float* w_dense, int c_out, int kh, int kw, int c_in, int n_keep, int m_group, int tile_t,
                     void* cuda_stream, nm_weights_t** out)
{
    if (!w_dense) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_prune: w_dense is NULL");
    nm_weights* h = nullptr;
    nm_status_t s = make_handle("nm_prune", c_out, kh, kw, c_in, n_keep, m_group, tile_t, &h);
    if (s != NM_OK) return s;
    s = nmhost::prune_on_device(w_dense, h, static_cast<cudaStream_t>(cuda_stream));
    if (s != NM_OK) {
        free_handle_memory(h, false);
        return s;
    }
    *out = h;
    return NM_OK;
}

nm_status_t nm_weights_import(const float* values, const uint16_t* indices, int c_out, int kh, int kw, int c_in,
                              int n_keep, int m_group, int tile_t, void* cuda_stream, nm_weights_t** out)
{
    if (!values || !indices) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_import: values or indices is NULL");
    nm_weights* h = nullptr;
    nm_status_t s = make_handle("nm_weights_import", c_out, kh, kw, c_in, n_keep, m_group, tile_t, &h);
    if (s != NM_OK) return s;
    s = nmhost::build_from_compressed(values, indices, h, static_cast<cudaStream_t>(cuda_stream));
    if (s != NM_OK) {
        free_handle_memory(h, false);
        *out = nullptr;
        return s;
    }
    *out = h;
    return NM_OK;
}

nm_status_t nm_weights_dims(const nm_weights_t* w, int* c_out, int* k, int* kk, int* n_tiles, int* tile_t)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_dims: bad weights handle");
    if (c_out) *c_out = w->c_out;
    if (k) *k = w->k;
    if (kk) *kk = w->kk;
    if (n_tiles) *n_tiles = w->n_tiles;
    if (tile_t) *tile_t = w->tile_t;
    return NM_OK;
}

nm_status_t nm_weights_retained_l1(const nm_weights_t* w, double* kept, double* total)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_retained_l1: bad weights handle");
    if (w->l1_total < 0.0)
        return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_weights_retained_l1: the handle was imported, the dense weights were never seen");
    if (kept) *kept = w->l1_kept;
    if (total) *total = w->l1_total;
    return NM_OK;
}

nm_status_t nm_weights_export(const nm_weights_t* w, float* values, uint16_t* indices, void* cuda_stream)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_export: bad weights handle");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    cudaError_t e = cudaSuccess;
    const size_t vb = static_cast<size_t>(w->c_out) * w->kk * sizeof(float), ib = static_cast<size_t>(w->n_tiles) * w->kk * sizeof(uint16_t);
    if (values && indices && w->kk > 0 && aligned16(values) && aligned16(indices) &&
        nmhost::kernel_may_touch(values, indices, w->device)) {
        // both arrays in one launch (512 x 2304 values: 33 us as two copies, 20)
        k_export<<<static_cast<unsigned>(std::min<size_t>((vb + ib) / 4096 + 1, 1184)), 256, 0, st>>>(
            reinterpret_cast<const char*>(w->values), reinterpret_cast<char*>(values), vb, reinterpret_cast<const char*>(w->indices),
            reinterpret_cast<char*>(indices), ib);
        nmhost::count_launch(1);
        e = cudaGetLastError();
    } else {
        if (values && w->kk > 0) e = cudaMemcpyAsync(values, w->values, vb, cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess && indices && w->kk > 0) e = cudaMemcpyAsync(indices, w->indices, ib, cudaMemcpyDeviceToDevice, st);
    }
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_weights_export: %s", cudaGetErrorString(e));
    return NM_OK;
}

nm_status_t nm_plan_scratch_bytes(const nm_weights_t* w, int batch, int h, int wd, int stride_h, int stride_w,
                                  int pad_h, int pad_w, int dil_h, int dil_w, const nm_plan_t* plan, size_t* bytes)
{
    if (!bytes) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_scratch_bytes: bytes is NULL");
    *bytes = 0;
    ConvParams p;
    float* const dummy = reinterpret_cast<float*>(static_cast<uintptr_t>(256));   // geometry only: never dereferenced
    nm_status_t s = make_params("nm_plan_scratch_bytes", w, dummy, batch, h, wd, stride_h, stride_w, pad_h, pad_w,
                                dil_h, dil_w, nullptr, 0, dummy, &p);
    if (s != NM_OK) return s;
    if (plan && plan->variant == 4 && plan->split > 1) *bytes = nmhost::expand_splitk_bytes(p, plan->split);
    if (plan && plan->variant == 4 && plan->split == -1) *bytes = nmhost::expand_balanced_bytes(plan->bn > 0 ? plan->bn : 256);
    if (plan && plan->variant == 8 && plan->ksplit > 1) *bytes = nmhost::select_splitk_bytes(p, plan->ksplit);
    return NM_OK;
}

nm_status_t nm_weights_reserve(nm_weights_t* w, size_t bytes)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_reserve: bad weights handle");
    if (bytes <= w->splitk_bytes) return NM_OK;
    const OnDevice on(w->device);
    cudaDeviceSynchronize();
    cudaFree(w->splitk);
    w->splitk = nullptr;
    w->splitk_bytes = 0;
    if (nmhost::device_malloc(reinterpret_cast<void**>(&w->splitk), bytes) != cudaSuccess)
        return nmhost::fail(NM_ERR_ALLOC, "nm_weights_reserve: cannot allocate %zu bytes", bytes);
    // balanced plans keep flag words in the scratch: they start cleared, before a launch on any stream can read them
    if (cudaMemset(w->splitk, 0, bytes) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) {
        (void)cudaGetLastError();
        cudaFree(w->splitk);
        w->splitk = nullptr;
        return nmhost::fail(NM_ERR_CUDA, "nm_weights_reserve: cannot clear the scratch");
    }
    w->splitk_bytes = bytes;
    return NM_OK;
}

nm_status_t nm_weights_check(const nm_weights_t* w, void* cuda_stream)
{
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_check: bad weights handle");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    int host[4] = {0, 0, 0, 0};
    cudaError_t e = cudaMemcpyAsync(host, w->status, sizeof(host), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_weights_check: %s", cudaGetErrorString(e));
    if (host[0] != 0) {
        cudaMemsetAsync(w->status, 0, 3 * sizeof(int), st);
        // a balanced launch that gave up may have left flags raised at the start of the scratch
        if (w->splitk) cudaMemsetAsync(w->splitk, 0, w->splitk_bytes < 16384 ? w->splitk_bytes : 16384, st);
        cudaStreamSynchronize(st);
        return nmhost::fail(static_cast<nm_status_t>(host[0]), "device-side wait expired (site %d, block %d)", host[1],
                            host[2]);
    }
    return NM_OK;
}

nm_status_t nm_weights_free(nm_weights_t* w)
{
    if (!w) return NM_OK;
    if (!valid(w)) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_weights_free: bad weights handle");
    const OnDevice on(w->device);
    const bool idle = cudaDeviceSynchronize() == cudaSuccess;
    free_handle_memory(w, idle);
    return NM_OK;
}

nm_status_t nm_memory_trim(void)
{
    nmhost::device_blocks_trim();
    return NM_OK;
}

nm_status_t nm_conv2d(const nm_weights_t* w, const float* x, int batch, int h, int wd, int stride_h, int stride_w,
                      int pad_h, int pad_w, int dil_h, int dil_w, const float* bias, int relu, float* y,
                      const nm_plan_t* plan, void* cuda_stream)
{
    ConvParams p;
    nm_status_t s = make_params("nm_conv2d", w, x, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, bias,
                                relu, y, &p);
    if (s != NM_OK) return s;
    return run_plan(p, plan, static_cast<cudaStream_t>(cuda_stream));
}

nm_status_t nm_conv2d_res(const nm_weights_t* w, const float* x, int batch, int h, int wd, int stride_h, int stride_w,
                          int pad_h, int pad_w, int dil_h, int dil_w, const float* bias, const float* residual,
                          int relu, float* y, const nm_plan_t* plan, void* cuda_stream)
{
    ConvParams p;
    nm_status_t s = make_params("nm_conv2d_res", w, x, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w,
                                bias, relu, y, &p);
    if (s != NM_OK) return s;
    if (residual && !aligned16(residual))
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_conv2d_res: residual must be 16-byte aligned");
    if (residual && p.c_out % 4 != 0)
        return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_conv2d_res: c_out must be a multiple of 4");
    p.residual = residual;
    return run_plan(p, plan, static_cast<cudaStream_t>(cuda_stream));
}

nm_status_t nm_conv2d_host(const nm_weights_t* w, const float* x_host, float* x_dev, int batch, int h, int wd,
                           int stride_h, int stride_w, int pad_h, int pad_w, int dil_h, int dil_w,
                           const float* bias_host, float* bias_dev, int relu, float* y_host, float* y_dev,
                           const nm_plan_t* plan, void* cuda_stream)
{
    if (!x_host || !y_host) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_conv2d_host: x_host or y_host is NULL");
    if (bias_host && !bias_dev) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_conv2d_host: bias_dev is NULL");
    ConvParams p;
    nm_status_t s = make_params("nm_conv2d_host", w, x_dev, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h,
                                dil_w, bias_host ? bias_dev : nullptr, relu, y_dev, &p);
    if (s != NM_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const size_t xb = static_cast<size_t>(batch) * h * wd * w->c_in * sizeof(float);
    const size_t yb = static_cast<size_t>(p.pixels) * w->c_out * sizeof(float);
    cudaError_t e = cudaMemcpyAsync(x_dev, x_host, xb, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && bias_host)
        e = cudaMemcpyAsync(bias_dev, bias_host, static_cast<size_t>(w->c_out) * sizeof(float), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_conv2d_host: H2D copy: %s", cudaGetErrorString(e));
    s = run_plan(p, plan, st);
    if (s != NM_OK) return s;
    e = cudaMemcpyAsync(y_host, y_dev, yb, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_conv2d_host: D2H copy: %s", cudaGetErrorString(e));
    return NM_OK;
}

nm_status_t nm_plan_key(int c_out, int kh, int kw, int c_in, int n_keep, int m_group, int tile_t, int batch, int h, int wd,
                        int stride_h, int stride_w, int pad_h, int pad_w, int dil_h, int dil_w, int has_bias, int relu,
                        char* key, size_t key_bytes)
{
    if (!key || key_bytes == 0) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_key: key buffer missing");
    const int n = std::snprintf(key, key_bytes, "co%d_k%dx%d_ci%d_nm%d:%d_t%d_b%d_hw%dx%d_s%dx%d_p%dx%d_d%dx%d_bias%d_relu%d", c_out, kh,
                                kw, c_in, n_keep, m_group, tile_t, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w,
                                has_bias ? 1 : 0, relu ? 1 : 0);
    if (n < 0 || static_cast<size_t>(n) >= key_bytes) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_key: key buffer too small");
    return NM_OK;
}

nm_status_t nm_plan_cache_store(const char* path, const char* key, const nm_plan_t* plan)
{
    if (!path || !key || !plan || !key[0] || std::strpbrk(key, " \t\n"))
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_cache_store: path, key (no blanks) and plan are required");
    std::FILE* f = std::fopen(path, "a");
    if (!f) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_cache_store: cannot open %s", path);
    const int n = std::fprintf(f, "%s %d %d %d %d %d %d %d %d\n", key, plan->variant, plan->bn, plan->stages, plan->split, plan->kblk,
                               plan->loads, plan->issuers, plan->ksplit);
    const bool ok = n > 0 && std::fclose(f) == 0;
    if (!ok) return nmhost::fail(NM_ERR_INTERNAL, "nm_plan_cache_store: write to %s failed", path);
    return NM_OK;
}

nm_status_t nm_plan_cache_lookup(const char* path, const char* key, nm_plan_t* plan)
{
    if (!path || !key || !plan) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_plan_cache_lookup: path, key and plan are required");
    std::FILE* f = std::fopen(path, "r");
    if (!f) return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_plan_cache_lookup: no cache file %s", path);
    char line[512], k[384];
    bool found = false;
    nm_plan_t p;
    while (std::fgets(line, sizeof(line), f)) {
        std::memset(&p, 0, sizeof(p));
        if (std::sscanf(line, "%383s %d %d %d %d %d %d %d %d", k, &p.variant, &p.bn, &p.stages, &p.split, &p.kblk, &p.loads,
                        &p.issuers, &p.ksplit) == 9 &&
            std::strcmp(k, key) == 0) {
            *plan = p;      // the last line of a key wins
            found = true;
        }
    }
    std::fclose(f);
    if (!found) return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_plan_cache_lookup: no entry for %s", key);
    return NM_OK;
}

}  // extern "C"

namespace {

// nm_autotune; *rank_ms (may be NULL): the time by which the candidates were compared, for a cached plan measured in the same way.
nm_status_t tune(nm_weights_t* w, const float* x, int batch, int h, int wd, int stride_h, int stride_w, int pad_h, int pad_w,
                 int dil_h, int dil_w, const float* bias, int relu, float* y_scratch, void* cuda_stream, nm_plan_t* best,
                 float* best_ms, float* rank_ms)
{
    if (!best) return nmhost::fail(NM_ERR_INVALID_ARG, "nm_autotune: best is NULL");
    ConvParams p;
    nm_status_t s = make_params("nm_autotune", w, x, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w,
                                bias, relu, y_scratch, &p);
    if (s != NM_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // Layers with fewer work items than SMs and a long reduction axis are also tried with the axis
    // split over several CTAs; the partial sums need scratch memory, which belongs to the handle
    // and is reserved here (nm_conv2d itself never allocates).
    {
        nm_weights* hw = w;
        int n_sm = 148, dev = 0;
        if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        const long long pix_blocks = (p.pixels + 127) / 128;
        const bool few_items = pix_blocks * ((p.c_out + 255) / 256) < n_sm && p.k / 32 >= 32;
        size_t need = few_items && (p.wx || p.w3) ? nmhost::expand_splitk_bytes(p, 4) : 0;
        // ... and layers with fewer than three rounds of work items with (item, stage) ranges balanced over the SMs
        const bool uneven = pix_blocks * ((p.c_out + 255) / 256) < 3ll * n_sm;
        if (uneven && p.wx && nmhost::expand_balanced_bytes(256) > need) need = nmhost::expand_balanced_bytes(256);
        if (need > hw->splitk_bytes) (void)nm_weights_reserve(hw, need);   // no scratch: the split plans are simply not candidates
        p.splitk = hw->splitk;
        p.splitk_bytes = hw->splitk_bytes;
    }
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
        if (e0) cudaEventDestroy(e0);
        return nmhost::fail(NM_ERR_CUDA, "nm_autotune: cannot create events");
    }
    // A layer is timed as a network meets it.  Where its input and output together stay well inside the L2, they are still there from
    // the layer before, and a launch overlaps its neighbours' ends: bursts of launches.  Larger layers are timed one launch at a time
    // and cold: a buffer larger than the L2 is overwritten first (without the buffer the launches run warm).  With cold launches
    // for all, whole networks came to 226 us instead of 207 (ResNet-18 1:4, batch 8) and 312 instead of 300 (ResNet-50, batch 1); with bursts for
    // all, ResNet-101 at batch 128 sometimes got plans 9 % slower.  The time reported is the best plan's, cold.
    constexpr double kNearBytes = 64e6;
    constexpr int kBurst = 10;
    const bool near = 4.0 * (static_cast<double>(batch) * h * wd * w->c_in + static_cast<double>(p.pixels) * w->c_out) <= kNearBytes;
    constexpr size_t kFlushBytes = size_t(288) << 20;
    void* flush = nullptr;
    (void)nmhost::device_malloc(&flush, kFlushBytes);   // (NULL where there is no room)
    constexpr int kWarm = 2, kReps = 9, kBurstReps = 5;
    float best_t = -1.f;
    // One launch, cold, or the mean of a burst; false when a launch fails.
    auto measure = [&](const nm_plan_t& plan, int launches, std::vector<float>* t) {
        if (launches == 1 && flush) cudaMemsetAsync(flush, static_cast<int>(t->size()), kFlushBytes, st);
        cudaEventRecord(e0, st);
        bool ok = true;
        for (int k = 0; k < launches && ok; ++k) ok = run_plan(p, &plan, st) == NM_OK;
        cudaEventRecord(e1, st);
        if (cudaEventSynchronize(e1) != cudaSuccess) ok = false;
        float ms = 0.f;
        if (ok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess) t->push_back(ms / static_cast<float>(launches));
        return ok;
    };
    // Median over a plan's launches or bursts, by which candidates are compared; negative when it does not run.  `reach`: three
    // launches, or one burst, tell a candidate that is slower than this (tuning a layer takes half the time this way).
    auto rank = [&](const nm_plan_t& plan, float reach) {
        bool ok = true;
        for (int i = 0; i < kWarm && ok; ++i) ok = run_plan(p, &plan, st) == NM_OK;
        if (!ok || cudaStreamSynchronize(st) != cudaSuccess) return -1.f;
        std::vector<float> t;
        for (int i = 0; i < (near ? kBurstReps : kReps) && ok; ++i) {
            if (t.size() == (near ? 1u : 3u) && reach > 0.f && *std::min_element(t.begin(), t.end()) > reach) break;
            ok = measure(plan, near ? kBurst : 1, &t);
        }
        if (!ok || t.empty()) return -1.f;
        std::sort(t.begin(), t.end());
        return t[t.size() / 2];
    };
    // plan cache: a cached plan that still runs on this layer is returned with its time over three launches
    char key[384] = "";
    const char* cache = std::getenv("NM_PLAN_CACHE");
    if (cache && cache[0] &&
        nm_plan_key(w->c_out, w->kh, w->kw, w->c_in, w->n_keep, w->m_group, w->tile_t, batch, h, wd, stride_h, stride_w, pad_h,
                    pad_w, dil_h, dil_w, bias != nullptr, relu, key, sizeof(key)) == NM_OK) {
        nm_plan_t cached;
        if (nm_plan_cache_lookup(cache, key, &cached) == NM_OK) {
            size_t need = 0;
            if (nm_plan_scratch_bytes(w, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, &cached, &need) == NM_OK &&
                (need <= w->splitk_bytes || nm_weights_reserve(w, need) == NM_OK)) {
                p.splitk = w->splitk;
                p.splitk_bytes = w->splitk_bytes;
                bool ok = run_plan(p, &cached, st) == NM_OK && cudaStreamSynchronize(st) == cudaSuccess;
                float ms = 0.f;
                if (ok) {
                    cudaEventRecord(e0, st);
                    for (int i = 0; i < 3 && ok; ++i) ok = run_plan(p, &cached, st) == NM_OK;
                    cudaEventRecord(e1, st);
                    ok = ok && cudaEventSynchronize(e1) == cudaSuccess && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
                }
                if (ok) {
                    *best = cached;
                    if (best_ms) *best_ms = ms / 3.f;
                    if (rank_ms) *rank_ms = rank(cached, -1.f);
                    if (flush) cudaFree(flush);
                    cudaEventDestroy(e0);
                    cudaEventDestroy(e1);
                    return nm_weights_check(w, cuda_stream);
                }
            }
            (void)cudaGetLastError();
        }
    }
    for (const nm_plan_t& cand : candidate_plans(w, p)) {
        const float med = rank(cand, best_t > 0.f ? 1.25f * best_t : -1.f);
        if (med < 0.f) continue;
        // candidates come most promising first: a later one must win by more than the timing noise
        if (best_t < 0.f || med < best_t * 0.99f) {
            best_t = med;
            *best = cand;
        }
    }
    if (rank_ms) *rank_ms = best_t;
    if (near && best_t >= 0.f) {
        std::vector<float> t;
        for (int i = 0; i < kReps; ++i)
            if (!measure(*best, 1, &t)) break;
        if (!t.empty()) {
            std::sort(t.begin(), t.end());
            best_t = t[t.size() / 2];
        }
    }
    if (flush) cudaFree(flush);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (best_t < 0.f) return nmhost::fail(NM_ERR_UNSUPPORTED, "nm_autotune: no candidate plan ran");
    if (best_ms) *best_ms = best_t;
    if (cache && cache[0] && key[0]) (void)nm_plan_cache_store(cache, key, best);
    return nm_weights_check(w, cuda_stream);
}

}  // namespace

extern "C" {

nm_status_t nm_autotune(nm_weights_t* w, const float* x, int batch, int h, int wd, int stride_h, int stride_w,
                        int pad_h, int pad_w, int dil_h, int dil_w, const float* bias, int relu, float* y_scratch,
                        void* cuda_stream, nm_plan_t* best, float* best_ms)
{
    return tune(w, x, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, bias, relu, y_scratch, cuda_stream, best, best_ms,
                nullptr);
}

nm_status_t nm_autotune_tile(const float* w_dense, int c_out, int kh, int kw, int c_in, int n_keep, int m_group,
                             const int* tile_candidates, int n_candidates, const float* x, int batch, int h, int wd,
                             int stride_h, int stride_w, int pad_h, int pad_w, int dil_h, int dil_w, const float* bias,
                             int relu, float* y_scratch, void* cuda_stream, int* best_tile, nm_plan_t* best,
                             float* best_ms)
{
    if (!tile_candidates || n_candidates < 1 || !best_tile || !best)
        return nmhost::fail(NM_ERR_INVALID_ARG, "nm_autotune_tile: candidates / outputs missing");
    float best_t = -1.f, reported = 0.f;
    nm_status_t last = NM_ERR_UNSUPPORTED;
    for (int i = 0; i < n_candidates; ++i) {
        nm_weights_t* hnd = nullptr;
        last = nm_prune(w_dense, c_out, kh, kw, c_in, n_keep, m_group, tile_candidates[i], cuda_stream, &hnd);
        if (last != NM_OK) continue;
        nm_plan_t plan;
        float ms = 0.f, rank_ms = -1.f;
        last = tune(hnd, x, batch, h, wd, stride_h, stride_w, pad_h, pad_w, dil_h, dil_w, bias, relu, y_scratch, cuda_stream, &plan, &ms,
                    &rank_ms);
        nm_weights_free(hnd);
        if (last != NM_OK || rank_ms < 0.f) continue;
        // widths are compared by what their plans were compared by, not by the reported time (cold, or a cached plan's few launches)
        if (best_t < 0.f || rank_ms < best_t) {
            best_t = rank_ms;
            reported = ms;
            *best_tile = tile_candidates[i];
            *best = plan;
        }
    }
    if (best_t < 0.f) return last == NM_OK ? nmhost::fail(NM_ERR_UNSUPPORTED, "nm_autotune_tile: nothing ran") : last;
    if (best_ms) *best_ms = reported;
    return NM_OK;
}

const char* nm_status_string(nm_status_t s)
{
    switch (s) {
        case NM_OK: return "NM_OK";
        case NM_ERR_INVALID_ARG: return "NM_ERR_INVALID_ARG";
        case NM_ERR_UNSUPPORTED: return "NM_ERR_UNSUPPORTED";
        case NM_ERR_CUDA: return "NM_ERR_CUDA";
        case NM_ERR_ALLOC: return "NM_ERR_ALLOC";
        case NM_ERR_TIMEOUT: return "NM_ERR_TIMEOUT";
        case NM_ERR_INTERNAL: return "NM_ERR_INTERNAL";
    }
    return "NM_ERR_UNKNOWN";
}

const char* nm_last_error(void) { return g_err; }

uint64_t nm_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

}  // extern "C"
