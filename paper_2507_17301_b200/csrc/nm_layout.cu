// Memory of the weight handles and construction of the kernel-side copies of the compressed form.
//
// A handle is ONE device allocation: the canonical values / indices, the status word and every layout the
// convolution kernels read are carved out of it.  (Fourteen cudaMalloc / cudaFree calls per handle used to be nearly all of
// nm_prune's time: 3.1 ms for a 512 x 3 x 3 x 512 layer whose kernels take about 0.1 ms.)  Blocks of freed handles
// are kept for the next one, within bounds: at most kCacheBytes per process, none that kCacheAge later frees did not
// want, all of them returned to the driver before an allocation of the library is reported as failed and when
// nm_memory_trim asks for it.  A block enters the cache only
// after its device has been synchronised, so whoever takes it next may use it on any stream; the list is guarded by a
// mutex.
//
// All layouts are written by ONE kernel from the index array and the values (k_build_layouts), after one memset of those
// that have padding or pruned columns: a thread decodes a retained column once and stores the values of a few rows to each of
// them.  It is bound by the writes (28 MB for 512 x 3 x 3 x 512 at 2:4).
#include <algorithm>
#include <mutex>
#include <vector>

#include "nm_internal.h"
#include "nm_ptx.cuh"

namespace {

constexpr size_t kCacheBytes = size_t(256) << 20;
constexpr uint64_t kCacheAge = 64;

struct Block {
    void* ptr;
    size_t bytes;
    int device;
    uint64_t stamp;   // number of the free that put it here
};
std::mutex g_mu;
std::vector<Block> g_cache;
size_t g_cached = 0;
uint64_t g_frees = 0;

size_t rounded(size_t bytes)
{
    const size_t unit = bytes < (size_t(1) << 20) ? size_t(1) << 16 : size_t(1) << 20;
    return (bytes + unit - 1) / unit * unit;
}

// Gives the i-th cached block back to the driver (g_mu held; cudaFree takes pointers of any device).
void drop(size_t i)
{
    cudaFree(g_cache[i].ptr);
    g_cached -= g_cache[i].bytes;
    g_cache.erase(g_cache.begin() + static_cast<long>(i));
}

void drop_all()
{
    while (!g_cache.empty()) drop(g_cache.size() - 1);
}

// Pinned words for the few bytes a creating call reads back (L1 masses, validity): pageable memory would make the
// copy take a staging detour.  A caller that finds no free slot uses pageable memory.
constexpr int kSlots = 32;
struct Readback {
    double mass[2];
    int bad;
};
std::mutex g_slot_mu;
Readback* g_slots = nullptr;
bool g_slots_tried = false;
uint32_t g_slot_used = 0;

Readback* take_slot()
{
    std::lock_guard<std::mutex> lock(g_slot_mu);
    if (!g_slots_tried) {
        g_slots_tried = true;
        if (cudaHostAlloc(reinterpret_cast<void**>(&g_slots), kSlots * sizeof(Readback), cudaHostAllocPortable) != cudaSuccess) {
            (void)cudaGetLastError();
            g_slots = nullptr;
        }
    }
    if (!g_slots) return nullptr;
    for (int i = 0; i < kSlots; ++i)
        if (!(g_slot_used >> i & 1u)) {
            g_slot_used |= 1u << i;
            return g_slots + i;
        }
    return nullptr;
}
void give_slot(Readback* s)
{
    std::lock_guard<std::mutex> lock(g_slot_mu);
    g_slot_used &= ~(1u << (s - g_slots));
}

struct LayoutArgs {
    const float* src;            // dense weights [c_out][k] (import = 0) or retained values [c_out][kk] (import = 1)
    const uint16_t* idx;         // [n_tiles][kk]
    int import;
    int c_out, k, kk, kk_pad, tile_t, n_tiles, n_keep, m_group, c_in, kh, kw;
    float* values;
    uint16_t* indices;           // import: the handle's copy of idx
    float* wt;
    uint32_t* taps;
    float* wt2; uint8_t* rel2; int v2_s, v2_kc, v2_chunks;         // NULL: not built
    float* wx; int wx_rows;
    float* w3; uint8_t* sel3; int sel_s, sel_kc;
    float* ws;
    int* bad;
};

// Place of retained column e of a select step among the step's `kc` columns, given by their indices `idx`: quads of columns
// that differ modulo 4 as far as the columns allow (the kernel loads a quad at a time, and columns equal modulo 4 share
// their banks).  The i-th column of a class (its index modulo 4) goes to quad i; what a class has beyond the number of quads fills
// the places the others leave, from the last quad down.
__device__ int select_place(const uint16_t* idx, int kc, int e)
{
    const int quads = kc / 4;
    uint32_t count = 0;   // of the four classes, a byte each
    int left_over = 0, place = -1;
#pragma unroll 8
    for (int i = 0; i < kc; ++i) {
        const uint32_t cls = idx[i] & 3u;
        const int rank = static_cast<int>(count >> (8 * cls) & 255u);
        count += 1u << (8 * cls);
        if (i == e && rank < quads) place = rank * 4 + static_cast<int>(cls);
        left_over += rank >= quads && i < e ? 1 : 0;
    }
    if (place >= 0) return place;
    for (int quad = quads - 1; quad >= 0; --quad)
        for (int c = 0; c < 4; ++c)
            if (static_cast<int>(count >> (8 * c) & 255u) <= quad && left_over-- == 0) return quad * 4 + c;
    return 0;   // (not reached: as many free places as columns left over)
}

constexpr int ROWS = 8;   // output channels per thread: a column is decoded and placed once for all of them (512 x 3 x 3 x 512: 106 us with one, 85 with 4, 82)

// One thread per (retained column or padding column, ROWS output channels of a tile).
__global__ void k_build_layouts(const LayoutArgs a)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int parts = (a.tile_t + ROWS - 1) / ROWS;
    const int r = blockIdx.y / parts, rr0 = (blockIdx.y - r * parts) * ROWS;
    const bool first_row = rr0 == 0;   // this thread also writes what the tile's rows share
    if (j >= a.kk_pad) return;
    if (j >= a.kk) {
        if (first_row) a.taps[static_cast<size_t>(r) * a.kk_pad + j] = NM_TAP_PAD;
        return;
    }
    const uint16_t* idx = a.idx + static_cast<size_t>(r) * a.kk;
    const int col = idx[j];
    if (a.import) {
        // strictly ascending below K, and retained column j in group j / N of M consecutive columns (a tail group of
        // m' < M columns keeps min(N, m'), which the same quotient covers); nothing is stored for a bad column
        const bool bad = col >= a.k || col / a.m_group != j / a.n_keep;
        if (first_row && (bad || (j > 0 && idx[j - 1] >= col))) atomicExch(a.bad, 1);
        if (first_row) a.indices[static_cast<size_t>(r) * a.kk + j] = static_cast<uint16_t>(col);
        if (bad) return;
    }
    const int tap = col / a.c_in, c = col - tap * a.c_in;
    if (first_row)
        a.taps[static_cast<size_t>(r) * a.kk_pad + j] =
            (static_cast<uint32_t>(tap / a.kw) << 24) | (static_cast<uint32_t>(tap % a.kw) << 16) | static_cast<uint32_t>(c);

    // slab layout: kept column j lies in chunk col / S at position j - chunk * KC (every group before the last is
    // full, so a chunk of whole groups holds exactly KC kept columns)
    const size_t pitch2 = static_cast<size_t>(a.v2_chunks) * 32;
    size_t at2 = 0;
    if (a.wt2) {
        const int chunk = col / a.v2_s, jj = j - chunk * a.v2_kc;
        at2 = static_cast<size_t>(chunk) * 32 + jj;
        if (first_row) a.rel2[static_cast<size_t>(r) * pitch2 + at2] = static_cast<uint8_t>(col - chunk * a.v2_s);
    }
    // select layout: w3[chunk][o][32], a chunk being as many steps (one tap of S source columns, of which KC are kept) as fit,
    // the steps ordered by block of S channels, then tap; swizzled like wx.  The
    // column tables hold, per chunk and tile, the byte offset of each column in its 128-byte row (and its 32-channel block in
    // bit 7 and up), in the order in which a thread reads them: [step][place in a quad][quad].
    int chunk3 = 0, k3 = 0;
    if (a.w3) {
        const int spc = 32 / a.sel_kc, cb = c / a.sel_s, cc = c - cb * a.sel_s, n_cb = a.c_in / a.sel_s;
        const int step = cb * a.kh * a.kw + tap, sub = step % spc;
        chunk3 = step / spc;
        const int js = (tap * n_cb + cb) * a.sel_kc;   // the step's first retained column
        const int place = select_place(idx + js, a.sel_kc, j - js);
        k3 = sub * a.sel_kc + (place >> 3) * 8 + (place & 3) * 2 + (place >> 2 & 1);   // (a thread's columns of two quads are neighbours)
        if (first_row) {
            reinterpret_cast<uint32_t*>(a.sel3)[(static_cast<size_t>(chunk3) * a.n_tiles + r) * 32 + sub * a.sel_kc + (place & 3) * (a.sel_kc / 4) + (place >> 2)] =
                static_cast<uint32_t>((cc & 31) * 4 | (cc >> 5) << 7);
        }
    }
    // plane layout: ws[kh][c_out][32]: a row holds the taps of one kernel row as (kw, c), c padded to 4 and kw to 8,
    // its 16-byte pieces (one tap each) XOR-ed with (o % 8)
    const int khi = tap / a.kw, kwi = tap - khi * a.kw;

    for (int rr = rr0; rr < min(rr0 + ROWS, a.tile_t); ++rr) {
        const int o = r * a.tile_t + rr;
        if (o >= a.c_out) break;
        const float v = a.import ? a.src[static_cast<size_t>(o) * a.kk + j] : a.src[static_cast<size_t>(o) * a.k + col];
        const float t = nmk::to_tf32(v);
        a.values[static_cast<size_t>(o) * a.kk + j] = v;
        {
            // gather layout: per (tile, chunk of 32 retained columns) the shared-memory image of the tile's rows, swizzled like wx;
            // as many rows as the tile has, so it is as large as the values whatever the tile width (padded to the MMA's 16 rows,
            // 512 x 3 x 3 x 512 at 2:4 and T = 1 took 75 MB here instead of 4.7)
            const int jj = j & (NM_KCHUNK - 1), rows = min(a.tile_t, a.c_out - r * a.tile_t);
            a.wt[static_cast<size_t>(r) * a.tile_t * a.kk_pad + (static_cast<size_t>(j / NM_KCHUNK) * rows + rr) * NM_KCHUNK + ((((jj >> 2) ^ (rr & 7)) << 2) | (jj & 3))] = t;
        }
        if (a.wt2) a.wt2[static_cast<size_t>(o) * pitch2 + at2] = t;
        if (a.wx) {
            // expanded layout: the shared-memory image the tensor core reads: blocks of 32 columns, inside a block one
            // 128-byte row per output channel whose 16-byte pieces are XOR-ed with (o % 8) (the 128-byte swizzle), so that
            // any run of channels starting at a multiple of 8 is one contiguous bulk copy
            const int blk = col >> 5, kc = col & 31;
            a.wx[(static_cast<size_t>(blk) * a.wx_rows + o) * 32 + ((((kc >> 2) ^ (o & 7)) << 2) | (kc & 3))] = t;
        }
        if (a.w3) a.w3[(static_cast<size_t>(chunk3) * a.c_out + o) * 32 + ((((k3 >> 2) ^ (o & 7)) << 2) | (k3 & 3))] = t;
        if (a.ws) a.ws[(static_cast<size_t>(khi) * a.c_out + o) * 32 + ((kwi ^ (o & 7)) << 2) + c] = t;
    }
}

}  // namespace

namespace nmhost {

bool kernel_may_touch(const void* a, const void* b, int device)
{
    int current = -1;
    if (cudaGetDevice(&current) != cudaSuccess || current != device) return false;
    for (const void* ptr : {a, b}) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, ptr) != cudaSuccess) {
            (void)cudaGetLastError();
            return false;
        }
        if (!kernel_may_touch(at.type, at.device, current)) return false;
    }
    return true;
}

void* device_block_alloc(size_t bytes, int device, size_t* got)
{
    const size_t want = rounded(bytes);
    std::lock_guard<std::mutex> lock(g_mu);
    size_t best = g_cache.size();
    for (size_t i = 0; i < g_cache.size(); ++i)
        if (g_cache[i].device == device && g_cache[i].bytes >= want && g_cache[i].bytes <= want + want / 4 + (size_t(1) << 20) &&
            (best == g_cache.size() || g_cache[i].bytes < g_cache[best].bytes))
            best = i;
    if (best < g_cache.size()) {
        void* p = g_cache[best].ptr;
        *got = g_cache[best].bytes;
        g_cached -= *got;
        g_cache.erase(g_cache.begin() + static_cast<long>(best));
        return p;
    }
    void* p = nullptr;
    if (cudaMalloc(&p, want) != cudaSuccess) {
        (void)cudaGetLastError();
        drop_all();   // before giving up
        if (cudaMalloc(&p, want) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
    }
    *got = want;
    return p;
}

void device_blocks_trim()
{
    std::lock_guard<std::mutex> lock(g_mu);
    drop_all();
}

cudaError_t device_malloc(void** ptr, size_t bytes)
{
    cudaError_t e = cudaMalloc(ptr, bytes);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        device_blocks_trim();
        e = cudaMalloc(ptr, bytes);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            *ptr = nullptr;
        }
    }
    return e;
}

void device_block_free(void* ptr, size_t bytes, int device, bool idle)
{
    if (!ptr) return;
    std::lock_guard<std::mutex> lock(g_mu);
    ++g_frees;
    if (!idle || bytes > kCacheBytes / 2) {
        cudaFree(ptr);
    } else {
        g_cache.push_back({ptr, bytes, device, g_frees});
        g_cached += bytes;
    }
    // oldest first: the list is in the order of the frees
    while (!g_cache.empty() && (g_cached > kCacheBytes || g_cache.front().stamp + kCacheAge < g_frees)) drop(0);
}

// Which layouts this layer's kernels can read, and their dimensions (no device work).
static void plan_layouts(nm_weights* h)
{
    // slab layout: keep-all is the 1:1 pattern; otherwise the chunk is the largest whole number of groups whose kept
    // columns number a multiple of 8 up to 32 and whose source columns number <= 64
    const int n = h->n_keep == h->m_group ? 1 : h->n_keep;
    const int m = h->n_keep == h->m_group ? 1 : h->m_group;
    for (int g = 32 / n; g >= 1 && h->kk > 0; --g)
        if ((g * n) % 8 == 0 && g * m <= 64) {
            h->v2_ok = 1;
            h->v2_g = g; h->v2_kc = g * n; h->v2_s = g * m;
            h->v2_chunks = (h->k + h->v2_s - 1) / h->v2_s;
            break;
        }
    // expanded layout: only shapes the kernels that read it take: output channels in whole float4s (rows are padded
    // with zeros to blocks of 32), and either whole 32-column slabs (expanded-operand kernel) or a short reduction axis
    // (row-run kernel, pointwise layers)
    if (h->c_out % 4 == 0 && h->kk > 0 && (h->c_in % 32 == 0 || h->k <= 512)) h->wx_rows = (h->c_out + 31) / 32 * 32;
    int s = 0, kc = 0;
    if (select_layout_dims(h, &s, &kc)) {
        const int spc = 32 / kc, steps = h->c_in / s * h->kh * h->kw;
        h->sel_s = s;
        h->sel_kc = kc;
        h->sel_chunks = (steps + spc - 1) / spc;
    }
}

nm_status_t alloc_handle_memory(nm_weights* h, const char* who)
{
    plan_layouts(h);
    const bool planes = h->c_in <= 4 && h->kw <= 8 && h->c_out % 32 == 0 && h->c_out <= 256 && h->kk > 0 &&
                        h->kh * h->c_out * 128 < (1 << 20);
    size_t total = 0;
    auto place = [&total](size_t bytes) {
        const size_t at = total;
        total += (std::max<size_t>(bytes, 16) + 255) / 256 * 256;
        return at;
    };
    const size_t kk1 = static_cast<size_t>(std::max(h->kk, 1));
    const size_t pitch2 = static_cast<size_t>(h->v2_chunks) * 32;
    const size_t chunks3 = static_cast<size_t>(h->sel_chunks);
    const size_t at_values = place(h->c_out * kk1 * sizeof(float));
    const size_t at_indices = place(h->n_tiles * kk1 * sizeof(uint16_t));
    const size_t at_taps = place(static_cast<size_t>(h->n_tiles) * h->kk_pad * sizeof(uint32_t));
    // Layouts that every word of is written come before the part of the block that the creating call clears (status, sums and layouts with
    // padding or zeros in the pruned columns): 512 x 3 x 3 x 512 at 2:4 has 9 of 24 MB to clear, 58 -> 51 us.
    const int spc = h->sel_s ? 32 / h->sel_kc : 1;
    const bool full_wt = h->kk % NM_KCHUNK == 0;
    const bool full_wt2 = h->v2_kc == 32 && h->k % std::max(h->v2_s, 1) == 0;
    const bool full_w3 = h->sel_s && h->sel_kc * spc == 32 && h->k / h->sel_s % spc == 0;
    size_t at_status = 0, at_mass = 0, at_wt = 0, at_wt2 = 0, at_rel2 = 0, at_wx = 0, at_w3 = 0, at_sel3 = 0, at_ws = 0;
    for (const bool full : {true, false}) {
        if (!full) {
            h->zero_from = total;
            at_status = place(4 * sizeof(int));
            at_mass = place(sizeof(Readback));
        }
        if (full_wt == full) at_wt = place(static_cast<size_t>(h->c_out) * h->kk_pad * sizeof(float));
        if (full_wt2 == full) {
            at_wt2 = place(h->v2_ok ? h->c_out * pitch2 * sizeof(float) : 0);
            at_rel2 = place(h->v2_ok ? h->n_tiles * pitch2 : 0);
        }
        if (full_w3 == full) {
            at_w3 = place(chunks3 * h->c_out * 128);
            at_sel3 = place(chunks3 * h->n_tiles * 128);
        }
    }
    at_wx = place(h->wx_rows ? static_cast<size_t>((h->k + 31) / 32) * h->wx_rows * 128 : 0);
    at_ws = place(planes ? static_cast<size_t>(h->kh) * h->c_out * 128 : 0);
    h->block_used = total;
    h->block = static_cast<uint8_t*>(device_block_alloc(total, h->device, &h->block_bytes));
    if (!h->block) return fail(NM_ERR_ALLOC, "%s: cannot allocate %zu bytes on the device", who, total);
    h->values = reinterpret_cast<float*>(h->block + at_values);
    h->indices = reinterpret_cast<uint16_t*>(h->block + at_indices);
    h->wt = reinterpret_cast<float*>(h->block + at_wt);
    h->taps = reinterpret_cast<uint32_t*>(h->block + at_taps);
    h->status = reinterpret_cast<int*>(h->block + at_status);
    h->mass = reinterpret_cast<double*>(h->block + at_mass);
    if (h->v2_ok) {
        h->wt2 = reinterpret_cast<float*>(h->block + at_wt2);
        h->rel2 = h->block + at_rel2;
    }
    if (h->wx_rows) h->wx = reinterpret_cast<float*>(h->block + at_wx);
    if (h->sel_s) {
        h->w3 = reinterpret_cast<float*>(h->block + at_w3);
        h->sel3 = h->block + at_sel3;
    }
    if (planes) h->ws = reinterpret_cast<float*>(h->block + at_ws);
    return NM_OK;
}

nm_status_t clear_handle_memory(nm_weights* h, cudaStream_t st)
{
    const cudaError_t e = cudaMemsetAsync(h->block + h->zero_from, 0, h->block_used - h->zero_from, st);
    return e == cudaSuccess ? NM_OK : fail(NM_ERR_CUDA, "clearing the handle's memory: %s", cudaGetErrorString(e));
}

nm_status_t build_layouts(nm_weights* h, const float* src, const uint16_t* idx, bool import, cudaStream_t st)
{
    LayoutArgs a = {};
    a.src = src; a.idx = idx; a.import = import ? 1 : 0;
    a.c_out = h->c_out; a.k = h->k; a.kk = h->kk; a.kk_pad = h->kk_pad; a.tile_t = h->tile_t; a.n_tiles = h->n_tiles;
    a.n_keep = h->n_keep; a.m_group = h->m_group; a.c_in = h->c_in; a.kh = h->kh; a.kw = h->kw;
    a.values = h->values; a.indices = h->indices; a.wt = h->wt; a.taps = h->taps;
    a.wt2 = h->wt2; a.rel2 = h->rel2; a.v2_s = h->v2_s; a.v2_kc = h->v2_kc; a.v2_chunks = h->v2_chunks;
    a.wx = h->wx; a.wx_rows = h->wx_rows;
    a.w3 = h->w3; a.sel3 = h->sel3; a.sel_s = h->sel_s; a.sel_kc = h->sel_kc;
    a.ws = h->ws;
    a.bad = &reinterpret_cast<Readback*>(h->mass)->bad;
    if (h->c_out > 65535) return fail(NM_ERR_CUDA, "weight layout kernel: more than 65535 output channels");   // bounds grid.y
    if (h->kk_pad > 0) {
        const dim3 grid((h->kk_pad + 127) / 128, h->n_tiles * ((h->tile_t + ROWS - 1) / ROWS));
        k_build_layouts<<<grid, 128, 0, st>>>(a);
        count_launch(1);
    }
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NM_OK : fail(NM_ERR_CUDA, "weight layout kernel: %s", cudaGetErrorString(e));
}

nm_status_t finish_handle(nm_weights* h, cudaStream_t st, double* mass2, int* bad)
{
    Readback local = {};
    Readback* slot = take_slot();
    Readback* dst = slot ? slot : &local;
    cudaError_t e = cudaMemcpyAsync(dst, h->mass, sizeof(Readback), cudaMemcpyDeviceToHost, st);
    const cudaError_t e2 = cudaStreamSynchronize(st);
    if (e == cudaSuccess) e = e2;
    const Readback got = *dst;
    if (slot) give_slot(slot);
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "building the weight handle: %s", cudaGetErrorString(e));
    if (mass2) { mass2[0] = got.mass[0]; mass2[1] = got.mass[1]; }
    if (bad) *bad = got.bad;
    return NM_OK;
}

}  // namespace nmhost
