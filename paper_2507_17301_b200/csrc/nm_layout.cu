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
// With groups of at most 128 columns a handle is built by ONE kernel (k_compress): a block owns a span of whole groups of one tile
// (up to 64 of its rows), reads that piece of the dense weights (import: of the retained values) once into shared memory, selects
// the columns there, and writes the piece's part of every layout, zeros of the expanded one included.  Wider groups are
// selected by the kernels of nm_prune.cu, and k_build_layouts writes the layouts from the index array after a memset; the layouts' rules
// are functions that both share.  k_compress writes 28 MB for 512 x 3 x 3 x 512 at 2:4 in 12 us, 2.3 TB/s: its blocks fit one wave and go
// through loading, scoring, placing and writing in step, so memory idles while they score.
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
// What the blocks of a creating call add up, one per pinned slot: zero before and after every call (its last block hands the sums over
// and clears them), so that no call has to.
struct Accum {
    Readback sum;
    unsigned done;
};
__device__ Accum g_accum[kSlots];
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
    int* status;
    Divisor by_c_in, by_kw, by_v2_s;
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

// Tap and channel of column k of a row of weights.
struct Column {
    int tap, c, kh, kw;
};
__device__ __forceinline__ Column column_of(const LayoutArgs& a, int k)
{
    Column at;
    at.tap = div_by(k, a.by_c_in);
    at.c = k - at.tap * a.c_in;
    at.kh = div_by(at.tap, a.by_kw);
    at.kw = at.tap - at.kh * a.kw;
    return at;
}
__device__ __forceinline__ uint32_t tap_word(const Column& at)
{
    return (static_cast<uint32_t>(at.kh) << 24) | (static_cast<uint32_t>(at.kw) << 16) | static_cast<uint32_t>(at.c);
}
// Float of column k in a 128-byte row whose 16-byte pieces are XOR-ed with (row % 8), the 128-byte swizzle.
__device__ __forceinline__ int swizzled(int row, int k) { return (((k >> 2) ^ (row & 7)) << 2) | (k & 3); }
// Gather layout: per (tile, chunk of 32 retained columns) the shared-memory image of the tile's rows; as many rows as the tile has, so it is as
// large as the values whatever the tile width (padded to the MMA's 16 rows, 512 x 3 x 3 x 512 at 2:4 and T = 1 took 75 MB here
// instead of 4.7).  The image of retained column j's chunk:
__device__ __forceinline__ float* gather_image(const LayoutArgs& a, int row0, int tile_rows, int j)
{
    return a.wt + static_cast<size_t>(row0) * a.kk_pad + static_cast<size_t>(j / NM_KCHUNK) * tile_rows * NM_KCHUNK;
}
__device__ __forceinline__ int gather_cell(int row_of_tile, int j) { return row_of_tile * NM_KCHUNK + swizzled(row_of_tile, j & (NM_KCHUNK - 1)); }
// Slab layout: retained column j (source column k) lies in chunk k / S at position j - chunk * KC (every group before the last is full, so a
// chunk of whole groups holds exactly KC kept columns); `rel`: its offset in the chunk's source columns.
__device__ __forceinline__ int slab_place(const LayoutArgs& a, int k, int j, uint8_t* rel)
{
    const int chunk = div_by(k, a.by_v2_s);
    *rel = static_cast<uint8_t>(k - chunk * a.v2_s);
    return chunk * 32 + (j - chunk * a.v2_kc);
}
// Expanded layout: the shared-memory image the tensor core reads: blocks of 32 columns, inside a block one swizzled row per output channel, so
// that any run of channels starting at a multiple of 8 is one contiguous bulk copy.
__device__ __forceinline__ float* expanded_cell(const LayoutArgs& a, int o, int k)
{
    return a.wx + (static_cast<size_t>(k >> 5) * a.wx_rows + o) * 32 + swizzled(o, k & 31);
}
// Plane layout: ws[kh][c_out][32]: a row holds the taps of one kernel row as (kw, c), c padded to 4 and kw to 8, swizzled.
__device__ __forceinline__ float* plane_cell(const LayoutArgs& a, int o, int kh, int kw_c) { return a.ws + (static_cast<size_t>(kh) * a.c_out + o) * 32 + swizzled(o, kw_c); }

constexpr int ROWS = 8;   // output channels per thread: a column is decoded and placed once for all of them (512 x 3 x 3 x 512 in groups of 600: 8.2 us with one, 6.1 with four, 5.6)

// Groups wider than a block of k_compress (the select layout has none): one thread per (retained column or padding column, ROWS output
// channels of a tile).
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
    const Column at = column_of(a, col);
    if (first_row) a.taps[static_cast<size_t>(r) * a.kk_pad + j] = tap_word(at);
    const size_t pitch2 = static_cast<size_t>(a.v2_chunks) * 32;
    int at2 = 0;
    if (a.wt2) {
        uint8_t rel;
        at2 = slab_place(a, col, j, &rel);
        if (first_row) a.rel2[static_cast<size_t>(r) * pitch2 + at2] = rel;
    }
    const int row0 = r * a.tile_t, tile_rows = min(a.tile_t, a.c_out - row0);
    float* const wt = gather_image(a, row0, tile_rows, j);
    for (int rr = rr0; rr < min(rr0 + ROWS, tile_rows); ++rr) {
        const int o = row0 + rr;
        const float v = a.import ? a.src[static_cast<size_t>(o) * a.kk + j] : a.src[static_cast<size_t>(o) * a.k + col];
        const float t = nmk::to_tf32(v);
        a.values[static_cast<size_t>(o) * a.kk + j] = v;
        wt[gather_cell(rr, j)] = t;
        if (a.wt2) a.wt2[static_cast<size_t>(o) * pitch2 + at2] = t;
        if (a.wx) *expanded_cell(a, o, col) = t;
        if (a.ws) *plane_cell(a, o, at.kh, at.kw << 2 | at.c) = t;
    }
}

constexpr int SPAN = 128;   // columns of a k_compress block, at most
constexpr int PART = 64;    // rows of a tile that a block writes, at most

// Selection (import: check) and every layout of a span of whole groups, PART rows of one tile.  The selection is the one described at the
// head of nm_prune.cu.  Threads: a column each while scores are summed (the tile's rows in order, PART at a time through shared memory).
// Then 128 threads work out where the retained columns go in every layout, while the others write the expanded layout, whose 128-byte rows
// a warp writes whole; then all write the other layouts, a retained column and every threads >> log_j-th row each.  The last warp
// adds the block's sums to the call's meanwhile (2 us with its fence, when it was part of the others' way).
// 512 x 3 x 3 x 512 at 2:4, T = 64 (28 MB written): 12 us; a memset, a kernel for the selection and one for the layouts took 18 and the
// gaps between them.  nm_prune and export of that layer 66 -> 46 us, import and export of 1024 -> 2048, 1x1 54 -> 45.
template <bool IMPORT>
__global__ void __launch_bounds__(544) k_compress(const LayoutArgs a, int span, int log_j, Readback* sums, int slot, Readback* host)
{
    __shared__ __align__(16) float s_tile[PART][SPAN];
    __shared__ double s_score[SPAN];
    __shared__ uint16_t s_idx[SPAN];   // retained columns of the span, 0xFFFF: a bad one (import)
    __shared__ short s_pos[SPAN];      // place of a column of the span among them, -1: pruned
    __shared__ uint32_t s_at2[SPAN], s_at3[SPAN], s_ats[SPAN];   // places of a retained column in wt2, w3 (chunk, position), ws
    const int tid = threadIdx.x, threads = blockDim.x - 32, r = blockIdx.y, row0 = r * a.tile_t;   // (without the last warp)
    const int c0 = blockIdx.x * span, cols = min(span, a.k - c0);
    const int tile_rows = min(a.tile_t, a.c_out - row0);
    const int p0 = blockIdx.z * PART, rows = max(0, min(PART, tile_rows - p0));   // (none in a short last tile: the block is only counted)
    const int groups = span / a.m_group, j0 = static_cast<int>(blockIdx.x) * groups * a.n_keep;
    const int nk = min(a.kk, j0 + groups * a.n_keep) - j0;
    const bool first = blockIdx.z == 0;   // this block also writes what the tile's rows share
    const int j = tid & ((1 << log_j) - 1);
    if (blockIdx.x == 0 && r == 0 && first && tid < 4) a.status[tid] = 0;

    if (!IMPORT) {
        double score = 0.0;
        const bool quads = ((a.k | span) & 3) == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0;
        auto load = [&](int from) {   // rows [from, from + PART) of the tile
            const int n = min(PART, tile_rows - from);
            const float* src = a.src + static_cast<size_t>(row0 + from) * a.k + c0;
            if (tid >= threads) return;
            if (quads) {
                const int t = (tid & (SPAN / 4 - 1)) * 4;
                if (t < cols)
#pragma unroll 8
                    for (int rr = tid / (SPAN / 4); rr < n; rr += threads / (SPAN / 4))
                        *reinterpret_cast<float4*>(&s_tile[rr][t]) = __ldg(reinterpret_cast<const float4*>(src + static_cast<size_t>(rr) * a.k + t));
            } else {
                const int t = tid & (SPAN - 1);
                if (t < cols)
#pragma unroll 8
                    for (int rr = tid / SPAN; rr < n; rr += threads / SPAN) s_tile[rr][t] = __ldg(src + static_cast<size_t>(rr) * a.k + t);
            }
        };
        int from = 0;
        for (;; from += PART) {
            load(from);
            __syncthreads();
            if (tid < cols) {
                const int n = min(PART, tile_rows - from);
#pragma unroll 8
                for (int rr = 0; rr < n; ++rr) score += fabs(static_cast<double>(s_tile[rr][tid]));
            }
            if (from + PART >= tile_rows) break;
            __syncthreads();
        }
        if (from != p0 && rows > 0) {
            __syncthreads();
            load(p0);
        }
        if (tid < cols) {
            if (!(score == score)) score = static_cast<double>(INFINITY);
            s_score[tid] = score;
        }
        __syncthreads();
        const int g_first = tid / a.m_group * a.m_group;
        bool keep = false;
        if (tid < cols) {
            const int g_end = min(g_first + a.m_group, cols);
            int beaten_by = 0;
            for (int i = g_first; i < g_end; ++i) {
                const double si = s_score[i];
                beaten_by += (si > score) || (si == score && i < tid);
            }
            keep = beaten_by < a.n_keep;
            s_pos[tid] = keep ? 1 : 0;
        }
        __syncthreads();
        int pos = -1;
        if (keep) {
            const int g = tid / a.m_group;
            pos = g * a.n_keep;   // every earlier group is a full one and kept exactly n_keep
            for (int i = g_first; i < tid; ++i) pos += s_pos[i];
            // the order of the scores is total, so a group keeps at most N columns; the bound makes sure that no input
            // whatsoever can place a column outside its group's slots
            if (pos >= min(nk, (g + 1) * a.n_keep)) pos = -1;
        }
        __syncthreads();
        if (tid < cols) s_pos[tid] = static_cast<short>(pos);
        if (pos >= 0) s_idx[pos] = static_cast<uint16_t>(c0 + tid);
    } else {
        if (tid < SPAN) s_pos[tid] = -1;
        __syncthreads();
        if (tid < nk) {
            // strictly ascending below K, and retained column j in group j / N of M consecutive columns (a tail group of
            // m' < M columns keeps min(N, m'), which the same quotient covers); nothing is stored for a bad column
            const uint16_t* idx = a.idx + static_cast<size_t>(r) * a.kk;
            const int jj = j0 + tid, col = idx[jj];
            const bool bad = col >= a.k || col / a.m_group != jj / a.n_keep;
            if (first && (bad || (jj > 0 && idx[jj - 1] >= col))) {
                atomicExch(slot >= 0 ? &g_accum[slot].sum.bad : &sums->bad, 1);
                __threadfence();
            }
            s_idx[tid] = bad ? 0xFFFFu : static_cast<uint16_t>(col);
            if (!bad) s_pos[col - c0] = static_cast<short>(tid);
        }
        const float* src = a.src + static_cast<size_t>(row0 + p0) * a.kk + j0;
        if (tid < threads && j < nk)
#pragma unroll 8
            for (int rr = tid >> log_j; rr < rows; rr += threads >> log_j) s_tile[rr][j] = src[static_cast<size_t>(rr) * a.kk + j];
    }
    __syncthreads();

    if (tid >= threads) {
        // L1 mass of all columns and of the retained ones
        const int lane = tid & 31;
        Readback* const acc = slot >= 0 ? &g_accum[slot].sum : sums;
        if (!IMPORT && first) {
            double all = 0.0, kept = 0.0;
            for (int i = lane; i < cols; i += 32) {
                all += s_score[i];
                if (s_pos[i] >= 0) kept += s_score[i];
            }
            for (int d = 16; d > 0; d >>= 1) {
                all += __shfl_down_sync(0xFFFFFFFFu, all, d);
                kept += __shfl_down_sync(0xFFFFFFFFu, kept, d);
            }
            if (lane == 0) {
                atomicAdd(acc->mass, all);
                atomicAdd(acc->mass + 1, kept);
            }
        }
        if (slot >= 0 && lane == 0) {
            __threadfence();
            if (atomicAdd(&g_accum[slot].done, 1u) + 1 == gridDim.x * gridDim.y * gridDim.z) {
                // the last block to add its sums hands them over (the host reads them once the stream is done)
                __threadfence();
                volatile Accum* const total = &g_accum[slot];
                volatile Readback* const out = host;
                out->mass[0] = total->sum.mass[0];
                out->mass[1] = total->sum.mass[1];
                out->bad = total->sum.bad;
                total->sum.mass[0] = total->sum.mass[1] = 0.0;
                total->sum.bad = 0;
                total->done = 0u;
            }
        }
        return;
    }
    const size_t pitch2 = static_cast<size_t>(a.v2_chunks) * 32;
    if (tid < SPAN) {
        const int jj = j0 + tid, col = tid < nk ? s_idx[tid] : 0xFFFF;
        if (col != 0xFFFF) {
            const Column at = column_of(a, col);
            if (first) {
                a.indices[static_cast<size_t>(r) * a.kk + jj] = static_cast<uint16_t>(col);
                a.taps[static_cast<size_t>(r) * a.kk_pad + jj] = tap_word(at);
            }
            if (a.wt2) {
                uint8_t rel;
                const int place = slab_place(a, col, jj, &rel);
                s_at2[tid] = static_cast<uint32_t>(place);
                if (first) a.rel2[static_cast<size_t>(r) * pitch2 + place] = rel;
            }
            // select layout: w3[chunk][o][32], a chunk being as many steps (one tap of S source columns, of which KC are kept) as fit,
            // the steps ordered by block of S channels, then tap; swizzled like wx.  The
            // column tables hold, per chunk and tile, the byte offset of each column in its 128-byte row (and its 32-channel block in
            // bit 7 and up), in the order in which a thread reads them: [step][place in a quad][quad].  (A span is whole steps.)
            if (a.w3) {
                // (steps of 32 or 64 columns; four, two or one of them in a chunk as 8, 16 or 24 columns stay; a step's columns begin at its column's)
                const int shift_s = a.sel_s == 64 ? 6 : 5, shift_c = a.sel_kc == 8 ? 2 : a.sel_kc == 16 ? 1 : 0, cb = at.c >> shift_s, cc = at.c - (cb << shift_s);
                const int step = cb * a.kh * a.kw + at.tap, chunk = step >> shift_c, sub = step - (chunk << shift_c), js = ((col - c0) >> shift_s) * a.sel_kc;
                const int place = select_place(s_idx + js, a.sel_kc, tid - js);
                // (a thread's columns of two quads are neighbours)
                s_at3[tid] = static_cast<uint32_t>(chunk * 32 + sub * a.sel_kc + (place >> 3) * 8 + (place & 3) * 2 + (place >> 2 & 1));
                if (first)
                    reinterpret_cast<uint32_t*>(a.sel3)[(static_cast<size_t>(chunk) * a.n_tiles + r) * 32 + sub * a.sel_kc + (place & 3) * (a.sel_kc / 4) + (place >> 2)] =
                        static_cast<uint32_t>((cc & 31) * 4 | (cc >> 5) << 7);
            }
            if (a.ws) s_ats[tid] = static_cast<uint32_t>(at.kh << 5 | at.kw << 2 | at.c);
        }
        if (first && blockIdx.x + 1 == gridDim.x)
            for (int i = a.kk + tid; i < a.kk_pad; i += SPAN) a.taps[static_cast<size_t>(r) * a.kk_pad + i] = NM_TAP_PAD;
    } else if (a.wx) {
        const int at = tid - SPAN, n = threads - SPAN, t = at & (SPAN - 1);
        if (t < cols) {
            const int pos = s_pos[t], from = IMPORT ? pos : t;
            for (int rr = at / SPAN; rr < rows; rr += n / SPAN) *expanded_cell(a, row0 + p0 + rr, c0 + t) = pos >= 0 ? nmk::to_tf32(s_tile[rr][from]) : 0.f;
        }
        // zeros: columns up to the last block's 32nd, rows up to the last 32nd
        const int pad_cols = blockIdx.x + 1 == gridDim.x ? (32 - (a.k & 31)) & 31 : 0;
        for (int i = at; i < rows * pad_cols; i += n) *expanded_cell(a, row0 + p0 + i / pad_cols, a.k + i % pad_cols) = 0.f;
        if (r + 1 == static_cast<int>(gridDim.y) && first)
            for (int i = at; i < (a.wx_rows - a.c_out) * (cols + pad_cols); i += n) *expanded_cell(a, a.c_out + i / (cols + pad_cols), c0 + i % (cols + pad_cols)) = 0.f;
    }
    asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");

    const int col = j < nk ? s_idx[j] : 0xFFFF;
    if (col == 0xFFFF) return;
    const int jj = j0 + j, from = IMPORT ? j : col - c0;
    float* const wt = gather_image(a, row0, tile_rows, jj);
    float* const wt2 = a.wt2 ? a.wt2 + s_at2[j] : nullptr;
    const int k3 = a.w3 ? s_at3[j] & 31 : 0;
    float* const w3 = a.w3 ? a.w3 + static_cast<size_t>(s_at3[j] >> 5) * a.c_out * 32 : nullptr;
    for (int rr = tid >> log_j; rr < rows; rr += threads >> log_j) {
        const int tr = p0 + rr, o = row0 + tr;
        const float v = s_tile[rr][from], t = nmk::to_tf32(v);
        a.values[static_cast<size_t>(o) * a.kk + jj] = v;
        wt[gather_cell(tr, jj)] = t;
        if (wt2) wt2[static_cast<size_t>(o) * pitch2] = t;
        if (w3) w3[static_cast<size_t>(o) * 32 + swizzled(o, k3)] = t;
        if (a.ws) *plane_cell(a, o, static_cast<int>(s_ats[j] >> 5), static_cast<int>(s_ats[j] & 31)) = t;
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

bool compressed_in_one(const nm_weights* h) { return h->m_group <= SPAN; }

// Which layouts this layer's kernels can read, and their dimensions (no device work).
static void plan_layouts(nm_weights* h)
{
    // slab layout: keep-all is the 1:1 pattern; otherwise the chunk is the largest whole number of groups whose kept
    // columns number a multiple of 8 up to 32 and whose source columns number <= 64
    const int n = h->n_keep == h->m_group ? 1 : h->n_keep;
    const int m = h->n_keep == h->m_group ? 1 : h->m_group;
    for (int g = 32 / n; g >= 1; --g)
        if ((g * n) % 8 == 0 && g * m <= 64) {
            h->v2_ok = 1;
            h->v2_g = g; h->v2_kc = g * n; h->v2_s = g * m;
            h->v2_chunks = (h->k + h->v2_s - 1) / h->v2_s;
            break;
        }
    // expanded layout: only shapes the kernels that read it take: output channels in whole float4s (rows are padded
    // with zeros to blocks of 32), and either whole 32-column slabs (expanded-operand kernel) or a short reduction axis
    // (row-run kernel, pointwise layers)
    if (h->c_out % 4 == 0 && (h->c_in % 32 == 0 || h->k <= 512)) h->wx_rows = (h->c_out + 31) / 32 * 32;
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
    const bool planes = h->c_in <= 4 && h->kw <= 8 && h->c_out % 32 == 0 && h->c_out <= 256 &&
                        h->kh * h->c_out * 128 < (1 << 20);
    size_t total = 0;
    auto place = [&total](size_t bytes) {
        const size_t at = total;
        total += (std::max<size_t>(bytes, 16) + 255) / 256 * 256;
        return at;
    };
    const size_t kk1 = static_cast<size_t>(h->kk);
    const size_t pitch2 = static_cast<size_t>(h->v2_chunks) * 32;
    const size_t chunks3 = static_cast<size_t>(h->sel_chunks);
    const size_t at_values = place(h->c_out * kk1 * sizeof(float));
    const size_t at_indices = place(h->n_tiles * kk1 * sizeof(uint16_t));
    const size_t at_taps = place(static_cast<size_t>(h->n_tiles) * h->kk_pad * sizeof(uint32_t));
    // Layouts that every word of is written come before the part of the block that the creating call clears (status, sums and layouts with
    // padding or zeros in the pruned columns).  512 x 3 x 3 x 512 at 2:4 has nothing to clear (with 9 of its 28 MB cleared it took 7 us more).
    const int spc = h->sel_s ? 32 / h->sel_kc : 1;
    const bool full_wx = compressed_in_one(h);
    const bool full_wt = h->kk % NM_KCHUNK == 0;
    const bool full_wt2 = h->v2_kc == 32 && h->k % std::max(h->v2_s, 1) == 0;
    const bool full_w3 = h->sel_s && h->sel_kc * spc == 32 && h->k / h->sel_s % spc == 0;
    size_t sums_end = 0, at_status = 0, at_mass = 0, at_wt = 0, at_wt2 = 0, at_rel2 = 0, at_wx = 0, at_w3 = 0, at_sel3 = 0, at_ws = 0;
    for (const bool full : {true, false}) {
        if (!full) {
            h->zero_from = total;
            at_status = place(4 * sizeof(int));
            at_mass = place(sizeof(Readback));
            sums_end = total;
        }
        if (h->wx_rows && full_wx == full) at_wx = place(static_cast<size_t>((h->k + 31) / 32) * h->wx_rows * 128);
        if (full_wt == full) at_wt = place(static_cast<size_t>(h->c_out) * h->kk_pad * sizeof(float));
        if (full_wt2 == full) {
            if (h->v2_ok) at_wt2 = place(h->c_out * pitch2 * sizeof(float)), at_rel2 = place(h->n_tiles * pitch2);
        }
        if (full_w3 == full) {
            if (h->sel_s) at_w3 = place(chunks3 * h->c_out * 128), at_sel3 = place(chunks3 * h->n_tiles * 128);
        }
    }
    if (planes) at_ws = place(static_cast<size_t>(h->kh) * h->c_out * 128);
    h->block_used = total;
    h->clear_layouts = total > sums_end;
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

static LayoutArgs layout_args(nm_weights* h, const float* src, const uint16_t* idx, bool import)
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
    a.status = h->status;
    a.by_c_in = divisor(h->c_in); a.by_kw = divisor(h->kw); a.by_v2_s = divisor(std::max(h->v2_s, 1));
    return a;
}

nm_status_t build_layouts(nm_weights* h, const float* src, const uint16_t* idx, bool import, cudaStream_t st)
{
    const LayoutArgs a = layout_args(h, src, idx, import);
    if (h->c_out > 65535) return fail(NM_ERR_CUDA, "weight layout kernel: more than 65535 output channels");   // bounds grid.y
    const dim3 grid((h->kk_pad + 127) / 128, h->n_tiles * ((h->tile_t + ROWS - 1) / ROWS));
    k_build_layouts<<<grid, 128, 0, st>>>(a);
    count_launch(1);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? NM_OK : fail(NM_ERR_CUDA, "weight layout kernel: %s", cudaGetErrorString(e));
}

nm_status_t compress_in_one(nm_weights* h, const float* src, const uint16_t* idx, cudaStream_t st, double* mass2, int* bad)
{
    if (h->c_out > 65535) return fail(NM_ERR_CUDA, "weight layout kernel: more than 65535 output channels");   // bounds grid.y
    Readback* slot = take_slot();
    // without a slot the sums lie in the handle, and are cleared and copied
    if (h->clear_layouts || !slot) {
        const nm_status_t s = clear_handle_memory(h, st);
        if (s != NM_OK) {
            if (slot) give_slot(slot);
            return s;
        }
    }
    const LayoutArgs a = layout_args(h, src, idx, idx != nullptr);
    const int span = SPAN / h->m_group * h->m_group, rows = std::min(h->tile_t, h->c_out);
    int log_j = 0;
    while ((1 << log_j) < span / h->m_group * h->n_keep) ++log_j;
    const dim3 grid((h->k + span - 1) / span, h->n_tiles, (rows + PART - 1) / PART);
    const unsigned threads = (rows > 16 ? 512u : 256u) + 32u;
    const int number = slot ? static_cast<int>(slot - g_slots) : -1;
    if (idx) k_compress<true><<<grid, threads, 0, st>>>(a, span, log_j, reinterpret_cast<Readback*>(h->mass), number, slot);
    else k_compress<false><<<grid, threads, 0, st>>>(a, span, log_j, reinterpret_cast<Readback*>(h->mass), number, slot);
    count_launch(1);
    cudaError_t e = cudaGetLastError();
    if (!slot && e == cudaSuccess) return finish_handle(h, st, mass2, bad);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    const Readback got = slot ? *slot : Readback{};
    if (slot) give_slot(slot);
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "building the weight handle: %s", cudaGetErrorString(e));
    if (mass2) { mass2[0] = got.mass[0]; mass2[1] = got.mass[1]; }
    if (bad) *bad = got.bad;
    return NM_OK;
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
