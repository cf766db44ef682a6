// Column-wise N:M pruning at tile level (Sec. 3.1) on the device, and construction of the
// kernel-side copies of the compressed form (Sec. 2.1; inputs W and Idx of Algorithm 1).
//
// The selection:
//   score    s[k]    = sum over the tile's rows of |w[o][k]|, fp64, ascending row order (bit-reproducible); a sum that
//            is NaN (a NaN weight) counts as +infinity, so that the order below is total
//   select   kept iff fewer than N columns of k's group beat it, where column i beats column k when s[i] > s[k], or
//            s[i] == s[k] and i < k (lower column wins ties)
//   place    position of a kept column = N * group + number of kept columns before it in its group
// It is the closed form of "pick the largest N times": both orderings are the sort by (score
// descending, column ascending), so the result is unique.  Where a group fits a block (M <= 128) one kernel of nm_layout.cu selects and
// writes values and kernel layouts.  Wider groups (the adaptive form, M up to K) take the steps as the kernels below with the scores in
// scratch memory; nm_layout.cu then writes the rest.
#include <algorithm>

#include "nm_internal.h"
#include "nm_ptx.cuh"

namespace {

__global__ void k_score(const float* __restrict__ w, int c_out, int k, int tile_t, double* __restrict__ score)
{
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (col >= k) return;
    const int row0 = r * tile_t;
    const int row1 = min(row0 + tile_t, c_out);
    double s = 0.0;
    for (int o = row0; o < row1; ++o) s += fabs(static_cast<double>(w[static_cast<size_t>(o) * k + col]));
    // NaN compares false with everything: such a column would neither beat nor be beaten, and its
    // group would keep more than N columns.  It ranks as +infinity instead (ties by column).
    score[static_cast<size_t>(r) * k + col] = (s == s) ? s : static_cast<double>(INFINITY);
}

__global__ void k_select(const double* __restrict__ score, int k, int n_keep, int m_group,
                         uint8_t* __restrict__ keep)
{
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (col >= k) return;
    const double* s = score + static_cast<size_t>(r) * k;
    const int g0 = (col / m_group) * m_group;
    const int g1 = min(g0 + m_group, k);
    const double mine = s[col];
    int beaten_by = 0;
    for (int i = g0; i < g1; ++i) {
        const double si = s[i];
        beaten_by += (si > mine) || (si == mine && i < col);
    }
    keep[static_cast<size_t>(r) * k + col] = beaten_by < n_keep ? 1 : 0;
}

// L1 mass of all columns and of the retained ones: mass[0] += score, mass[1] += score * keep.
__global__ void k_mass(const double* __restrict__ score, const uint8_t* __restrict__ keep, size_t cells,
                       double* __restrict__ mass)
{
    double all = 0.0, kept = 0.0;
    for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < cells;
         i += static_cast<size_t>(gridDim.x) * blockDim.x) {
        const double s = score[i];
        all += s;
        if (keep[i]) kept += s;
    }
    for (int d = 16; d > 0; d >>= 1) {
        all += __shfl_down_sync(0xFFFFFFFFu, all, d);
        kept += __shfl_down_sync(0xFFFFFFFFu, kept, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(mass + 0, all);
        atomicAdd(mass + 1, kept);
    }
}

__global__ void k_compact(const uint8_t* __restrict__ keep, int k, int kk, int n_keep, int m_group,
                          uint16_t* __restrict__ indices)
{
    const int col = blockIdx.x * blockDim.x + threadIdx.x;
    const int r = blockIdx.y;
    if (col >= k) return;
    const uint8_t* kp = keep + static_cast<size_t>(r) * k;
    if (!kp[col]) return;
    const int g = col / m_group;
    int pos = g * n_keep;  // every earlier group is a full one and kept exactly n_keep
    for (int i = g * m_group; i < col; ++i) pos += kp[i];
    // a group never holds more than N kept columns (the order of the scores is total); the bound
    // makes sure that no input whatsoever can place a column outside its group's slots
    if (pos >= min(kk, (g + 1) * n_keep)) return;
    indices[static_cast<size_t>(r) * kk + pos] = static_cast<uint16_t>(col);
}

// Groups wider than a block of k_compress.
nm_status_t prune_wide(const float* w_dense, nm_weights* h, cudaStream_t st, double* mass)
{
    using namespace nmhost;
    nm_status_t st_out = clear_handle_memory(h, st);
    if (st_out != NM_OK) return st_out;
    size_t scratch_bytes = 0;
    const size_t cells = static_cast<size_t>(h->n_tiles) * h->k;
    uint8_t* scratch = static_cast<uint8_t*>(device_block_alloc(cells * 9, h->device, &scratch_bytes));
    if (!scratch) return fail(NM_ERR_ALLOC, "nm_prune: cannot allocate %zu bytes of scratch", cells * 9);
    double* score = reinterpret_cast<double*>(scratch);
    uint8_t* keep = scratch + cells * sizeof(double);
    const dim3 blk(128), grid((h->k + 127) / 128, h->n_tiles);
    k_score<<<grid, blk, 0, st>>>(w_dense, h->c_out, h->k, h->tile_t, score);
    k_select<<<grid, blk, 0, st>>>(score, h->k, h->n_keep, h->m_group, keep);
    k_compact<<<grid, blk, 0, st>>>(keep, h->k, h->kk, h->n_keep, h->m_group, h->indices);
    k_mass<<<static_cast<unsigned>(std::min<size_t>((cells + 255) / 256, 1024)), 256, 0, st>>>(score, keep, cells, h->mass);
    count_launch(4);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) st_out = fail(NM_ERR_CUDA, "pruning kernels: %s", cudaGetErrorString(e));
    if (st_out == NM_OK) st_out = build_layouts(h, w_dense, h->indices, false, st);
    if (st_out == NM_OK) st_out = finish_handle(h, st, mass, nullptr);
    device_block_free(scratch, scratch_bytes, h->device, st_out == NM_OK);
    return st_out;
}

}  // namespace

namespace nmhost {

nm_status_t prune_on_device(const float* w_dense, nm_weights* h, cudaStream_t st)
{
    double mass[2] = {0.0, 0.0};
    // (either way the one synchronisation: the handle is complete when the call returns, whatever stream uses it next)
    nm_status_t st_out = compressed_in_one(h) ? compress_in_one(h, w_dense, nullptr, st, mass, nullptr) : prune_wide(w_dense, h, st, mass);
    if (st_out == NM_OK) {
        h->l1_total = mass[0];
        h->l1_kept = mass[1];
    }
    return st_out;
}

nm_status_t build_from_compressed(const float* values, const uint16_t* indices, nm_weights* h, cudaStream_t st)
{
    int bad = 0;
    nm_status_t s = compressed_in_one(h) ? NM_OK : clear_handle_memory(h, st);
    if (s == NM_OK && !kernel_may_touch(values, indices, h->device)) {
        // through the handle's own arrays, which the layout kernel then reads and writes back unchanged
        cudaError_t e = cudaMemcpyAsync(h->values, values, static_cast<size_t>(h->c_out) * h->kk * sizeof(float), cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(h->indices, indices, static_cast<size_t>(h->n_tiles) * h->kk * sizeof(uint16_t), cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return fail(NM_ERR_CUDA, "nm_weights_import: %s", cudaGetErrorString(e));
        values = h->values;
        indices = h->indices;
    }
    if (s == NM_OK && compressed_in_one(h)) {
        s = compress_in_one(h, values, indices, st, nullptr, &bad);
    } else {
        if (s == NM_OK) s = build_layouts(h, values, indices, true, st);
        if (s == NM_OK) s = finish_handle(h, st, nullptr, &bad);
    }
    if (s == NM_OK && bad)
        s = fail(NM_ERR_INVALID_ARG, "nm_weights_import: an index row is not strictly ascending below K, or does not hold N columns per group of M");
    return s;
}

}  // namespace nmhost
