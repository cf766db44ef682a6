// Variant 1: direct-gather sparse implicit GEMM (any shape).
//
// A CTA owns 128 output pixels and one pruning tile.  For every chunk of 32 retained columns eight warps gather the
// activations
//     a[p][j] = x[n][oh*s - pad + kh_j*dil][ow*s - pad + kw_j*dil][c_j]      (zero outside the image)
// straight from NHWC global memory (lane = retained column j, so a warp reads one pixel's retained channels:
// neighbouring addresses), round them to TF32 and store them in the 128-byte-swizzled K-major layout tcgen05 reads.  One
// thread fetches the weight chunk (stored as the shared-memory image) with a bulk copy, one issues four 128 x N x 8 TF32
// MMAs per chunk.  This is Algorithm 1 with the vector register replaced by a 128-pixel operand tile and the T
// accumulators by T TMEM columns; the gather is the fused im2col + packing of Sec. 3.2 without its buffer.
//
// It takes every shape the TMA-fed kernels do not (channel counts that are no multiple of 32, small or odd tile widths,
// small inputs), so it has to be good at all of them.  What bounds it is the gather's instruction stream: a chunk
// costs a CTA 0.70 us alone on its SM and 0.95 us beside a second one, where issue slots are 60 % busy; more operand slots (4
// for 2), more gathering warps (16 for 8) and several tiles per CTA (which share the chunk's lines in L1) changed
// neither figure.  Two chunks are kept in flight in registers, the operand slots decouple the gathering warps from
// the MMAs, and where there are far fewer pixel blocks and tiles than SMs the chunks are split over the CTAs of a thread-block
// cluster (partial sums move as bulk copies between their shared memories and are added in the order of the ranges).
// Before the pipelining and the split, and now: 3978 pixels, 242 chunks, one tile 295 -> 37 us; 6930 pixels, 54 chunks, 8 tiles of
// 64 152 -> 68 us.
//
//   warps 0-7  gather, then epilogue: TMEM -> staging in shared memory -> bias, shortcut, ReLU, coalesced NHWC stores
//   warp 8     MMA issuer, tensor memory      warp 9  weight producer
#include <algorithm>

#include "nm_internal.h"
#include "nm_ptx.cuh"

namespace {

using namespace nmk;

constexpr int BM = 128;                       // output pixels per CTA = MMA M
constexpr int A_BYTES = BM * NM_KCHUNK * 4;
constexpr int THREADS = 320;
constexpr int GATHER = 256;                   // threads of the gathering warps
constexpr int RPW = 16;                       // pixel rows per gathering warp
constexpr int NA = 2;                         // operand slots
constexpr int TAPS_AHEAD = 4;
constexpr int NW_MAX = 8;                     // weight slots
constexpr int PASS = 64;                      // output channels staged at a time

struct GatherCfg {
    int n;            // MMA width = accumulator columns
    int cs;           // CTAs per cluster = ranges of the chunks
    int chunks;
    int w_stages, w_bytes;
    int rps;          // pixel rows a CTA of the cluster finishes
    int tmem_cols;
};

__device__ __forceinline__ bool aborted(volatile int* flag) { return *flag != 0; }

// *p where `on` is non-zero, else 0; a predicated load (written as a conditional it becomes a branch per pixel row).
__device__ __forceinline__ float load_if(const float* p, uint32_t on)
{
    float v;
    asm volatile(
        "{\n\t"
        ".reg .pred q;\n\t"
        "setp.ne.u32 q, %2, 0;\n\t"
        "mov.f32 %0, 0f00000000;\n\t"
        "@q ld.global.nc.f32 %0, [%1];\n\t"
        "}\n"
        : "=f"(v)
        : "l"(p), "r"(on));
    return v;
}
__device__ __forceinline__ int pitch_of(int cols)
{
    // floats per staged row: whole 16-byte pieces, an odd number of them (rows of a quarter warp then start in different banks)
    const int c4 = (cols + 3) / 4;
    return (c4 | 1) * 4;
}

// WIDE: kernels of more than 64 taps, or pixel blocks whose input spans 4 GB or more: bounds by comparison and 64-bit
// addresses instead of a tap mask per pixel and 32-bit offsets.
template <bool WIDE>
__global__ void __launch_bounds__(THREADS, 2) k_conv_gather(const ConvParams p, const GatherCfg cfg)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_full[NA], s_free[NA], s_wfull[NW_MAX], s_wfree[NW_MAX], s_acc, s_part;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    // per pixel: WIDE image, first input row, first input column; else byte offset, tap mask
    __shared__ __align__(16) uint32_t s_off[BM], s_mask[WIDE ? 1 : 2][BM + 4];   // (+ 4: the two words of a row in different banks)
    __shared__ int s_col[BM];

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t w_ring = ring + NA * A_BYTES;
    const uint32_t part = w_ring + cfg.w_stages * cfg.w_bytes;
    volatile int* abort_flag = &s_abort;

    // ---- this CTA's pixels, tiles and chunks ------------------------------------------------------
    const uint32_t item = blockIdx.x / static_cast<uint32_t>(cfg.cs);
    const uint32_t block = item / static_cast<uint32_t>(p.n_tiles);
    const int tile = static_cast<int>(item - block * static_cast<uint32_t>(p.n_tiles));
    const long long pix0 = static_cast<long long>(block) * BM;
    const int count = p.pixels - pix0 < BM ? static_cast<int>(p.pixels - pix0) : BM;
    const int c_begin = static_cast<int>(rank) * cfg.chunks / cfg.cs, c_end = (static_cast<int>(rank) + 1) * cfg.chunks / cfg.cs;
    const int my_chunks = c_end - c_begin;
    const int hw = p.ho * p.wo;
    const int n_first = static_cast<int>(pix0 / hw);
    const int row0 = static_cast<int>(rank) * cfg.rps;   // first pixel row this CTA finishes
    const int my_rows = max(0, min(cfg.rps, count - row0));

    // ---- set-up --------------------------------------------------------------------------------
    if (warp == 8) tmem_alloc(smem_u32(&s_tmem), cfg.tmem_cols);
    if (tid == 0) {
        for (int i = 0; i < NA; ++i) {
            mbar_init(smem_u32(&s_full[i]), GATHER / 32);   // the gathering warps
            mbar_init(smem_u32(&s_free[i]), 1);
        }
        for (int i = 0; i < NW_MAX; ++i) {
            mbar_init(smem_u32(&s_wfull[i]), 1);
            mbar_init(smem_u32(&s_wfree[i]), 1);
        }
        mbar_init(smem_u32(&s_acc), 1);
        mbar_init(smem_u32(&s_part), 1);
        mbar_fence_init();
        s_abort = 0;
    }
    if (tid < BM) {
        uint32_t off = WIDE ? 0xFFFFFFFFu : 0u;
        unsigned long long mask = 0;
        int col = 0;
        if (tid < count) {
            const int rem0 = static_cast<int>(pix0 - static_cast<long long>(n_first) * hw) + tid;
            const int dn = rem0 / hw, rem = rem0 - dn * hw;
            const int oh = rem / p.wo, ow = rem - oh * p.wo;
            const int ih0 = oh * p.stride_h - p.pad_h, iw0 = ow * p.stride_w - p.pad_w;
            if (WIDE) {
                off = static_cast<uint32_t>(n_first + dn);
                mask = static_cast<uint32_t>(ih0);
                col = iw0;
            } else {
                unsigned long long cols = 0;
                for (int j = 0; j < p.kw; ++j) cols |= (static_cast<unsigned>(iw0 + j * p.dil_w) < static_cast<unsigned>(p.w) ? 1ull : 0ull) << j;
                for (int i = 0; i < p.kh; ++i)
                    if (static_cast<unsigned>(ih0 + i * p.dil_h) < static_cast<unsigned>(p.h)) mask |= cols << (i * p.kw);
                // taps outside the image are never read: the offset may wrap as long as offset + tap does not
                off = (static_cast<uint32_t>(dn * p.h + ih0) * static_cast<uint32_t>(p.w) + static_cast<uint32_t>(iw0)) *
                                     static_cast<uint32_t>(p.c_in) * 4u;
            }
        }
        s_off[tid] = off;
        s_mask[0][tid] = static_cast<uint32_t>(mask);
        if (!WIDE) s_mask[1][tid] = static_cast<uint32_t>(mask >> 32);
        s_col[tid] = col;
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const int nch = min(p.tile_t, p.c_out - tile * p.tile_t);   // channels this CTA computes
    const int passes = (nch + PASS - 1) / PASS;
    auto pass_cols = [&](int i) { return min(PASS, nch - i * PASS); };
    // Partial sums of this CTA's rows in pass i, from every CTA of the cluster.  A CTA without rows neither expects nor waits: an
    // expectation of nothing would complete its phase at once, and the next pass's the one after it, past a warp of this
    // CTA that has yet to look at the first (a wait by parity would then never end).
    auto expect_part = [&](int i) {
        if (my_rows == 0) return;
        mbar_arrive_expect_tx(smem_u32(&s_part), static_cast<uint32_t>(my_rows * pitch_of(pass_cols(i)) * 4 * cfg.cs));
    };
    if (cfg.cs > 1) {
        // the barrier knows what to expect, and every CTA of the cluster has started, before any of them sends (waited for below)
        if (tid == 0) expect_part(0);
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    pdl_launch_dependents();

    if (warp < 8) {
        // =========================== gather ===========================
        const int base_row = warp * RPW;
        const uint4* offs = reinterpret_cast<const uint4*>(s_off + base_row);    // four rows per load, the same for all lanes
        uint32_t all[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};   // taps inside the image for every row of this warp
        if (!WIDE)
            for (int i = 0; i < RPW; ++i) {
                all[0] &= s_mask[0][base_row + i];
                all[1] &= s_mask[1][base_row + i];
            }
        const char* xb = reinterpret_cast<const char*>(p.x) + (WIDE ? 0 : static_cast<size_t>(n_first) * p.h * p.w * p.c_in * 4);
        auto at = [xb](uint32_t bytes) { return reinterpret_cast<const float*>(xb + bytes); };
        auto on = [&](uint32_t bytes, uint32_t tap_inside) {   // self-checking build: the load lies in the input
            if (NM_SELF_CHECKING && tap_inside != 0u &&
                !NM_ALLOWED(nm_bytes_in_span(bytes, 4, 0, static_cast<uint64_t>(p.batch - n_first) * p.h * p.w * p.c_in * 4), p.status, 103, bytes))
                return 0u;
            return tap_inside;
        };
        const uint32_t* taps = p.taps + static_cast<size_t>(tile) * p.kk_pad + lane;
        // taps of the next chunks to be read: a chunk takes less time than its tap needs to arrive
        int fc = c_begin;
        auto fetch = [&]() {
            const uint32_t t = fc < c_end ? __ldg(taps + fc * NM_KCHUNK) : NM_TAP_PAD;
            ++fc;
            return t;
        };
        uint32_t queue[TAPS_AHEAD];
#pragma unroll
        for (int i = 0; i < TAPS_AHEAD; ++i) queue[i] = fetch();
        auto read = [&](float (&v)[RPW]) {
            const uint32_t tap = queue[0];
#pragma unroll
            for (int i = 0; i + 1 < TAPS_AHEAD; ++i) queue[i] = queue[i + 1];
            queue[TAPS_AHEAD - 1] = fetch();
            bool ok = tap != NM_TAP_PAD;
            if (NM_SELF_CHECKING) ok = ok && NM_ALLOWED(nm_tap_in_layer(tap, p.kh, p.kw, p.c_in), p.status, 101, tap);
            const int ki = static_cast<int>(tap >> 24), kj = static_cast<int>((tap >> 16) & 0xFFu), c = static_cast<int>(tap & 0xFFFFu);
            if (WIDE) {
                const int dh = ki * p.dil_h, dw = kj * p.dil_w;
#pragma unroll
                for (int i = 0; i < RPW; ++i) {
                    const int n = static_cast<int>(s_off[base_row + i]);
                    const int ih = static_cast<int>(s_mask[0][base_row + i]) + dh, iw = s_col[base_row + i] + dw;
                    const bool in = ok && n >= 0 && NM_ALLOWED(n < p.batch, p.status, 102, n) && static_cast<unsigned>(ih) < static_cast<unsigned>(p.h) && static_cast<unsigned>(iw) < static_cast<unsigned>(p.w);
                    v[i] = load_if(p.x + ((static_cast<size_t>(n) * p.h + ih) * p.w + iw) * p.c_in + c, in ? 1u : 0u);
                }
            } else {
                const uint32_t delta = (static_cast<uint32_t>(ki * p.dil_h * p.w + kj * p.dil_w) * static_cast<uint32_t>(p.c_in) + static_cast<uint32_t>(c)) * 4u;
                const int tap_no = ki * p.kw + kj, word = tap_no >> 5;
                const uint32_t bit = ok ? 1u << (tap_no & 31) : 0u;
                const uint4* masks = reinterpret_cast<const uint4*>(s_mask[0] + (ok ? word : 0) * (BM + 4) + base_row);
                if (!NM_SELF_CHECKING && __all_sync(0xFFFFFFFFu, ((word ? all[1] : all[0]) & bit) != 0u)) {   // inside the image for all rows and columns of this warp
#pragma unroll
                    for (int i = 0; i < RPW; i += 4) {
                        const uint4 o = offs[i / 4];
                        v[i] = __ldg(at(o.x + delta)); v[i + 1] = __ldg(at(o.y + delta)); v[i + 2] = __ldg(at(o.z + delta)); v[i + 3] = __ldg(at(o.w + delta));
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < RPW; i += 4) {
                        const uint4 o = offs[i / 4], m = masks[i / 4];
                        v[i] = load_if(at(o.x + delta), on(o.x + delta, m.x & bit));
                        v[i + 1] = load_if(at(o.y + delta), on(o.y + delta, m.y & bit));
                        v[i + 2] = load_if(at(o.z + delta), on(o.z + delta, m.z & bit));
                        v[i + 3] = load_if(at(o.w + delta), on(o.w + delta, m.w & bit));
                    }
                }
            }
        };
        RingPos rp;
        auto store = [&](const float (&v)[RPW]) {
            const bool ready = !rp.wrapped || mbar_wait_lone(smem_u32(&s_free[rp.s]), rp.parity ^ 1u);
            if (!__all_sync(0xFFFFFFFFu, ready)) { *abort_flag = 2; return false; }
            const uint32_t dst = ring + rp.s * A_BYTES + base_row * 128 + lane * 4;   // 16-byte pieces XOR-ed with the row: bits 4-6
#pragma unroll
            for (int i = 0; i < RPW; ++i)
                asm volatile("st.shared.f32 [%0], %1;" ::"r"((dst ^ ((i & 7) << 4)) + i * 128), "f"(to_tf32(v[i])) : "memory");
            fence_proxy_async();
            __syncwarp();
            if (elect_one()) mbar_arrive(smem_u32(&s_full[rp.s]));
            rp.advance(NA);
            return true;
        };
        pdl_wait();
        float va[RPW], vb[RPW];
        if (my_chunks > 0) read(va);
        if (my_chunks > 1) read(vb);
        for (int u = 0; u < my_chunks; u += 2) {
            if (aborted(abort_flag) || !store(va)) break;
            if (u + 2 < my_chunks) read(va);
            if (u + 1 >= my_chunks || !store(vb)) break;
            if (u + 3 < my_chunks) read(vb);
        }
        __syncwarp();
    } else if (warp == 8) {
        // =========================== MMA issuer ===========================
        if (elect_one()) {
            const uint32_t idesc = umma_idesc_tf32(BM, cfg.n);
            RingPos rp, rw;
            for (int c = c_begin; c < c_end; ++c) {
                if (!mbar_wait_lone(smem_u32(&s_wfull[rw.s]), rw.parity) || !mbar_wait_lone(smem_u32(&s_full[rp.s]), rp.parity)) {
                    *abort_flag = 3;
                    break;
                }
                tc_fence_after();
                const int steps = min(NM_KCHUNK, p.kk - c * NM_KCHUNK) + 7 >> 3;   // K-steps of eight columns that hold any
                const uint64_t adesc = umma_desc_k_sw128(ring + rp.s * A_BYTES, 1024);
                const uint64_t bdesc = umma_desc_k_sw128(w_ring + rw.s * cfg.w_bytes, 1024);
#pragma unroll
                for (int kq = 0; kq < 4; ++kq)
                    if (kq < steps) umma_tf32_ss(tmem, adesc + 2 * kq, bdesc + 2 * kq, idesc, (c > c_begin || kq > 0) ? 1u : 0u);
                umma_commit(smem_u32(&s_free[rp.s]));
                umma_commit(smem_u32(&s_wfree[rw.s]));
                rp.advance(NA);
                rw.advance(cfg.w_stages);
            }
            umma_commit(smem_u32(&s_acc));
        }
        __syncwarp();
    } else {
        // =========================== weight producer ===========================
        // The weights are no earlier kernel's output (a handle is complete when the call that built it returns): no pdl_wait.
        if (elect_one()) {
            // the tile's own rows; what the MMA reads behind them ends in accumulator columns nobody reads
            const uint32_t bytes = static_cast<uint32_t>(nch) * 128u;
            const float* src = p.wt + static_cast<size_t>(tile) * p.tile_t * p.kk_pad;
            RingPos rp;
            int issued = 0;
            for (int c = c_begin; c < c_end; ++c, ++issued) {
                if (rp.wrapped && !mbar_wait_lone(smem_u32(&s_wfree[rp.s]), rp.parity ^ 1u)) { *abort_flag = 4; break; }
                const uint32_t bar = smem_u32(&s_wfull[rp.s]);
                mbar_arrive_expect_tx(bar, bytes);
                bulk_load_1d(w_ring + rp.s * cfg.w_bytes, src + static_cast<size_t>(c) * nch * NM_KCHUNK, bytes, bar);
                rp.advance(cfg.w_stages);
            }
            if (aborted(abort_flag))   // loads already issued still target this CTA's shared memory: let them land (bounded)
                for (int back = 0; back < cfg.w_stages && back < issued; ++back) {
                    if (rp.s == 0) { rp.s = cfg.w_stages; rp.parity ^= 1u; }
                    --rp.s;
                    (void)mbar_wait_polls(smem_u32(&s_wfull[rp.s]), rp.parity, 1u << 16);
                }
        }
        __syncwarp();
    }

    // ---- epilogue ----------------------------------------------------------------------------------
    if (cfg.cs > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every CTA of the cluster is running
    if (warp < 8) {
        const bool ok = aborted(abort_flag) || mbar_wait(smem_u32(&s_acc), 0);
        if (!__all_sync(0xFFFFFFFFu, ok)) *abort_flag = 5;
        tc_fence_after();
    }
    const int q = warp & 3, half = warp >> 2;
    const int row = q * 32 + lane;
    for (int i = 0; i < passes; ++i) {
        const int cols = pass_cols(i);
        const int pitch = pitch_of(cols);
        if (warp < 8) {
            // accumulators -> staging [row][channel of the pass] over the ring, which is idle now; sixteen columns at a time
            for (int jb = half * 16; jb < cols; jb += 32) {
                uint32_t v[16];
                tmem_ld16(tmem + (static_cast<uint32_t>(q * 32) << 16) + i * PASS + jb, v);
                tmem_ld_wait();
                const uint32_t dst = ring + (row * pitch + jb) * 4;   // (a pitch is whole 16-byte pieces)
#pragma unroll
                for (int e = 0; e < 16; e += 4)
                    if (jb + e < cols)
                        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + e * 4), "r"(v[e]), "r"(v[e + 1]), "r"(v[e + 2]),
                                     "r"(v[e + 3])
                                     : "memory");
            }
            tc_fence_before();
            if (cfg.cs > 1) fence_proxy_async();
            asm volatile("bar.sync 1, %0;" ::"n"(GATHER) : "memory");
            if (cfg.cs > 1) {
                // a run of rows to every CTA of the cluster
                if (warp < cfg.cs) {
                    const int rows = min(cfg.rps, count - warp * cfg.rps);
                    if (rows > 0 && elect_one())
                        bulk_copy_cluster(mapa_shared(part + rank * cfg.rps * pitch * 4, static_cast<uint32_t>(warp)), ring + warp * cfg.rps * pitch * 4,
                                          static_cast<uint32_t>(rows * pitch * 4), mapa_shared(smem_u32(&s_part), static_cast<uint32_t>(warp)));
                }
                // a multiple of the other waits' limit: a CTA that gave up on one of those has sent by then
                const uint32_t bar = smem_u32(&s_part), par = static_cast<uint32_t>(i & 1);
                const bool landed = my_rows == 0 || mbar_wait_cluster(bar, par) || mbar_wait_cluster(bar, par) || mbar_wait_cluster(bar, par);
                if (!__all_sync(0xFFFFFFFFu, landed)) *abort_flag = 6;
            }
            if (!aborted(abort_flag)) {
                const uint32_t src = cfg.cs > 1 ? part : ring;
                const uint32_t src_step = static_cast<uint32_t>(cfg.rps * pitch * 4);
                const int o0 = tile * p.tile_t + i * PASS;
                const long long pix = pix0 + row0;
                if (((p.c_out | o0 | cols) & 3) == 0) {
                    const int c4 = cols >> 2;
                    for (int f = tid; f < my_rows * c4; f += GATHER) {
                        const int r = f / c4, c = f - r * c4;
                        const size_t at = static_cast<size_t>(pix + r) * p.c_out + o0 + c * 4;
                        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int k = 0; k < cfg.cs; ++k) {
                            float4 a;
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w)
                                         : "r"(src + k * src_step + (r * pitch + c * 4) * 4) : "memory");
                            nm_add4(s, a);
                        }
                        if (p.bias) nm_add4(s, __ldg(reinterpret_cast<const float4*>(p.bias + o0) + c));
                        if (p.residual) nm_add4(s, __ldg(reinterpret_cast<const float4*>(p.residual + at)));
                        if (p.relu) { s.x = fmaxf(s.x, 0.f); s.y = fmaxf(s.y, 0.f); s.z = fmaxf(s.z, 0.f); s.w = fmaxf(s.w, 0.f); }
                        *reinterpret_cast<float4*>(p.y + at) = s;
                    }
                } else {
                    for (int f = tid; f < my_rows * cols; f += GATHER) {
                        const int r = f / cols, c = f - r * cols;
                        const size_t at = static_cast<size_t>(pix + r) * p.c_out + o0 + c;
                        float s = 0.f;
                        for (int k = 0; k < cfg.cs; ++k) {
                            float a;
                            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(a) : "r"(src + k * src_step + (r * pitch + c) * 4) : "memory");
                            s += a;
                        }
                        if (p.bias) s += __ldg(p.bias + o0 + c);
                        if (p.residual) s += __ldg(p.residual + at);
                        p.y[at] = p.relu ? fmaxf(s, 0.f) : s;
                    }
                }
            }
        }
        if (cfg.cs > 1) {
            // nobody sends the next pass's sums (or leaves, its copies unread) before every CTA has used this one's
            if (tid == 0 && i + 1 < passes) expect_part(i + 1);
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        } else if (warp < 8 && i + 1 < passes) {
            asm volatile("bar.sync 1, %0;" ::"n"(GATHER) : "memory");   // the staging rows are free again
        }
    }

    // ---- teardown ------------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort != 0) {
        atomicExch(p.status + 0, static_cast<int>(NM_ERR_TIMEOUT));
        atomicExch(p.status + 1, s_abort);
        atomicExch(p.status + 2, static_cast<int>(blockIdx.x));
    }
    if (warp == 8) tmem_dealloc(tmem, cfg.tmem_cols);
}

}  // namespace

namespace nmhost {

// Ranges of the chunks (CTAs of a cluster) for a launch of `items` (pixel block, tile) pairs.
static int ranges_of(long long items, int chunks)
{
    // By an estimate of the time from the costs above: a chunk takes a CTA 0.95 us, 0.70 us where it has its
    // SM to itself; a wave has about 3 us of its own and 4 more with the exchange (clusters do not fit on every last SM).
    // Measured, us: 7 blocks x 5 tiles, 95 chunks, one range 69, two 42, four 28, eight (a second wave) 49; 55 blocks x 8 tiles, 54 chunks,
    // one range 68, two 83; 15 blocks x 8 tiles, 5 chunks, one range 14, two 16.
    const long long sms = sm_count();
    double best = 1e30;
    int ranges = 1;
    for (int cs = 1; cs <= 8 && (cs == 1 || chunks >= 2 * cs); cs *= 2) {
        const long long ctas = items * cs, slots = 2 * sms - (cs > 1 ? 32 : 0);
        const long long full = ctas / slots, rest = ctas - full * slots;
        const int range = (chunks + cs - 1) / cs;
        const double wave = cs > 1 ? 7.0 : 3.0;
        const double t = full * (range * 0.95 + wave) + (rest == 0 ? 0.0 : range * (rest <= sms ? 0.70 : 0.95) + wave);
        if (t < best * 0.95) { best = t; ranges = cs; }
    }
    return ranges;
}

// The time over all sizes, fitted to 900 layers that the stream kernel takes as well (c_in 32-512, c_out 16-1024, 1x1 to 5x5, T 16-128; 12 % rms).  A row
// of a chunk reads as many sectors more as there are source columns to a kept one.
double gather_estimate_us(const ConvParams& p)
{
    const int chunks = p.kk_pad / NM_KCHUNK;
    const long long items = (p.pixels + BM - 1) / BM * p.n_tiles, sms = sm_count();
    const int cs = ranges_of(items, chunks);
    const long long ctas = items * cs, slots = 2 * sms - (cs > 1 ? 32 : 0), full = ctas / slots, rest = ctas - full * slots;
    const double range = (chunks + cs - 1) / cs, spread = static_cast<double>(p.m_group) / p.n_keep, width = p.tile_t / 32.0;
    const double wave = (cs > 1 ? 4.8 : 2.6) + 1.0 * width;
    const double beside = range * (0.675 + 0.08 * spread + 0.084 * width) + wave, alone = range * (0.475 + 0.023 * spread + 0.072 * width) + wave;
    return full * beside + (rest == 0 ? 0.0 : rest <= sms ? alone : beside);
}

double gather_time_us(const ConvParams& p)
{
    const double chunks = p.kk_pad / NM_KCHUNK, channels = std::min(p.tile_t, p.c_out);
    return cta_rounds((p.pixels + BM - 1) / BM * p.n_tiles, nmhost::sm_count()) * (3.0 + 0.80 * chunks + 0.040 * channels) + 0.7 + 0.19 * chunks;
}

nm_status_t launch_conv_gather(const ConvParams& p, cudaStream_t st)
{
    GatherCfg cfg = {};
    cfg.n = gather_width(p.tile_t, p.c_out);
    if (cfg.n > 256) return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: tile_t %d exceeds 256", p.tile_t);
    cfg.chunks = p.kk_pad / NM_KCHUNK;
    const long long blocks = (p.pixels + BM - 1) / BM;
    cfg.cs = ranges_of(blocks * p.n_tiles, cfg.chunks);
    cfg.rps = BM / cfg.cs;
    cfg.tmem_cols = 32;
    while (cfg.tmem_cols < cfg.n) cfg.tmem_cols <<= 1;
    const long long grid = blocks * p.n_tiles * cfg.cs;
    if (grid > 0x7FFFFFFFll) return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: too many output pixels");
    cfg.w_bytes = cfg.n * 128;   // a multiple of 2 KB
    // A weight chunk takes about 1 us to arrive from L2, more than a chunk's time: its ring is deeper than the operands'.
    // The staging of a pass (128 rows of at most PASS + 4 floats) lies over the rings, with a cluster the received sums take
    // as much again.
    const int stage_out = BM * (PASS + 4) * 4;
    cfg.w_stages = cfg.n <= 32 ? 6 : cfg.n <= 64 ? 4 : cfg.n <= 128 && cfg.cs == 1 ? 3 : 2;
    size_t smem = 1024 + static_cast<size_t>(NA) * A_BYTES + static_cast<size_t>(cfg.w_stages) * cfg.w_bytes + (cfg.cs > 1 ? stage_out : 0);
    // No more CTAs on an SM than its tensor memory holds; a cluster's CTAs, which wait for one another, take at least their
    // columns' share of the shared memory (see NM_EXCLUSIVE_SMEM).
    const size_t share = cfg.cs > 1 ? static_cast<size_t>(cfg.tmem_cols) * (228 * 1024 / 512)
                                    : std::min<size_t>(static_cast<size_t>(cfg.tmem_cols) * (222 * 1024 / 512), 111 * 1024);
    smem = std::max(std::max(smem, share), NM_BESIDE_EXCLUSIVE);

    const long long images = BM / (static_cast<long long>(p.ho) * p.wo) + 2;   // images a pixel block can touch
    const bool wide = p.kh * p.kw > 64 || images * p.h * p.w * p.c_in * 4 >= (1ll << 32);
    const auto kernel = wide ? k_conv_gather<true> : k_conv_gather<false>;
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "cudaFuncSetAttribute (variant 1): %s", cudaGetErrorString(e));
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(static_cast<unsigned>(grid));
    lc.blockDim = dim3(THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute attr[3];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cfg.cs);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributePreferredSharedMemoryCarveout;   // the rest of two CTAs' SM is L1
    attr[1].val.sharedMemCarveout = static_cast<unsigned>(std::min<size_t>(100, (2 * (smem + 3072) * 100 + 228 * 1024 - 1) / (228 * 1024)));
    attr[2].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[2].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 3 : 2;
    e = cudaLaunchKernelEx(&lc, kernel, p, cfg);
    count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "nm_conv2d launch (variant 1): %s", cudaGetErrorString(e));
    return NM_OK;
}

}  // namespace nmhost
