// Variant 8: select kernel — persistent, warp-specialised sparse implicit GEMM that contracts over
// the RETAINED columns only (Algorithm 1); the fused im2col + packing pass of Sec. 3.2 is one 32-bit shared-memory load
// per retained element and tile.
//
// One CTA per SM walks a static list of work items: 128 output pixels x BN output channels
// (BN = G pruning tiles of T channels), optionally one of several ranges of the reduction axis.
// A STEP is one kernel tap of S source columns (32; 64 for 1:8), of which every tile keeps KC = 8, 16 or 24; steps are ordered
// by block of S channels, then tap.  A CHUNK is as many steps as fit 32 retained columns, a UNIT one tile's part of a
// chunk.  Roles, connected by mbarriers (every wait bounded):
//
//   activation producer   TMA brings the DENSE activations into shared memory, one 128-byte row per pixel
//   (1 thread)            and 32-channel block (128-byte swizzle), in one of two forms.  "im2col": a slot is one
//                         step, one im2col-mode load (stride, dilation, tap offset and zero padding done by the
//                         hardware).  "patch" (stride 1, output size = input size): the pixels of a block and
//                         their halo are CONSECUTIVE rows of the [pixels][channels] view of the input,
//                         so one plain 2-D load per channel block brings everything all kh*kw taps
//                         need; a tap is the same rows shifted by a constant, and where it falls outside the
//                         image a row of zeros behind the slot is read instead.  A 3x3 layer so moves
//                         a ninth of the im2col form's bytes through the TMA unit.
//   weight producer       one bulk copy per chunk brings the G tiles' retained weights [G*T x 32]
//   (1 thread)            (stored as the swizzled shared-memory image), another their column tables.
//   compactors (4 teams   a unit's operand [128 x 32] goes from the dense rows to the unit's columns of tensor memory:
//   of 4 warps)           a warp owns a lane quadrant; lane l loads columns 8 i + 2 (l % 4) and the next in rows
//                         l / 4 + 8 j, the fragment that tcgen05.st.16x256b stores.  The 8 rows of a load lie in
//                         8 different 16-byte pieces of the banks (the swizzle), so the load is free of conflicts
//                         where its four columns differ modulo 4: the order of a step's retained columns, which is
//                         free (the weights follow it), is chosen so at pruning time as far as the columns allow.
//                         A team works on two tiles at a time (they share the rows' addresses and the waits) where
//                         the item has two or four, and the teams take pairs and chunks in turn.
//   MMA issuers           D[128 x T] += A[tmem] * W[smem]^T, KC / 8 tcgen05.mma per step and unit, a thread per tile
//   (up to 4 threads)     (the T accumulators of Algorithm 1 are T TMEM columns).
//   epilogue (4 warps)    TMEM -> registers, + bias, (+ shortcut), ReLU, staged through shared memory
//                         and written to NHWC with TMA stores; with two accumulator buffers it
//                         overlaps the next item's main loop.
//
// What bounds it is the latency of its chains of barriers, loads, TMEM stores and MMAs, not a pipe: of 256 -> 256, 3x3 at
// 14x14, batch 128, 2:8 (32 us) 21 us remain without the shared-memory loads, the stores and the MMAs, and doubling the loads, the
// stores or the arithmetic costs nothing; sharing the address work and the waits between two tiles (55 -> 37 us), a second weight slot per
// team (37 -> 34) and short divisions per item (34 -> 32) did.  Before, with whole rows in registers and a chain of M - N
// bitwise selects per element, 93 us; the dense kernel 46.  The gain over the dense kernel grows with M / N: at 2:8
// 55 -> 38 us (128 -> 128 at 28x28), 74 -> 62 (64 -> 64 at 56x56), at 2:4, batch 64, 30 -> 29 and 45 -> 41, but 28.5 -> 31.5 at 14x14.
//
// Activations are fed to the tensor core as they are (it reads the upper 19 bits: truncation to
// TF32); weights were rounded to nearest at pruning time.
#include <algorithm>

#include "nm_internal.h"
#include "nm_ptx.cuh"
#include "nm_tmap.cuh"

namespace {

using namespace nmk;

constexpr int BM = 128;
constexpr int THREADS = 832;   // warps: 0 activation producer, 1 weight producer, 2 3 24 25 MMA issuers, 4-7 epilogue, 8-23 compactors
constexpr int TEAMS = 4;
constexpr int COMPACTORS = TEAMS * 4;
constexpr int MAX_P = 8;       // activation ring slots
constexpr int MAX_W = 8;       // weight ring slots
constexpr int N_SETS = TEAMS * 2;   // operand sets in tensor memory, 32 columns each
constexpr int MAX_ISS = 4;
constexpr int MAX_TAPS = 32;
constexpr int A_COL0 = 256;    // TMEM: accumulators in columns [0, 256), operand sets above
constexpr int MAX_BOXES = 8;       // per epilogue warp
constexpr int BOX_BYTES = 4096;    // staging box: 32 pixels x 32 channels
constexpr int RING_BUDGET = 227 * 1024 - 1024 - 1024;   // alignment slack, static shared
constexpr int TABLE_BYTES = 128;   // column table of a unit: [step][place in a quad][quad] 32-bit words

struct SelCfg {
    int g, bn, n_slices, n_acc, n_iss;
    int mma_n, sub;     // accumulator columns per MMA; MMAs (issuers) side by side in a tile: T = sub * mma_n
    int rows2d;         // 1 = 2-D loads of consecutive pixels, 0 = im2col loads
    int halo;           // 1 = patch form: a slot serves all taps of a channel block
    int taps;           // kh * kw
    int n_cb;           // blocks of S channels
    int steps;          // of the whole reduction axis: (channel block, tap), taps innermost
    int prow;           // rows the loads of one 32-channel block bring
    int lo;             // patch: first patch row relative to the block's first pixel (<= 0)
    int seg_bytes;      // one 32-channel block of a slot: prow rows, and eight rows of zeros in the patch form
    int p_bytes;        // activation slot
    int w_bytes;        // g * T * 128
    int m_bytes;        // g * TABLE_BYTES
    int wstage_bytes;   // w_bytes + m_bytes rounded up to 1024
    int n_p, n_w;
    int cycle;          // teams that take the chunks of a tile in turn (the weight ring has a multiple of it)
    int ksplit, p_pad;
    int alias_staging;  // 1: the output staging boxes lie over the start of the activation ring (one work item per CTA)
    int boxes;          // staging boxes per epilogue warp: 1 or 2, or one per channel block when aliased
    int staging_bytes;  // of all of them, 0 when aliased
    int chunks;         // of the whole reduction axis
    long long n_work;
    Divisor by_ksplit, by_slices, by_taps, by_hw, by_wo;
};

__device__ __forceinline__ bool aborted(volatile int* flag) { return *flag != 0; }

// Bounded wait that also gives up once another role has raised the abort flag (looked at every 64 polls, off
// the path of a wait that is already satisfied).
__device__ __forceinline__ bool wait_or_abort(uint32_t bar, uint32_t parity, volatile int* flag)
{
    if (mbar_test_wait(bar, parity)) return true;
    for (uint32_t i = 0; i < kWaitPolls; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 63u && *flag != 0) return false;
    }
    return false;
}

// The compactors' wait: gives up like the above, but its warp carries on (with whatever the buffers hold: the flag is set and the result
// is reported as failed), so that the loop needs no vote per wait.
__device__ __forceinline__ void wait_on(uint32_t bar, uint32_t parity, volatile int* flag)
{
    if (mbar_test_wait(bar, parity)) return;
    for (uint32_t i = 1; !mbar_try_wait(bar, parity); ++i)
        if (i == kWaitPolls || ((i & 63u) == 0 && *flag != 0)) { *flag = 3; break; }
}
__device__ __forceinline__ void arrive_if(bool on, uint32_t bar)
{
    asm volatile(
        "{\n\t"
        ".reg .pred p;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t"
        "}\n" ::"r"(bar), "r"(static_cast<uint32_t>(on))
        : "memory");
}

// Four consecutive 32-bit words of shared memory into dst[0..3].
__device__ __forceinline__ void lds128(uint32_t addr, uint32_t* dst)
{
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(dst[0]), "=r"(dst[1]), "=r"(dst[2]), "=r"(dst[3]) : "r"(addr));
}
template <int OFFSET>
__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(addr), "n"(OFFSET));
    return v;
}
// 16 lanes x 8 N columns: of columns 8 k .. 8 k + 7 thread l holds 8 k + 2 (l % 4) and the next, of lane l / 4 (v[4 k], v[4 k + 1]) and of
// lane l / 4 + 8 (v[4 k + 2], v[4 k + 3]).
template <int N>
__device__ __forceinline__ void tmem_st_frag(uint32_t taddr, const uint32_t* v)
{
    if constexpr (N == 3) {
        tmem_st_frag<2>(taddr, v);
        tmem_st_frag<1>(taddr + 16, v + 8);
    } else if constexpr (N == 2) {
        asm volatile("tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(v[0]), "r"(v[1]),
                     "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                     : "memory");
    } else {
        static_assert(N == 1, "unsupported operand width");
        asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
                     : "memory");
    }
}

// Retained columns of a step, source columns of a step, steps per chunk.
template <int KC_, int S_>
struct Pattern {
    static constexpr int KC = KC_, S = S_;
    static constexpr int SEGS = S / 32;
    static constexpr int SPC = 32 / KC;
    static constexpr int QUADS = KC / 4;
};

// This lane's words of a step's column table.
template <class P>
__device__ __forceinline__ void load_table(uint32_t at, uint32_t (&table)[P::QUADS])
{
    if constexpr (P::QUADS == 4) {
        lds128(at, table);
    } else {
#pragma unroll
        for (int i = 0; i < P::QUADS; i += 2)
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(table[i]), "=r"(table[i + 1]) : "r"(at + i * 4));
    }
}

// What a warp moves at a time: one step of G units, 32 rows x KC columns each; v[..][0] and [1]: lanes 0-15 and 16-31 of the quadrant.
// (Loading the next piece before this one is stored gained nothing: 37 us for 34.)
template <class P, int G>
struct Piece {
    uint32_t v[G][2][2 * P::QUADS];
    // r: this lane's rows, with their swizzle phase folded in; WHOLE: all at their places (8 rows apart: the same phase);
    // slot: where the activation slot begins (looked at by the self-checking build: a word outside it reads as zero)
    template <bool WHOLE>
    __device__ __forceinline__ void load(const uint32_t* r, uint32_t table_at, uint32_t seg_bytes, uint32_t slot, int* status)
    {
        auto in_slot = [&](uint32_t a) { return NM_ALLOWED(nm_bytes_in_span(a, 4, slot, slot + P::SEGS * seg_bytes), status, 802, a - slot); };
        uint32_t table[G][P::QUADS];
#pragma unroll
        for (int t = 0; t < G; ++t) load_table<P>(table_at + t * TABLE_BYTES, table[t]);
#pragma unroll
        for (int t = 0; t < G; ++t)
#pragma unroll
            for (int i = 0; i < P::QUADS; ++i) {
                const uint32_t at = P::SEGS == 1 ? table[t][i] : table[t][i] & 127u;
                const uint32_t seg = P::SEGS == 1 ? 0u : (table[t][i] >> 7) * seg_bytes;
                const int k = (i >> 1) * 4 + (i & 1);
                if (NM_SELF_CHECKING) {
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t a = ((WHOLE ? r[0] : r[e]) ^ at) + seg + (WHOLE ? e * 1024u : 0u);
                        v[t][e >> 1][k + (e & 1) * 2] = in_slot(a) ? lds32<0>(a) : 0u;
                    }
                } else if (WHOLE) {
                    const uint32_t a = (r[0] ^ at) + seg;
                    v[t][0][k] = lds32<0>(a);
                    v[t][0][k + 2] = lds32<1024>(a);
                    v[t][1][k] = lds32<2048>(a);
                    v[t][1][k + 2] = lds32<3072>(a);
                } else {
                    v[t][0][k] = lds32<0>((r[0] ^ at) + seg);
                    v[t][0][k + 2] = lds32<0>((r[1] ^ at) + seg);
                    v[t][1][k] = lds32<0>((r[2] ^ at) + seg);
                    v[t][1][k + 2] = lds32<0>((r[3] ^ at) + seg);
                }
            }
    }
    __device__ __forceinline__ void store(uint32_t dst) const
    {
#pragma unroll
        for (int t = 0; t < G; ++t) {
            tmem_st_frag<P::QUADS / 2>(dst + t * 32, v[t][0]);
            tmem_st_frag<P::QUADS / 2>(dst + t * 32 + (16u << 16), v[t][1]);
        }
    }
};

struct Item {
    int split, slice;
    uint32_t pix0;
    int c_begin, c_end;   // chunks
};
__device__ __forceinline__ Item item_of(uint32_t work, const SelCfg& cfg)
{
    Item it;
    const int rest = div_by(static_cast<int>(work), cfg.by_ksplit), block = div_by(rest, cfg.by_slices);
    it.split = static_cast<int>(work) - rest * cfg.ksplit;
    it.slice = rest - block * cfg.n_slices;
    it.pix0 = static_cast<uint32_t>(block) * BM;
    it.c_begin = div_by(it.split * cfg.chunks, cfg.by_ksplit);
    it.c_end = div_by((it.split + 1) * cfg.chunks, cfg.by_ksplit);
    return it;
}

template <class P, int HALO, int TPW>
__global__ void __launch_bounds__(THREADS, 1)
k_conv_select(const ConvParams p, const SelCfg cfg, const __grid_constant__ CUtensorMap tm_x,
              const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_res)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_pfull[MAX_P], s_pfree[MAX_P], s_wfull[MAX_W], s_wfree[MAX_W], s_aready[N_SETS], s_afree[N_SETS], s_accfull[2],
        s_accfree[2], s_res[4][MAX_BOXES];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort, s_shift[MAX_TAPS];

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const uint32_t n_work = static_cast<uint32_t>(cfg.n_work);   // below 2^31: per-item arithmetic stays 32-bit
    const int g = cfg.g;
    const uint32_t p_ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t w_ring = p_ring + cfg.n_p * cfg.p_bytes;
    const uint32_t ring_end = w_ring + cfg.n_w * cfg.wstage_bytes;
    // with one work item per CTA the epilogue starts when every load has been consumed: its staging boxes reuse the ring
    const uint32_t staging = cfg.alias_staging ? p_ring : ring_end;
    volatile int* abort_flag = &s_abort;

    // ---- set-up ----------------------------------------------------------------------------------
    if (warp == 2) tmem_alloc(smem_u32(&s_tmem), 512);
    if (tid == 0) {
        for (int i = 0; i < MAX_P; ++i) {
            mbar_init(smem_u32(&s_pfull[i]), 1);              // producer's expect-tx arrival
            mbar_init(smem_u32(&s_pfree[i]), COMPACTORS);     // every warp waits for and releases every slot: a wait by parity has to see all uses
        }
        for (int i = 0; i < MAX_W; ++i) {
            mbar_init(smem_u32(&s_wfull[i]), 1);
            // The warps that work on a slot's chunks (always the same: `cycle` divides the number of slots), one MMA commit per issuer
            mbar_init(smem_u32(&s_wfree[i]), 4 * (g / TPW) + cfg.n_iss);
        }
        for (int i = 0; i < TEAMS * 2; ++i) {
            mbar_init(smem_u32(&s_aready[i]), 4);         // the team's warps: operands written AND weights landed
            mbar_init(smem_u32(&s_afree[i]), TPW * cfg.sub);   // the tiles' issuers
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&s_accfull[i]), cfg.n_iss);
            mbar_init(smem_u32(&s_accfree[i]), 4);  // epilogue warps
        }
        for (int i = 0; i < 4 * MAX_BOXES; ++i) mbar_init(smem_u32(&s_res[0][0] + i), 1);   // a shortcut box has landed
        mbar_fence_init();
        s_abort = 0;
        tma_prefetch_desc(&tm_x);
        tma_prefetch_desc(&tm_y);
    }
    if (HALO && tid < cfg.taps)   // patch form: rows between the first patch row and a pixel's source row of the tap
        s_shift[tid] = (tid / p.kw * p.dil_h - p.pad_h) * p.w + tid % p.kw * p.dil_w - p.pad_w - cfg.lo;
    if (HALO)   // the rows of zeros behind every 32-channel block: eight, one per swizzle phase (no conflict with the others' banks)
        for (int i = tid; i < cfg.n_p * P::SEGS * 64; i += blockDim.x) {
            const uint32_t at = p_ring + static_cast<uint32_t>(i >> 6) * cfg.seg_bytes + cfg.prow * 128u + static_cast<uint32_t>(i & 63) * 16u;
            asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(at), "r"(0u) : "memory");
        }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    pdl_launch_dependents();   // the next kernel may start its own set-up as SMs become free
    if (warp != 1) pdl_wait(); // from here on global memory written by the previous kernel is read (weights are no kernel's output)

    if (warp == 0) {
        // =========================== activation producer ===========================
        if (elect_one()) {
            const int hw = p.ho * p.wo;
            RingPos rp;
            int issued = 0;
            for (uint32_t work = blockIdx.x; work < n_work && !aborted(abort_flag); work += gridDim.x) {
                const Item it = item_of(work, cfg);
                const int n0 = div_by(static_cast<int>(it.pix0), cfg.by_hw), rem = static_cast<int>(it.pix0) - n0 * hw;
                const int oh0 = div_by(rem, cfg.by_wo), ow0 = rem - oh0 * p.wo;
                const int w0 = ow0 * p.stride_w - p.pad_w, h0 = oh0 * p.stride_h - p.pad_h;
                auto load = [&](int cb, int ti, int tj) {
                    if (rp.wrapped && !mbar_wait_lone(smem_u32(&s_pfree[rp.s]), rp.parity ^ 1u)) *abort_flag = 2;
                    if (aborted(abort_flag)) return;
                    const uint32_t dst = p_ring + rp.s * cfg.p_bytes;
                    const uint32_t bar = smem_u32(&s_pfull[rp.s]);
                    mbar_arrive_expect_tx(bar, static_cast<uint32_t>(P::SEGS * cfg.prow) * 128u);
#pragma unroll
                    for (int seg = 0; seg < P::SEGS; ++seg) {
                        const int ch = (cb * P::SEGS + seg) * 32;
                        if (cfg.rows2d)
                            tma_load_2d(dst + seg * cfg.seg_bytes, &tm_x, bar, ch, static_cast<int>(it.pix0) + cfg.lo);
                        else
                            tma_load_im2col_4d(dst + seg * cfg.seg_bytes, &tm_x, bar, ch, w0, h0, n0,
                                               static_cast<uint16_t>(tj * p.dil_w), static_cast<uint16_t>(ti * p.dil_h));
                    }
                    rp.advance(cfg.n_p);
                    ++issued;
                };
                const int first = it.c_begin * P::SPC, last = min(it.c_end * P::SPC, cfg.steps) - 1;
                int cb = div_by(first, cfg.by_taps);
                if (HALO) {
                    for (const int cb_last = div_by(last, cfg.by_taps); cb <= cb_last && !aborted(abort_flag); ++cb) load(cb, 0, 0);
                } else {
                    int tap = first - cb * cfg.taps;
                    int ti = tap / p.kw, tj = tap - ti * p.kw;
                    for (int i = first; i <= last && !aborted(abort_flag); ++i) {
                        load(cb, ti, tj);
                        if (++tj == p.kw) { tj = 0; ++ti; }
                        if (++tap == cfg.taps) { tap = ti = tj = 0; ++cb; }
                    }
                }
            }
            if (aborted(abort_flag)) {
                // loads already issued still target this CTA's shared memory: let them land
                for (int back = 0; back < cfg.n_p && back < issued; ++back) {
                    if (rp.s == 0) { rp.s = cfg.n_p; rp.parity ^= 1u; }
                    --rp.s;
                    (void)mbar_wait(smem_u32(&s_pfull[rp.s]), rp.parity);
                }
            }
        }
    } else if (warp == 1) {
        // =========================== weight producer ===========================
        if (elect_one()) {
            RingPos rw;
            int issued = 0;
            const size_t chunk_floats = static_cast<size_t>(p.c_out) * 32;
            const size_t chunk_mbytes = static_cast<size_t>(p.n_tiles) * TABLE_BYTES;
            const uint32_t tx = static_cast<uint32_t>(cfg.w_bytes + cfg.m_bytes);
            for (uint32_t work = blockIdx.x; work < n_work && !aborted(abort_flag); work += gridDim.x) {
                const Item it = item_of(work, cfg);
                const float* wsl = p.w3 + static_cast<size_t>(it.slice) * cfg.bn * 32;
                const uint8_t* msl = p.sel3 + static_cast<size_t>(it.slice) * g * TABLE_BYTES;
                for (int c = it.c_begin; c < it.c_end; ++c) {
                    if (rw.wrapped && !mbar_wait_lone(smem_u32(&s_wfree[rw.s]), rw.parity ^ 1u)) *abort_flag = 9;
                    if (aborted(abort_flag)) break;
                    const uint32_t dst = w_ring + rw.s * cfg.wstage_bytes;
                    const uint32_t bar = smem_u32(&s_wfull[rw.s]);
                    mbar_arrive_expect_tx(bar, tx);
                    bulk_load_1d(dst, wsl + static_cast<size_t>(c) * chunk_floats, static_cast<uint32_t>(cfg.w_bytes), bar);
                    bulk_load_1d(dst + cfg.w_bytes, msl + static_cast<size_t>(c) * chunk_mbytes, static_cast<uint32_t>(cfg.m_bytes), bar);
                    rw.advance(cfg.n_w);
                    ++issued;
                }
            }
            if (aborted(abort_flag)) {
                for (int back = 0; back < cfg.n_w && back < issued; ++back) {
                    if (rw.s == 0) { rw.s = cfg.n_w; rw.parity ^= 1u; }
                    --rw.s;
                    (void)mbar_wait(smem_u32(&s_wfull[rw.s]), rw.parity);
                }
            }
        }
    } else if (warp == 2 || warp == 3 || warp == 24 || warp == 25) {
        // =========================== MMA issuers ===========================
        const int iss = warp < 4 ? warp - 2 : warp - 22;
        if (iss < cfg.n_iss && elect_one()) {
            const uint32_t idesc = umma_idesc_tf32(BM, cfg.mma_n);
            const int tile = iss / cfg.sub;
            const int cycle = cfg.cycle;         // teams that take this tile's chunks in turn
            const int first_team = tile / TPW, step_team = g / TPW;
            RingPos rw;
            int turn = 0;
            uint32_t use = 0;                    // how often the team at its turn has had one
            uint32_t ab = 0, acc_par = 0;
            bool acc_wrapped = false;
            // A chunk is ready when its compactor team has arrived: the team waits for the chunk's weights (they
            // come with its table) before it starts, so this one barrier stands for both.
            for (uint32_t work = blockIdx.x; work < n_work && !aborted(abort_flag); work += gridDim.x) {
                const Item it = item_of(work, cfg);
                if (acc_wrapped && !wait_or_abort(smem_u32(&s_accfree[ab]), acc_par ^ 1u, abort_flag)) {
                    *abort_flag = 5;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + ab * cfg.bn + iss * cfg.mma_n;
                for (int c = it.c_begin; c < it.c_end; ++c) {
                    // two operand sets per team: for its two tiles, or for every other unit of its one
                    const uint32_t team2 = static_cast<uint32_t>(first_team + turn * step_team) * 2;
                    const uint32_t bar = TPW == 2 ? team2 : team2 + (use & 1u);
                    const uint32_t set = TPW == 2 ? team2 + (tile & 1) : bar;
                    if (!wait_or_abort(smem_u32(&s_aready[bar]), (TPW == 2 ? use : use >> 1) & 1u, abort_flag)) { *abort_flag = 7; break; }
                    tc_fence_after();
                    const uint32_t b_smem = w_ring + rw.s * cfg.wstage_bytes + iss * cfg.mma_n * 128;
                    const uint32_t a_set = tmem + A_COL0 + set * 32;
                    const uint64_t bdesc = umma_desc_k_sw128(b_smem, 1024);
                    const int ksteps = min(P::SPC, cfg.steps - c * P::SPC) * (P::KC / 8);
#pragma unroll
                    for (int kq = 0; kq < P::SPC * P::KC / 8; ++kq)
                        if (kq < ksteps) {
                            NM_CHECKED(((acc - tmem) & 0xFFFFu) + cfg.mma_n <= 256u && ((a_set - tmem) & 0xFFFFu) + kq * 8 + 8 <= 512u &&
                                           b_smem + cfg.mma_n * 128 <= ring_end && b_smem >= w_ring,
                                       p.status, 801, iss * 1000 + kq)
                            umma_tf32_ts(acc, a_set + kq * 8, bdesc + 2 * kq, idesc, (c > it.c_begin || kq > 0) ? 1u : 0u);
                        }
                    umma_commit(smem_u32(&s_afree[bar]));
                    umma_commit(smem_u32(&s_wfree[rw.s]));
                    rw.advance(cfg.n_w);
                    if (++turn == cycle) {
                        turn = 0;
                        ++use;
                    }
                }
                if (aborted(abort_flag)) break;
                umma_commit(smem_u32(&s_accfull[ab]));
                if (cfg.n_acc == 2) {
                    if (ab == 1) { acc_par ^= 1u; acc_wrapped = true; }
                    ab ^= 1u;
                } else {
                    acc_par ^= 1u;
                    acc_wrapped = true;
                }
            }
        }
    } else if (warp >= 4 && warp < 8) {
        // =========================== epilogue ===========================
        const int q = warp & 3;
        const uint32_t lane_addr = static_cast<uint32_t>(q * 32) << 16;
        const uint32_t my_staging = staging + q * cfg.boxes * BOX_BYTES;
        const uint32_t rx = static_cast<uint32_t>(lane & 7);
        const int n_blk = cfg.bn / 32;
        const int n_box = cfg.boxes;
        int bx = 0;                 // staging box of the next block, parity of its shortcut barrier
        uint32_t bpar = 0;
        // The shortcut comes by TMA into the very boxes the sums are staged in, n_box - 1 blocks ahead: the cursor of its requests.
        uint32_t rwork = blockIdx.x, asked = 0, taken = 0;
        int rblk = 0, rbx = 0;
        auto request = [&]() {
            if (rwork >= n_work) return;
            if (elect_one()) {
                const Item it = item_of(rwork, cfg);
                const uint32_t bar = smem_u32(&s_res[q][rbx]);
                mbar_arrive_expect_tx(bar, BOX_BYTES);
                tma_load_2d(my_staging + rbx * BOX_BYTES, &tm_res, bar, it.slice * cfg.bn + rblk * 32, static_cast<int>(it.pix0) + q * 32);
            }
            ++asked;
            if (++rblk == n_blk) { rblk = 0; rwork += gridDim.x; }
            if (++rbx == n_box) rbx = 0;
        };
        const bool res = p.residual != nullptr;
        auto request_first = [&]() {
            for (int i = 0; i + 1 < n_box; ++i) request();
        };
        if (res && !cfg.alias_staging) request_first();
        uint32_t ti = 0;
        for (uint32_t work = blockIdx.x; work < n_work; work += gridDim.x, ++ti) {
            const Item it = item_of(work, cfg);
            const int ab = cfg.n_acc == 2 ? static_cast<int>(ti & 1u) : 0;
            const int o0 = it.slice * cfg.bn;
            // bias of the item's blocks, a channel per lane, fetched while the main loop runs
            float bias_of[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) bias_of[i] = i < n_blk ? bias_lane_load(p.bias, o0 + i * 32, p.c_out, lane) : 0.f;
            const bool ok = aborted(abort_flag) ||
                            mbar_wait(smem_u32(&s_accfull[ab]), (cfg.n_acc == 2 ? (ti >> 1) : ti) & 1u);
            if (!__all_sync(0xFFFFFFFFu, ok)) *abort_flag = 8;
            if (__any_sync(0xFFFFFFFFu, aborted(abort_flag))) break;
            tc_fence_after();
            if (res && cfg.alias_staging) request_first();   // (the rings the boxes lie over are idle now)
            // a split of the reduction axis stores raw partial sums [split][pixel][channel] (bias, shortcut and
            // activation are switched off by the launcher and applied by the reduction pass)
            const long long box_pix = static_cast<long long>(it.pix0) + q * 32;
            const int store_row = it.split * cfg.p_pad + static_cast<int>(it.pix0) + q * 32;
            const bool in_range = cfg.ksplit > 1 || box_pix < p.pixels;
            for (int blk = 0; blk < n_blk; ++blk) {
                uint32_t v[32];
                tmem_ld32(tmem + lane_addr + ab * cfg.bn + blk * 32, v);
                tmem_ld_wait(v);
                if (blk + 1 == n_blk) {
                    // the accumulator buffer may be overwritten from here on
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&s_accfree[ab]));
                }
                if (res) {
                    // the store of the block before this one must have read its box, the next one to be loaded
                    if (elect_one()) tma_store_wait_read();
                    __syncwarp();
                    request();
                    const bool landed = mbar_wait_lone(smem_u32(&s_res[q][bx]), bpar);
                    if (!__all_sync(0xFFFFFFFFu, landed)) *abort_flag = 11;
                    ++taken;
                } else {
                    // the store that last read this box must be done with it
                    if (elect_one()) {
                        if (n_box >= 2) tma_store_wait_read_n<1>();
                        else tma_store_wait_read();
                    }
                    __syncwarp();
                }
                const uint32_t box = my_staging + bx * BOX_BYTES;
                const uint32_t stage_row = box + lane * 128;
                // (All shuffles and loads before the first store: they are ordered statements, one would wait for the other's result.  With this and
                // the bias fetched ahead 82 pairs of layer and plan take 0.979 of the time in the middle, split ones 0.93: 256 -> 256, 3x3 at 14x14, batch 64,
                // 2:4 30.9 -> 30.6 us, 64 -> 256, 1x1 at 56x56, batch 64 59.7 -> 48.5.  64 -> 64, 3x3 at 56x56, batch 128 got slower: 2:8 58.6 -> 59.5, 1:4
                // in one group of two tiles 66.8 -> 70.4.  So it did with the bias through shared memory, loaded a block ahead or after the wait,
                // with four loads at a time, and with a load through L2 as the only change: the selecting warps' schedule, not the epilogue.)
                float4 o8[8];
#pragma unroll
                for (int qq = 0; qq < 8; ++qq) {
                    o8[qq] = make_float4(__uint_as_float(v[qq * 4 + 0]), __uint_as_float(v[qq * 4 + 1]), __uint_as_float(v[qq * 4 + 2]),
                                         __uint_as_float(v[qq * 4 + 3]));
                    nm_add4(o8[qq], bias_quad(bias_of[0], qq));
                }
#pragma unroll
                for (int i = 0; i < 7; ++i) bias_of[i] = bias_of[i + 1];
                if (res) {
#pragma unroll
                    for (int half = 0; half < 8; half += 4) {
                        float4 x[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[i].x), "=f"(x[i].y), "=f"(x[i].z), "=f"(x[i].w)
                                         : "r"(stage_row + (((half + i) ^ rx) << 4)));
#pragma unroll
                        for (int i = 0; i < 4; ++i) nm_add4(o8[half + i], x[i]);
                    }
                }
#pragma unroll
                for (int qq = 0; qq < 8; ++qq) {
                    const uint32_t at = stage_row + ((qq ^ rx) << 4);
                    float4 o = o8[qq];
                    if (p.relu) { o.x = fmaxf(o.x, 0.f); o.y = fmaxf(o.y, 0.f); o.z = fmaxf(o.z, 0.f); o.w = fmaxf(o.w, 0.f); }
                    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(o.x), "f"(o.y), "f"(o.z), "f"(o.w) : "memory");
                }
                fence_proxy_async();
                __syncwarp();
                if (elect_one()) {
                    if (in_range) tma_store_2d(&tm_y, box, o0 + blk * 32, store_row);
                    tma_store_commit();
                }
                if (++bx == n_box) { bx = 0; bpar ^= 1u; }
            }
        }
        if (aborted(abort_flag))   // shortcut boxes still on their way to this CTA's shared memory (bounded)
            for (; taken != asked; ++taken) {
                (void)mbar_wait_polls(smem_u32(&s_res[q][bx]), bpar, 1u << 16);
                if (++bx == n_box) { bx = 0; bpar ^= 1u; }
            }
        if (elect_one()) tma_store_wait_read();   // shared memory must outlive the stores' reads; the writes complete with the grid
    } else if (warp >= 8 && warp < 24) {
        // =========================== compactors ===========================
        const int team = (warp - 8) >> 2;
        const int q = warp & 3;                                       // TMEM lane quadrant
        const int cycle = cfg.cycle, groups = g / TPW;                // teams side by side
        const int tile0 = team % groups * TPW;
        const int first_row = q * 32 + (lane >> 2);                   // and 8, 16, 24 rows on
        const int hw = p.ho * p.wo;
        // chunks until this team's next (three tiles leave the fourth team none)
        int until = team / groups < cycle ? team / groups : 0x0FFFFFFF;
        const uint32_t set_col = tmem + (static_cast<uint32_t>(q * 32) << 16) + A_COL0 + static_cast<uint32_t>(team) * 64;
        const uint32_t aready = smem_u32(&s_aready[team * 2]), afree = smem_u32(&s_afree[team * 2]);
        const uint32_t wfull = smem_u32(&s_wfull[0]), wfree = smem_u32(&s_wfree[0]);
        const uint32_t pfull = smem_u32(&s_pfull[0]), pfree = smem_u32(&s_pfree[0]);
        const uint32_t table_base = w_ring + cfg.w_bytes + tile0 * TABLE_BYTES + (lane & 3) * (P::QUADS * 4);
        const bool first_lane = lane == 0;
        // places in the rings (ws, ps: of their barriers)
        uint32_t ws = static_cast<uint32_t>(team / groups) * 8, wpar = 0, tab = table_base + static_cast<uint32_t>(team / groups) * cfg.wstage_bytes;
        uint32_t ps = 0, ppar = 0, act = p_ring;
        uint32_t uses = 0;                                            // chunks of this team so far
        // this chunk's operand sets; they were last read by the MMAs of the team's chunk before (two before)
        auto set_at = [&]() { return TPW == 2 ? set_col : set_col + (uses & 1u) * 32; };
        auto set_free = [&]() {
            const uint32_t n = TPW == 2 ? uses : uses >> 1;   // uses of these sets so far
            if (n > 0) wait_on(TPW == 2 ? afree : afree + (uses & 1u) * 8, (n & 1u) ^ 1u, abort_flag);
            __syncwarp();
            tc_fence_after();
        };
        auto begin_chunk = [&]() {   // weights and table landed
            wait_on(wfull + ws, wpar, abort_flag);
            __syncwarp();
        };
        auto end_chunk = [&]() {
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            arrive_if(first_lane, TPW == 2 ? aready : aready + (uses & 1u) * 8);
            arrive_if(first_lane, wfree + ws);
            ++uses;
            ws += static_cast<uint32_t>(cycle) * 8;
            tab += cycle * cfg.wstage_bytes;
            if (ws >= static_cast<uint32_t>(cfg.n_w) * 8) {
                ws -= static_cast<uint32_t>(cfg.n_w) * 8;
                tab -= cfg.n_w * cfg.wstage_bytes;
                wpar ^= 1u;
            }
        };
        Piece<P, TPW> piece;
        auto next_slot = [&]() {
            __syncwarp();
            arrive_if(first_lane, pfree + ps);
            ps += 8;
            act += cfg.p_bytes;
            if (ps == static_cast<uint32_t>(cfg.n_p) * 8) { ps = 0; act = p_ring; ppar ^= 1u; }
        };
        for (uint32_t work = blockIdx.x; work < n_work; work += gridDim.x) {
            const Item it = item_of(work, cfg);
            uint32_t v0 = 0, v1 = 0, v2 = 0, v3 = 0, all = 0;   // taps inside the image for this lane's rows; for all the warp's rows
            if (HALO) {
                uint32_t mine = 0;   // lane l: row l of the quadrant
                const long long pix = static_cast<long long>(it.pix0) + q * 32 + lane;
                if (pix < p.pixels) {
                    const int rem = static_cast<int>(pix) - div_by(static_cast<int>(pix), cfg.by_hw) * hw;
                    const int oh = div_by(rem, cfg.by_wo), ow = rem - oh * p.wo;
                    uint32_t cols = 0;
                    for (int j = 0; j < p.kw; ++j)
                        cols |= (static_cast<uint32_t>(ow + j * p.dil_w - p.pad_w) < static_cast<uint32_t>(p.w) ? 1u : 0u) << j;
                    for (int i = 0; i < p.kh; ++i)
                        if (static_cast<uint32_t>(oh + i * p.dil_h - p.pad_h) < static_cast<uint32_t>(p.h)) mine |= cols << (i * p.kw);
                }
                all = __reduce_and_sync(0xFFFFFFFFu, mine);
                v0 = __shfl_sync(0xFFFFFFFFu, mine, lane >> 2);
                v1 = __shfl_sync(0xFFFFFFFFu, mine, (lane >> 2) + 8);
                v2 = __shfl_sync(0xFFFFFFFFu, mine, (lane >> 2) + 16);
                v3 = __shfl_sync(0xFFFFFFFFu, mine, (lane >> 2) + 24);
            }
            if (__any_sync(0xFFFFFFFFu, aborted(abort_flag))) break;
            if (HALO) {
                const int first = it.c_begin * P::SPC, end = min(it.c_end * P::SPC, cfg.steps), left = it.c_end - it.c_begin;
                const int cb0 = div_by(first, cfg.by_taps);
                int slots = div_by(end - 1, cfg.by_taps) - cb0;              // after the current one
                int tap = first - cb0 * cfg.taps + until * P::SPC;   // of the next step, counted from the current slot's first
                auto turn_slot = [&]() {
                    next_slot();
                    --slots;
                    tap -= cfg.taps;
                    wait_on(pfull + ps, ppar, abort_flag);
                    __syncwarp();
                };
                wait_on(pfull + ps, ppar, abort_flag);
                __syncwarp();
                for (; until < left; until += cycle) {
                    while (tap >= cfg.taps) turn_slot();
                    begin_chunk();
                    const int steps = min(P::SPC, end - first - until * P::SPC);
                    const uint32_t dst = set_at();
#pragma unroll
                    for (int s = 0; s < P::SPC; ++s) {
                        if (s >= steps) break;
                        if (tap == cfg.taps) turn_slot();
                        const uint32_t row = static_cast<uint32_t>(first_row + s_shift[tap]);
                        const uint32_t phase = (row & 7u) << 4, bit = 1u << tap;
                        uint32_t rows[4] = {act + row * 128u + phase};
                        const uint32_t table_at = tab + s * (P::KC * 4);
                        if (all & bit) {
                            piece.template load<true>(rows, table_at, cfg.seg_bytes, act, p.status);
                        } else {
                            const uint32_t zero = act + cfg.prow * 128u + (phase << 3) + phase;
                            rows[1] = v1 & bit ? rows[0] + 1024u : zero;
                            rows[2] = v2 & bit ? rows[0] + 2048u : zero;
                            rows[3] = v3 & bit ? rows[0] + 3072u : zero;
                            rows[0] = v0 & bit ? rows[0] : zero;
                            piece.template load<false>(rows, table_at, cfg.seg_bytes, act, p.status);
                        }
                        if (s == 0) set_free();
                        piece.store(dst + s * P::KC);
                        ++tap;
                    }
                    end_chunk();
                    tap += (cycle - 1) * P::SPC;
                }
                until -= left;
                while (slots > 0) turn_slot();
                next_slot();
            } else {
                for (int c = it.c_begin; c < it.c_end; ++c) {
                    const int steps = min(P::SPC, cfg.steps - c * P::SPC);
                    const bool mine = until == 0;
                    if (mine) begin_chunk();
                    const uint32_t dst = set_at();
#pragma unroll
                    for (int s = 0; s < P::SPC; ++s) {
                        if (s >= steps) break;
                        wait_on(pfull + ps, ppar, abort_flag);
                        __syncwarp();
                        if (mine) {
                            const uint32_t row = act + first_row * 128u + ((lane >> 2) << 4);
                            piece.template load<true>(&row, tab + s * (P::KC * 4), cfg.seg_bytes, act, p.status);
                            if (s == 0) set_free();
                            piece.store(dst + s * P::KC);
                        }
                        next_slot();
                    }
                    if (mine) end_chunk();
                    until = mine ? cycle - 1 : until - 1;
                }
            }
        }
    }

    // ---- common exit ---------------------------------------------------------------------------------
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort != 0) {
        atomicExch(p.status + 0, static_cast<int>(NM_ERR_TIMEOUT));
        atomicExch(p.status + 1, 80 + s_abort);
        atomicExch(p.status + 2, static_cast<int>(blockIdx.x));
    }
    if (warp == 2) tmem_dealloc(tmem, 512);
}

// ---- launch configuration --------------------------------------------------------------------------

// Source and retained columns of a step: 32 source columns, or 64 where those keep too few for an MMA's depth of 8.  Groups
// may not cross steps.  False: the kernel does not cover the pattern.
bool pattern_dims(int n_keep, int m_group, int* s, int* kc)
{
    if (n_keep < 1 || n_keep >= m_group) return false;
    for (int S : {32, 64}) {
        const int KC = S % m_group == 0 ? S / m_group * n_keep : 0;
        if ((S == 32 && (KC == 8 || KC == 16 || KC == 24)) || (S == 64 && KC == 8)) {
            *s = S;
            *kc = KC;
            return true;
        }
    }
    return false;
}

bool make_cfg(const ConvParams& p, const nm_plan_t* plan, SelCfg* cfg)
{
    if (!p.w3 || !p.sel3 || !nmtm::available()) return false;
    int S = 0, KC = 0;
    if (!pattern_dims(p.n_keep, p.m_group, &S, &KC)) return false;
    if (p.sel_s != S || p.sel_kc != KC) return false;   // the handle's layout is this kernel's
    const int T = p.tile_t;
    if (p.c_in % S != 0 || T % 16 != 0 || T > 256 || p.c_out % T != 0) return false;
    if (static_cast<long long>(p.batch) * p.h * p.w * p.c_in * 4 < 131072) return false;   // tensor maps of tiny inputs: other kernels
    if (p.pixels >= (1ll << 31) - BM) return false;
    const int taps = p.kh * p.kw;
    // activation loads: consecutive pixels need stride 1, an output of the input's size, and a halo that fits a TMA box
    const int lo = -(p.pad_h * p.w + p.pad_w);
    const int hi = ((p.kh - 1) * p.dil_h - p.pad_h) * p.w + (p.kw - 1) * p.dil_w - p.pad_w;
    const bool patch_ok = p.stride_h == 1 && p.stride_w == 1 && p.ho == p.h && p.wo == p.w && taps <= MAX_TAPS && hi >= 0 &&
                          BM + hi - lo <= 256 && static_cast<long long>(p.batch) * p.h * p.w < (1ll << 31);
    int loads = plan ? plan->loads : 0;
    if (loads == 0) loads = patch_ok ? 2 : 1;
    if (loads == 2 && !patch_ok) return false;
    if (loads == 1 && !nmtm::im2col_geometry_ok(p)) return false;
    if (loads != 1 && loads != 2) return false;
    cfg->rows2d = loads == 2;
    cfg->halo = loads == 2 && taps > 1;
    cfg->taps = taps;
    cfg->n_cb = p.c_in / S;
    cfg->steps = cfg->n_cb * taps;
    cfg->chunks = (cfg->steps + 32 / KC - 1) / (32 / KC);
    cfg->lo = cfg->halo ? lo : 0;
    cfg->prow = cfg->halo ? ((BM + hi - lo + 7) / 8) * 8 : BM;
    cfg->seg_bytes = (cfg->prow + (cfg->halo ? 8 : 0)) * 128;
    cfg->p_bytes = (S / 32) * cfg->seg_bytes;
    int g;
    if (plan && plan->bn > 0) {
        if (plan->bn % T != 0) return false;
        g = plan->bn / T;
    } else {
        g = 1;
        for (int cand = 4; cand >= 1; --cand)
            if (cand * T <= 256 && p.n_tiles % cand == 0 && (cand * T) % 32 == 0) { g = cand; break; }
    }
    if (g < 1 || g > 4 || g * T > 256 || p.n_tiles % g != 0 || (g * T) % 32 != 0) return false;
    cfg->g = g;
    cfg->bn = g * T;
    cfg->n_slices = p.n_tiles / g;
    cfg->n_acc = cfg->bn <= 128 ? 2 : 1;
    // An issuer per tile, or several side by side where the plan asks for more.
    const int want = plan && plan->issuers > 0 ? plan->issuers : g;
    if (want > MAX_ISS) return false;
    int sub = 1;
    while (g * sub < want && g * sub * 2 <= MAX_ISS) sub *= 2;
    while (sub > 1 && (T % sub != 0 || (T / sub) % 16 != 0)) sub /= 2;
    cfg->sub = sub;
    cfg->mma_n = T / sub;
    cfg->n_iss = g * sub;
    cfg->cycle = g == 4 ? 2 : g == 3 ? 1 : 4;
    cfg->w_bytes = cfg->bn * 128;
    cfg->m_bytes = g * TABLE_BYTES;
    cfg->wstage_bytes = ((cfg->w_bytes + cfg->m_bytes + 1023) / 1024) * 1024;
    // split of the reduction axis: whole chunks per range
    if (plan && (plan->ksplit > 8 || plan->split < 0 || plan->split > 2)) return false;
    const int asked = plan && plan->ksplit > 1 ? plan->ksplit : 1, ksplit = std::min(asked, cfg->chunks);   // (no more ranges than chunks)
    cfg->ksplit = ksplit;
    cfg->p_pad = static_cast<int>(((p.pixels + BM - 1) / BM) * BM);
    if (asked > 1 && (!p.splitk || p.c_out % 4 != 0 ||
                      p.splitk_bytes < static_cast<size_t>(asked) * cfg->p_pad * p.c_out * sizeof(float) ||
                      static_cast<long long>(asked) * cfg->p_pad >= (1ll << 31)))
        return false;   // the partial-sum scratch is reserved by nm_autotune / nm_weights_reserve
    const long long pix_blocks = (p.pixels + BM - 1) / BM;
    cfg->n_work = pix_blocks * cfg->n_slices * ksplit;
    if (cfg->n_work >= (1ll << 31)) return false;
    cfg->by_ksplit = divisor(ksplit);
    cfg->by_slices = divisor(cfg->n_slices);
    cfg->by_taps = divisor(taps);
    cfg->by_hw = divisor(p.ho * p.wo);
    cfg->by_wo = divisor(p.wo);
    cfg->alias_staging = cfg->n_work <= nmhost::sm_count();
    // Staging boxes per warp: three with a shortcut (it is requested two blocks ahead; fewer where a plan's rings need the room), one
    // where the epilogue has a long main loop beside it and the rings need it (256 -> 256, 3x3 at 14x14, 2:8: 37 -> 34 us),
    // else two.
    cfg->boxes = p.residual ? 3 : cfg->n_acc == 2 && cfg->chunks / ksplit >= 16 ? 1 : 2;
    const int ring_min = (plan && plan->stages > 0 ? plan->stages : 1) * cfg->p_bytes + std::max(2, cfg->cycle) * cfg->wstage_bytes;
    while (cfg->boxes > 1 && !cfg->alias_staging && ring_min + 4 * cfg->boxes * BOX_BYTES > RING_BUDGET) --cfg->boxes;
    cfg->staging_bytes = cfg->alias_staging ? 0 : 4 * cfg->boxes * BOX_BYTES;
    // Shared memory: alignment slack, static shared, the output staging unless it can lie over the ring; two activation
    // slots, two weight slots per team (one is refilled while the team works from the other), more activation slots, the rest to the
    // weights.
    const int budget = RING_BUDGET - cfg->staging_bytes;
    int n_p = 1;
    if (plan && plan->stages > 0) {
        n_p = plan->stages;
        if (n_p > MAX_P) return false;
        // (one slot fewer where only the zero rows behind the blocks are too much)
        const int zeros = cfg->halo ? S / 32 * 1024 : 0;
        if (n_p > 1 && n_p * cfg->p_bytes + 2 * cfg->wstage_bytes > budget && n_p * (cfg->p_bytes - zeros) + 2 * cfg->wstage_bytes <= budget) --n_p;
    } else {
        auto fits = [&](int a, int w) { return a * cfg->p_bytes + w * cfg->wstage_bytes <= budget; };
        // (where a team gets less than a chunk from a slot, a third slot is worth more than its second weight slot)
        const int w = cfg->halo && taps < cfg->cycle * (32 / KC) ? cfg->cycle : 2 * cfg->cycle;
        if (fits(2, std::max(2, cfg->cycle))) n_p = 2;
        while (n_p < (cfg->halo ? 3 : MAX_P) && fits(n_p + 1, fits(n_p, w) ? w : std::max(2, cfg->cycle))) ++n_p;
    }
    int n_w = (budget - n_p * cfg->p_bytes) / cfg->wstage_bytes;
    if (n_w > MAX_W) n_w = MAX_W;
    // A plan's activation slots may leave room for two weight slots only: two teams then take the chunks in turn, the others idle.
    while (cfg->cycle > 2 && n_w < cfg->cycle) cfg->cycle /= 2;
    n_w -= n_w % cfg->cycle;
    if (n_w < 2) return false;
    cfg->n_p = n_p;
    cfg->n_w = n_w;
    if (cfg->alias_staging) {
        // one work item per CTA: the rings are idle when the epilogue runs, every channel block gets a box of its own
        const int ring_bytes = n_p * cfg->p_bytes + n_w * cfg->wstage_bytes;
        const int blocks = cfg->bn / 32;
        if (blocks >= 2 && ring_bytes >= 4 * blocks * BOX_BYTES) {
            cfg->boxes = blocks;   // at most 256 / 32 = MAX_BOXES
        } else if (ring_bytes < 4 * cfg->boxes * BOX_BYTES) {
            cfg->alias_staging = 0;
            cfg->staging_bytes = 4 * cfg->boxes * BOX_BYTES;
        }
    }
    return true;
}

template <class P>
nm_status_t launch(const ConvParams& p, const SelCfg& cfg, cudaStream_t st)
{
    ConvParams q = p;
    if (cfg.ksplit > 1) {
        q.y = p.splitk;
        q.pixels = static_cast<long long>(cfg.ksplit) * cfg.p_pad;   // rows of the store map
        q.bias = nullptr;
        q.residual = nullptr;
        q.relu = 0;
    }
    alignas(64) CUtensorMap tm_x, tm_y, tm_res;
    const bool ok_x = cfg.rows2d ? nmtm::encode_x_rows(p, cfg.prow, &tm_x) : nmtm::encode_x_im2col(p, BM, &tm_x);
    if (!ok_x || !nmtm::encode_y_tiled(q, &tm_y))
        return nmhost::fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 8)");
    tm_res = tm_y;
    if (q.residual && !nmtm::encode_y_tiled(q, &tm_res, 32, q.residual))
        return nmhost::fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 8)");
    q.pixels = p.pixels;
    size_t smem = 1024 + static_cast<size_t>(cfg.n_p) * cfg.p_bytes + static_cast<size_t>(cfg.n_w) * cfg.wstage_bytes +
                  cfg.staging_bytes;
    if (smem < NM_EXCLUSIVE_SMEM) smem = NM_EXCLUSIVE_SMEM;   // one CTA per SM: it owns all 512 TMEM columns
    const bool pairs = cfg.g % 2 == 0;
    const auto kernel = cfg.halo ? (pairs ? k_conv_select<P, 1, 2> : k_conv_select<P, 1, 1>) : (pairs ? k_conv_select<P, 0, 2> : k_conv_select<P, 0, 1>);
    cudaError_t e = nmhost::ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "cudaFuncSetAttribute (variant 8): %s", cudaGetErrorString(e));
    const long long grid = cfg.n_work < nmhost::sm_count() ? cfg.n_work : nmhost::sm_count();
    e = nmhost::launch_pdl(kernel, static_cast<unsigned>(grid), THREADS, smem, st, q, cfg, tm_x, tm_y, tm_res);
    nmhost::count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return nmhost::fail(NM_ERR_CUDA, "nm_conv2d launch (variant 8): %s", cudaGetErrorString(e));
    if (cfg.ksplit > 1) return nmhost::launch_splitk_reduce(p, cfg.ksplit, cfg.p_pad, st);
    return NM_OK;
}

}  // namespace

namespace nmhost {

bool select_layout_dims(const nm_weights* h, int* s, int* kc)
{
    return pattern_dims(h->n_keep, h->m_group, s, kc) && h->k % h->m_group == 0 && h->c_in % *s == 0 && h->tile_t % 16 == 0 &&
           h->c_out % h->tile_t == 0;
}

bool select_plan_ok(const ConvParams& p, const nm_plan_t* plan)
{
    SelCfg cfg;
    return make_cfg(p, plan, &cfg);
}

int select_ranges(const ConvParams& p, const nm_plan_t* plan)
{
    SelCfg cfg;
    return make_cfg(p, plan, &cfg) ? cfg.ksplit : 0;
}

size_t select_splitk_bytes(const ConvParams& p, int splits)
{
    const size_t p_pad = static_cast<size_t>((p.pixels + BM - 1) / BM) * BM;
    return static_cast<size_t>(splits) * p_pad * p.c_out * sizeof(float);
}

nm_status_t launch_conv_select(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st)
{
    SelCfg cfg;
    if (!make_cfg(p, plan, &cfg))
        return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: the select kernel does not take this layer / plan%s",
                    plan && plan->ksplit > 1 ? " (a split plan needs scratch: nm_weights_reserve)" : "");
    switch (p.sel_kc * (p.sel_s / 32)) {
        case 8: return launch<Pattern<8, 32>>(p, cfg, st);
        case 16: return p.sel_s == 32 ? launch<Pattern<16, 32>>(p, cfg, st) : launch<Pattern<8, 64>>(p, cfg, st);
        case 24: return launch<Pattern<24, 32>>(p, cfg, st);
    }
    return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: N:M pattern not covered by the select kernel");
}

}  // namespace nmhost
