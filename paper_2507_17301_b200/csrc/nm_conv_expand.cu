// Variant 4: expanded-operand kernel — persistent implicit GEMM that feeds the tensor core the
// DENSE activation slab straight from shared memory and lets zero weights stand for the pruned
// columns.
//
// Nothing is compacted: the slab [128 pixels x 32 source columns] that TMA's im2col mode lays
// down in the 128-byte-swizzled K-major layout IS the A operand, and the B operand is the pruned
// weight matrix re-expanded to its dense [channels x K] shape (TF32, zeros in the pruned
// columns, built once per handle).  The tensor core therefore spends M/N times the kept FLOPs,
// but no thread ever touches an activation.  It moves the same HBM bytes as the gathering
// kernels (with N:M groups along the channel axis every 16-byte vector holds survivors, so a
// gather cannot skip input bytes either), which makes it the right choice wherever the layer is
// bound by HBM and the tensor pipe has slack; the auto-tuner decides per layer by measurement.
// The pruning tile width plays no role here, so any tile_t is accepted.
//
//   activation producer   TMA load of the slab per stage: im2col mode, or plain 2-D rows for pointwise layers of stride 1;
//   (1 thread)
//   weight producer       one contiguous bulk copy of the weight block per stage (stored pre-swizzled, so it costs no per-row
//   (1 thread)            TMA requests); a weight slice of at most 128 KB is instead fetched once and stays resident
//                         (the grid is then a multiple of the slice count, so a CTA keeps its slice)
//   MMA issuer (1 thread) four 128 x BN x 8 TF32 tcgen05.mma (SS) per stage into one of two
//                         accumulator buffers in tensor memory
//   epilogue (8 warps)    TMEM -> registers, + bias, ReLU, swizzled staging, TMA store to NHWC;
//                         overlaps the next work item's main loop
// Work items (up to 128 pixels x BN channels) are walked in a static persistent schedule; every wait is
// bounded and reports through the handle's status word.
// Pixels per item: as few as keep the number of rounds (items / CTAs, rounded up) what it is with 128.  A layer whose items
// fill 1.32 rounds of the SMs takes two rounds either way, and with 128-pixel items it spends the second one with
// a third of the SMs pulling in all of the bytes; equal items of 88 pixels spread them over all SMs.
//
// Balanced mode (plan.split = -1), for layers with fewer work items than would keep every SM busy:
// the (item, stage) pairs of the whole layer are laid end to end and cut into one contiguous,
// equally long range per CTA, so an item may be shared by two or more CTAs.  A CTA whose range
// begins inside an item handles that part FIRST, stores the raw partial accumulator to its own
// slot of the handle's scratch and raises a per-warp flag; the CTA whose range holds the item's
// first stage handles it next, before its whole items, waits (bounded) for the flags of the others, adds their partial sums
// to its accumulator, lowers the flags again (every flag has exactly one reader, so the scratch is
// back in its cleared state when the launch ends and a recorded launch can be replayed) and runs
// the normal epilogue.  Ranges are handed out from the end of the
// layer to CTA 0 upwards, so a CTA only ever waits for CTAs with a lower index, whose first action
// is the store it waits for.
#include <algorithm>

#include "nm_internal.h"
#include "nm_ptx.cuh"
#include "nm_tmap.cuh"

namespace {

using namespace nmk;

constexpr int BM = 128;
constexpr int NSTAGE_MAX = 14;
constexpr int WRES_MAX = 128 * 1024;            // largest weight slice kept resident
constexpr int THREADS = 384;                   // 4 service warps + 8 epilogue warps
constexpr int BOX_BYTES = 4096;                // one 32-pixel x 32-channel output box
constexpr int BOXES_MAX = 3;                   // staging boxes per epilogue warp

struct ExpandCfg {
    int bn;           // output channels per work item
    int n_slices;
    int stages;       // activation ring: slots
    int w_stages;     // weight ring: slots, at most `stages` (0 with resident weights)
    int b_bytes;      // bytes of a weight block (bn rows of 128 bytes)
    int a_bytes;      // bytes a 32-column block of activations takes in a slot (rows of 128 bytes, rounded up to 1 KB)
    int w_res;        // 1: this CTA's weight slice stays resident in shared memory (it is loaded once)
    int wres_bytes;   // bytes of the resident slice: all 32-column blocks of bn rows
    int n_sub;        // pipeline stages one work item reduces over: (K / 32) / ksplit / kblk
    int kblk;         // 32-column blocks per stage (1 or 2): one barrier round trip then covers kblk * 4 MMAs
    int n_iss;        // MMA issuer threads (1 or 2): two take alternate pipeline stages of an item, each into an accumulator of its own
    int n_acc;        // accumulator buffers (of n_iss accumulators each) in tensor memory: 2 when they fit, else 1
    int rows;         // pixels per work item
    int flat;         // 1: activations as 2-D rows (pointwise, stride 1), 0: im2col
    int ksplit;       // K splits (1 = none): a work item covers one of them and stores raw partial sums
    int p_pad;        // pixel blocks * 128: rows of one split in the partial-sum scratch
    int boxes;        // output staging boxes per epilogue warp: 2 for short reductions, 1 when the ring needs the room;
                      // with a shortcut input, which is loaded into them ahead of time, 3 (2 when the ring needs the room)
    int last_tile;    // >= 0: pixel tiles are taken from this one down (see make_cfg), -1: from the first up
    int sl_shift;     // log2 of n_slices, -1 where it is no power of two
    int balanced;     // 1: contiguous (item, stage) ranges per CTA, partial sums through per-CTA scratch slots
    long long n_work;
};

__device__ __forceinline__ bool aborted(volatile int* flag) { return *flag != 0; }

// Wait of a producer for a ring slot.  The abort flag is looked at only here, i.e. when the slot was not free at once: a
// pipeline whose other end has given up comes to a halt, so nobody runs past this point for long.
__device__ __forceinline__ bool wait_stage(uint32_t bar, uint32_t parity, volatile int* flag, int site)
{
    for (uint32_t i = 0; i < kWaitPolls; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 15u) == 0u && *flag != 0) return false;
    }
    *flag = site;
    return false;
}
// After an abort: loads already issued still target this CTA's shared memory, let them land (bounded).
__device__ __forceinline__ void drain_ring(RingPos rp, int issued, int n, uint64_t* full)
{
    for (int back = 0; back < n && back < issued; ++back) {
        if (rp.s == 0) { rp.s = n; rp.parity ^= 1u; }
        --rp.s;
        (void)mbar_wait_polls(smem_u32(&full[rp.s]), rp.parity, 1u << 16);
    }
}

// One piece of work of a CTA: stages [sb, se) of work item `work`.
struct Seg {
    uint32_t work;
    int sb, se;
};
struct ItemPos {
    uint32_t tile, slice, ks;   // pixel tile, channel slice, range of the reduction axis
};
__device__ __forceinline__ ItemPos item_of(uint32_t work, const ExpandCfg& cfg)
{
    ItemPos it = {work, 0u, 0u};
    if (cfg.sl_shift > 0) {
        it.tile = work >> cfg.sl_shift;
        it.slice = work - (it.tile << cfg.sl_shift);
    } else if (cfg.sl_shift < 0) {
        it.tile = work / static_cast<uint32_t>(cfg.n_slices);
        it.slice = work - it.tile * static_cast<uint32_t>(cfg.n_slices);
    }
    if (cfg.ksplit > 1) {
        const uint32_t t = it.tile / static_cast<uint32_t>(cfg.ksplit);
        it.ks = it.tile - t * static_cast<uint32_t>(cfg.ksplit);
        it.tile = t;
    }
    if (cfg.last_tile >= 0) it.tile = static_cast<uint32_t>(cfg.last_tile) - it.tile;
    return it;
}
// Walks a CTA's pieces: whole items `first, first + stride, ...` in the static schedule, or the
// contiguous range of (item, stage) units of balanced mode: the rest of an item begun elsewhere first, then the part of
// the item that is continued elsewhere, then the whole items.  The part that waits for other CTAs' sums is so finished while
// the main loop of a whole item runs, instead of after the last of them.
template <bool BAL>
struct SegIter {
    uint32_t cur, end, stride;   // balanced: stride counts the phases done
    int stages;
    __device__ __forceinline__ bool next(Seg& g)
    {
        if (!BAL) {
            if (cur >= end) return false;
            g.work = cur; g.sb = 0; g.se = stages;
            cur += stride;
            return true;
        }
        const uint32_t n = static_cast<uint32_t>(stages);
        if (stride == 0) {
            stride = 1;
            g.work = cur / n;
            g.sb = static_cast<int>(cur - g.work * n);
            if (g.sb > 0 && cur < end) {
                const uint32_t room = n - static_cast<uint32_t>(g.sb), len = end - cur < room ? end - cur : room;
                g.se = g.sb + static_cast<int>(len);
                cur += len;
                return true;
            }
        }
        if (stride == 1) {
            stride = 2;
            g.work = end / n;
            const uint32_t part = end - g.work * n;
            if (part > 0 && end - part >= cur) {
                g.sb = 0;
                g.se = static_cast<int>(part);
                end -= part;
                return true;
            }
        }
        if (cur >= end) return false;
        g.work = cur / n; g.sb = 0; g.se = stages;
        cur += n;
        return true;
    }
};
// First (item, stage) unit of the range at position j of `n` equal ranges over `units`.
__device__ __forceinline__ uint32_t range_begin(uint32_t j, uint32_t n, uint32_t units)
{
    return static_cast<uint32_t>(static_cast<unsigned long long>(j) * units / n);
}
template <bool BAL>
__device__ __forceinline__ SegIter<BAL> make_iter(const ExpandCfg& cfg)
{
    SegIter<BAL> it;
    it.stages = cfg.n_sub;
    if (!BAL) {
        it.cur = blockIdx.x; it.end = static_cast<uint32_t>(cfg.n_work); it.stride = gridDim.x;
    } else {
        // ranges are handed out from the end of the layer: CTA b takes position gridDim.x - 1 - b
        const uint32_t units = static_cast<uint32_t>(cfg.n_work) * static_cast<uint32_t>(cfg.n_sub);
        const uint32_t j = gridDim.x - 1u - blockIdx.x;
        it.cur = range_begin(j, gridDim.x, units);
        it.end = range_begin(j + 1u, gridDim.x, units);
        it.stride = 0;
    }
    return it;
}
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* ptr)
{
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ptr) : "memory");
    return v;
}
__device__ __forceinline__ void st_release_gpu(uint32_t* ptr, uint32_t v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(ptr), "r"(v) : "memory");
}

// KBLK: 32-column blocks per pipeline stage; BAL: balanced mode.  Compile-time, so that the lone producer and
// issuer threads of the common configuration (1, false) run exactly the instructions they need.
template <int KBLK, bool BAL>
__global__ void __launch_bounds__(THREADS, 1)
k_conv_expand(const ConvParams p, const ExpandCfg cfg, const __grid_constant__ CUtensorMap tm_x,
              const __grid_constant__ CUtensorMap tm_y, const __grid_constant__ CUtensorMap tm_tail,
              const __grid_constant__ CUtensorMap tm_res)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_full[NSTAGE_MAX], s_free[NSTAGE_MAX], s_accfull[2], s_accfree[2], s_wres, s_res[8][BOXES_MAX];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ __align__(16) float s_bias[8][32];   // bias of the block an epilogue warp works on

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    const int NS = cfg.stages, n_sub = cfg.n_sub;
    const uint32_t wres = (smem_u32(smem_raw) + 1023u) & ~1023u;   // resident weight slice (may be empty)
    const uint32_t ring = wres + cfg.wres_bytes;
    const uint32_t a_slot = static_cast<uint32_t>(KBLK * cfg.a_bytes), w_slot = static_cast<uint32_t>(KBLK * cfg.b_bytes);
    // activation ring, weight ring, output staging; an MMA reads 128 rows from an activation slot's start, rows past the
    // item's come from whatever lies behind and end in accumulator rows nobody reads
    const uint32_t w_ring = ring + NS * a_slot;
    const uint32_t staging = w_ring + cfg.w_stages * w_slot;
    volatile int* abort_flag = &s_abort;

    if (warp == 2) tmem_alloc(smem_u32(&s_tmem), 512);
    if (tid == 0) {
        for (int i = 0; i < NSTAGE_MAX; ++i) {
            mbar_init(smem_u32(&s_full[i]), cfg.w_res ? 1 : 2);   // the producers' expect-tx arrivals
            mbar_init(smem_u32(&s_free[i]), 1);   // the commit of the issuer that read the stage
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(smem_u32(&s_accfull[i]), cfg.n_iss);   // MMA commits
            mbar_init(smem_u32(&s_accfree[i]), 8);   // epilogue warps
        }
        mbar_init(smem_u32(&s_wres), 1);
        for (int i = 0; i < 8 * BOXES_MAX; ++i) mbar_init(smem_u32(&s_res[0][0] + i), 1);   // a shortcut box has landed
        mbar_fence_init();
        s_abort = 0;
        tma_prefetch_desc(&tm_x);
        tma_prefetch_desc(&tm_y);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    pdl_launch_dependents();   // the next kernel may start its own set-up as SMs become free
    if (warp != 2) pdl_wait(); // from here on global memory written by the previous kernel is read (weights are no kernel's output)

    if (warp == 0) {
        // =========================== activation producer ===========================
        if (elect_one()) {
            int issued = 0;
            const int hw = p.ho * p.wo;
            const uint32_t tx = static_cast<uint32_t>(KBLK) * static_cast<uint32_t>(cfg.rows) * 128u;
            const int n_blk32 = n_sub * KBLK;   // 32-column blocks per work item
            RingPos rp;
            SegIter<BAL> it = make_iter<BAL>(cfg);
            Seg seg;
            bool ok = true, free_now = true;   // free_now: the slot's release was seen while the stage before it was issued
            while (ok && it.next(seg)) {
                const ItemPos item = item_of(seg.work, cfg);
                const uint32_t ks = item.ks;
                const int pix0 = static_cast<int>(item.tile) * cfg.rows;
                int n0 = 0, w0 = 0, h0 = 0;
                if (!cfg.flat) {
                    n0 = static_cast<int>(static_cast<uint32_t>(pix0) / static_cast<uint32_t>(hw));
                    const int rem = pix0 - n0 * hw;
                    const int oh0 = rem / p.wo, ow0 = rem - oh0 * p.wo;
                    w0 = ow0 * p.stride_w - p.pad_w;
                    h0 = oh0 * p.stride_h - p.pad_h;
                }
                // first 32-column block of this item's share of the reduction axis
                const int c0 = static_cast<int>(ks) * n_blk32 + seg.sb * KBLK;
                int ch = 0, tw = 0, off_w = 0, off_h = 0;
                if (c0 != 0) {
                    const int tap0 = (c0 * 32) / p.c_in, th = tap0 / p.kw;
                    ch = c0 * 32 - tap0 * p.c_in;
                    tw = tap0 - th * p.kw;
                    off_w = tw * p.dil_w;
                    off_h = th * p.dil_h;
                }
                for (int c = seg.sb; c < seg.se; ++c) {
                    if (!free_now && !wait_stage(smem_u32(&s_free[rp.s]), rp.parity ^ 1u, abort_flag, 2)) { ok = false; break; }
                    uint32_t a_smem = ring + rp.s * a_slot;
                    const uint32_t bar = smem_u32(&s_full[rp.s]);
                    mbar_arrive_expect_tx(bar, tx);
                    rp.advance(NS);
                    free_now = !rp.wrapped || mbar_test_wait(smem_u32(&s_free[rp.s]), rp.parity ^ 1u);
#pragma unroll
                    for (int j = 0; j < KBLK; ++j) {
                        if (cfg.flat)
                            tma_load_2d(a_smem, &tm_x, bar, ch, pix0);
                        else
                            tma_load_im2col_4d(a_smem, &tm_x, bar, ch, w0, h0, n0, static_cast<uint16_t>(off_w),
                                               static_cast<uint16_t>(off_h));
                        a_smem += cfg.a_bytes;
                        ch += 32;
                        if (ch >= p.c_in) {
                            ch = 0;
                            off_w += p.dil_w;
                            if (++tw == p.kw) { tw = 0; off_w = 0; off_h += p.dil_h; }
                        }
                    }
                    ++issued;
                }
            }
            if (aborted(abort_flag)) drain_ring(rp, issued, NS, s_full);
        }
    } else if (warp == 2) {
        // =========================== weight producer ===========================
        if (elect_one()) {
            const int n_blk32 = n_sub * KBLK;
            const uint32_t w_bytes = static_cast<uint32_t>(cfg.bn) * 128u;
            const size_t w_step = static_cast<size_t>(p.wx_rows) * 32;   // floats between two 32-column blocks
            if (cfg.w_res) {
                // the grid is a multiple of the slice count, so every work item of this CTA has the
                // same channel slice: its weights are fetched once
                const int slice = static_cast<int>(blockIdx.x % static_cast<uint32_t>(cfg.n_slices));
                mbar_arrive_expect_tx(smem_u32(&s_wres), static_cast<uint32_t>(n_blk32) * w_bytes);
                for (int c = 0; c < n_blk32; ++c)
                    bulk_load_1d(wres + c * cfg.b_bytes, p.wx + static_cast<size_t>(c) * w_step + static_cast<size_t>(slice) * cfg.bn * 32,
                                 w_bytes, smem_u32(&s_wres));
            } else {
                // Stage t joins the full barrier of its activation slot, t modulo the activation ring; its weight slot, t modulo
                // the (shorter) weight ring, is free once the MMAs of stage t - w_stages are done, which is what the free
                // barrier of THAT stage's activation slot says.
                int issued = 0;
                RingPos rp, rf;      // full barrier of this stage, free barrier of the stage that used the weight slot before
                int ws = 0;
                bool wrapped = false;
                SegIter<BAL> it = make_iter<BAL>(cfg);
                Seg seg;
                bool ok = true, free_now = true;
                while (ok && it.next(seg)) {
                    const ItemPos item = item_of(seg.work, cfg);
                    const int c0 = static_cast<int>(item.ks) * n_blk32 + seg.sb * KBLK;
                    const float* wsrc = p.wx + static_cast<size_t>(item.slice) * cfg.bn * 32 + static_cast<size_t>(c0) * w_step;
                    for (int c = seg.sb; c < seg.se; ++c) {
                        if (!free_now && !wait_stage(smem_u32(&s_free[rf.s]), rf.parity, abort_flag, 9)) { ok = false; break; }
                        if (wrapped) rf.advance(NS);
                        uint32_t b_smem = w_ring + ws * w_slot;
                        const uint32_t bar = smem_u32(&s_full[rp.s]);
                        mbar_arrive_expect_tx(bar, static_cast<uint32_t>(KBLK) * w_bytes);
                        rp.advance(NS);
                        if (++ws == cfg.w_stages) { ws = 0; wrapped = true; }
                        free_now = !wrapped || mbar_test_wait(smem_u32(&s_free[rf.s]), rf.parity);
#pragma unroll
                        for (int j = 0; j < KBLK; ++j) {
                            bulk_load_1d(b_smem, wsrc, w_bytes, bar);
                            b_smem += cfg.b_bytes;
                            wsrc += w_step;
                        }
                        ++issued;
                    }
                }
                if (aborted(abort_flag)) drain_ring(rp, issued, NS, s_full);
            }
            if (cfg.w_res && aborted(abort_flag)) (void)mbar_wait(smem_u32(&s_wres), 0);
        }
    } else if (warp == 1 || warp == 3) {
        // =========================== MMA issuers ===========================
        // A thread issues a tcgen05.mma about every 124 cycles whatever its width, and a barrier test and a commit per
        // stage on top of that, while the tensor core completes a 128 x 256 x 8 MMA in 128 cycles and narrower ones
        // sooner: one thread cannot keep it busy.  A plan may therefore have two issuer threads that take ALTERNATE
        // stages of a work item, each accumulating into columns of its own (the epilogue adds the two): the reduction
        // axis is split, not the channels, so both issue full-width MMAs.  A ring slot is released by the one commit of
        // the thread that read it.  Ownership goes by SLOT (even slots the first thread, odd slots the second; the ring
        // then has an even number of slots): a wait by phase parity is only right for a waiter that has seen every
        // earlier use of the slot, and with ownership by position inside the item a thread would skip uses of a slot
        // at the seams between items (found as a fault on the GPU, reproduced and fixed in a CPU model of the protocol).
        const int iss = warp >> 1;
        if (iss < cfg.n_iss && elect_one()) {
            const uint32_t idesc = umma_idesc_tf32(BM, cfg.bn);
            const bool shared_k = cfg.n_iss == 2;
            if (cfg.w_res && !mbar_wait(smem_u32(&s_wres), 0)) *abort_flag = 9;
            RingPos rp;
            int ws = 0;
            uint32_t ab = 0, acc_par = 0;   // accumulator buffer of this item, parity of its current use
            bool acc_wrapped = false;
            SegIter<BAL> it = make_iter<BAL>(cfg);
            Seg seg;
            while (!aborted(abort_flag) && it.next(seg)) {
                if (acc_wrapped && !mbar_wait_lone(smem_u32(&s_accfree[ab]), acc_par ^ 1u)) {
                    *abort_flag = 5;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + (ab * cfg.n_iss + iss) * cfg.bn;
                uint32_t started = 0;   // 0 until this thread's first MMA of the item, which overwrites the accumulator
                for (int c = seg.sb; c < seg.se; ++c) {
                    if (shared_k && (rp.s & 1) != iss) {   // the other thread's slot
                        rp.advance(NS);
                        if (++ws == cfg.w_stages) ws = 0;
                        continue;
                    }
                    if (!mbar_wait_lone(smem_u32(&s_full[rp.s]), rp.parity)) { *abort_flag = 6; break; }
                    tc_fence_after();
                    uint64_t adesc = umma_desc_k_sw128(ring + rp.s * a_slot, 1024);
                    uint64_t bdesc = umma_desc_k_sw128(cfg.w_res ? wres + c * KBLK * cfg.b_bytes : w_ring + ws * w_slot, 1024);
#pragma unroll
                    for (int j = 0; j < KBLK; ++j) {
#pragma unroll
                        for (int kq = 0; kq < 4; ++kq)
                            umma_tf32_ss(acc, adesc + 2 * kq, bdesc + 2 * kq, idesc, (j > 0 || kq > 0) ? 1u : started);
                        if (j + 1 < KBLK) {
                            adesc += static_cast<uint32_t>(cfg.a_bytes) >> 4;   // next 32-column block (start address field, 16-byte units)
                            bdesc += static_cast<uint32_t>(cfg.b_bytes) >> 4;
                        }
                    }
                    started = 1u;
                    umma_commit(smem_u32(&s_free[rp.s]));
                    rp.advance(NS);
                    if (++ws == cfg.w_stages) ws = 0;
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
    } else if (warp >= 4) {
        // =========================== epilogue ===========================
        const int q = warp & 3;            // TMEM lane quadrant
        // Which channel blocks of 32: blk = 2 * i + half; with an odd number of blocks the two warps of a quadrant change places from item to
        // item, so that both have the same work (one block: every other item).  32 -> 16 at 112x112, batch 32: 22.4 -> 17.3 us,
        // 16 -> 96 37.0 -> 32.1 us.
        const int half = (warp - 4) >> 2;
        const uint32_t lane_addr = static_cast<uint32_t>(q * 32) << 16;
        const uint32_t my_staging = staging + (warp - 4) * cfg.boxes * BOX_BYTES;
        const uint32_t rx = static_cast<uint32_t>(lane & 7);
        const int n_blk = cfg.bn / 32;
        auto first_block = [&](uint32_t i) { return BAL || (n_blk & 1) == 0 ? half : half ^ static_cast<int>(i & 1u); };
        const int box_rows = cfg.rows - q * 32 < 0 ? 0 : cfg.rows - q * 32 < 32 ? cfg.rows - q * 32 : 32;   // pixels of this warp's boxes
        uint32_t ti = 0;
        uint32_t stage_count = 0;   // stages of all earlier pieces of this CTA
        // balanced mode: this CTA's partial-sum slot (128 rows x bn) and its warps' flags, in the handle's scratch
        const uint32_t units = static_cast<uint32_t>(cfg.n_work) * static_cast<uint32_t>(cfg.n_sub);
        const size_t slot_floats = static_cast<size_t>(BM) * cfg.bn;
        // scratch layout: eight flag words per CTA first, then the slots
        uint32_t* const flags = reinterpret_cast<uint32_t*>(p.splitk);
        float* const slots = p.splitk + static_cast<size_t>(gridDim.x) * 8;
        const int my_row = q * 32 + lane;
        SegIter<BAL> it = make_iter<BAL>(cfg);
        Seg seg;
        // Shortcut input: the box of a block is loaded into the block's staging box, cfg.boxes - 1 blocks ahead (the walk
        // `nit` runs ahead of `it` by that much), added there and stored from there.  (Held in registers a block
        // ahead it cost two passes over the box and left too little in flight: 64 -> 256 at 56x56, batch 64, took 101-106 us,
        // now 82-87 with the bytes' own time at 70; 256 -> 1024 at 14x14, batch 128, 58 -> 45 us.)
        const bool res = p.residual != nullptr;
        const uint32_t n_box = static_cast<uint32_t>(cfg.boxes);
        uint32_t bx = 0, bpar = 0;      // this block's staging box, parity of its current use
        uint32_t nbx = 0, asked = 0, taken = 0;
        SegIter<BAL> nit = make_iter<BAL>(cfg);
        Seg nseg;
        int nblk = n_blk, no0 = 0, npix = 0;
        uint32_t nti = 0;
        auto request = [&]() {
            while (nblk >= n_blk) {
                if (!nit.next(nseg)) return;
                const int first = first_block(nti++);
                const ItemPos item = item_of(nseg.work, cfg);
                no0 = static_cast<int>(item.slice) * cfg.bn;
                npix = static_cast<int>(item.tile) * cfg.rows + q * 32;
                if (box_rows > 0 && npix < p.pixels && !(BAL && nseg.sb > 0)) nblk = first;
            }
            if (elect_one()) {
                const uint32_t bar = smem_u32(&s_res[warp - 4][nbx]);
                mbar_arrive_expect_tx(bar, BOX_BYTES);
                tma_load_2d(my_staging + nbx * BOX_BYTES, &tm_res, bar, no0 + nblk * 32, npix);
            }
            nblk += 2;
            nbx = nbx + 1 == n_box ? 0 : nbx + 1;
            ++asked;
        };
        if (res)
            for (uint32_t k = 1; k < n_box; ++k) request();
        for (; it.next(seg); ++ti) {
            const uint32_t work = seg.work;
            const bool publish = BAL && seg.sb > 0;                   // a later part of an item: store raw sums
            const bool finish = BAL && seg.sb == 0 && seg.se < n_sub;  // the first part: add the others' sums
            const ItemPos item = item_of(work, cfg);
            const int pix0 = static_cast<int>(item.tile) * cfg.rows + q * 32;   // first pixel of this warp's boxes
            const int o0 = static_cast<int>(item.slice) * cfg.bn;
            const bool live = box_rows > 0 && pix0 < p.pixels;
            const int ab = cfg.n_acc == 2 ? static_cast<int>(ti & 1u) : 0;
            // two issuers: stages went to them by ring slot, i.e. by the parity of the running stage count; a piece of
            // one stage is in the accumulator of that stage's owner, a longer one in both
            const uint32_t piece_first = stage_count;
            stage_count += static_cast<uint32_t>(seg.se - seg.sb);
            const bool two_acc = cfg.n_iss == 2 && seg.se - seg.sb >= 2;
            const uint32_t acc_first = (cfg.n_iss == 2 && seg.se - seg.sb == 1) ? (piece_first & 1u) : 0u;
            // positions (of the equal ranges) that hold the rest of this item: first_pos + 1 .. last_pos.  Their
            // partial sums were stored long ago (they are those CTAs' first piece of work), so the flags are
            // checked and the first counterpart's sums of this warp's first block are requested BEFORE the wait for this CTA's own accumulator.
            uint32_t first_pos = 0, last_pos = 0;
            bool ahead = false;
            float4 rv[8];
            if (finish) {
                first_pos = gridDim.x - 1u - blockIdx.x;
                const uint32_t u_last = (work + 1u) * static_cast<uint32_t>(n_sub) - 1u;
                last_pos = static_cast<uint32_t>(static_cast<unsigned long long>(u_last) * gridDim.x / units);
                while (last_pos + 1u < gridDim.x && range_begin(last_pos + 1u, gridDim.x, units) <= u_last) ++last_pos;
                while (last_pos > first_pos && range_begin(last_pos, gridDim.x, units) > u_last) --last_pos;
                // each of this warp's counterparts has stored its rows and raised its flag (bounded wait)
                for (uint32_t pos = first_pos + 1u; pos <= last_pos; ++pos) {
                    const uint32_t* f = flags + (gridDim.x - 1u - pos) * 8u + (warp - 4);
                    bool seen = false;
                    for (uint32_t poll = 0; poll < kWaitPolls && !seen; ++poll) seen = ld_acquire_gpu(f) == 1u;
                    if (!seen) *abort_flag = 10;
                }
                if (half < n_blk && !aborted(abort_flag)) {
                    const float4* src = reinterpret_cast<const float4*>(slots + slot_floats * (gridDim.x - 2u - first_pos)) +
                                        static_cast<size_t>(half) * 8 * BM + my_row;
#pragma unroll
                    for (int qq = 0; qq < 8; ++qq) rv[qq] = __ldcg(src + qq * BM);
                    ahead = true;
                }
            }
            // Bias of this warp's blocks, a channel per lane, fetched while the main loop runs: a block's bias is a line of its own that
            // the first-level cache does not hold yet, and loaded at its use it held every block up.  With that and the loads of a block
            // ahead of its first store a block takes 0.48 us instead of 0.68 (a 128 x 256 item 2.1 instead of 2.9): 1024 -> 256 at 14x14, batch
            // 64, 15.5 -> 14.6 us, 64 -> 256 at 56x56 45.4 -> 43.1, 24 -> 144 at 56x56, batch 32, 14.7 -> 12.3, 64 -> 384 at 14x14 5.1 -> 4.95.
            const int first = first_block(ti);
            float bias_of[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) bias_of[i] = first + 2 * i < n_blk ? bias_lane_load(p.bias, o0 + (first + 2 * i) * 32, p.c_out, lane) : 0.f;
            const bool ok = aborted(abort_flag) || mbar_wait_lone(smem_u32(&s_accfull[ab]), (cfg.n_acc == 2 ? (ti >> 1) : ti) & 1u);
            if (!__all_sync(0xFFFFFFFFu, ok)) *abort_flag = 8;
            if (__any_sync(0xFFFFFFFFu, aborted(abort_flag))) break;
            tc_fence_after();
            if (!BAL && !live) {   // an item of fewer pixels: this warp's quadrant of the accumulator holds nothing
                if (lane == 0) mbar_arrive(smem_u32(&s_accfree[ab]));
                continue;
            }
            // The accumulator columns of a block are read while the block before it is finished (not in balanced mode, which
            // has partial sums in those registers).
            const uint32_t acc_addr = tmem + lane_addr + (ab * cfg.n_iss + acc_first) * cfg.bn;
            uint32_t vn[32];
            if (!BAL && first < n_blk) tmem_ld32(acc_addr + first * 32, vn);
            for (int blk = first; blk < n_blk; blk += 2) {
                s_bias[warp - 4][lane] = bias_of[0];   // (the block before it has been read: see its __syncwarp)
                bias_of[0] = bias_of[1]; bias_of[1] = bias_of[2]; bias_of[2] = bias_of[3];
                __syncwarp();
                float4 bias[8];
#pragma unroll
                for (int qq = 0; qq < 8; ++qq) bias[qq] = reinterpret_cast<const float4*>(s_bias[warp - 4])[qq];
                uint32_t v[32];
                if (BAL) tmem_ld32(acc_addr + blk * 32, vn);
                if (two_acc) {
                    uint32_t v2[32];
                    tmem_ld32(tmem + lane_addr + (ab * cfg.n_iss + 1) * cfg.bn + blk * 32, v2);
                    tmem_ld_wait(v2);
                    tmem_ld_wait(vn);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(vn[e]) + __uint_as_float(v2[e]));
                } else {
                    tmem_ld_wait(vn);
#pragma unroll
                    for (int e = 0; e < 32; ++e) v[e] = vn[e];
                }
                if (!BAL && blk + 2 < n_blk) tmem_ld32(acc_addr + (blk + 2) * 32, vn);
                if (blk + 2 >= n_blk) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&s_accfree[ab]));
                }
                if (publish) {
                    // raw partial sums of this thread's row; the slot is laid out [channel quad][row], so the 32
                    // lanes of a warp (32 consecutive rows) write 512 contiguous bytes per instruction
                    float4* dst = reinterpret_cast<float4*>(slots + slot_floats * blockIdx.x) +
                                  static_cast<size_t>(blk) * 8 * BM + my_row;
#pragma unroll
                    for (int qq = 0; qq < 8; ++qq)
                        __stcg(dst + qq * BM, make_float4(__uint_as_float(v[qq * 4 + 0]), __uint_as_float(v[qq * 4 + 1]),
                                                     __uint_as_float(v[qq * 4 + 2]), __uint_as_float(v[qq * 4 + 3])));
                    continue;
                }
                if (finish) {
                    uint32_t pos_from = first_pos + 1u;
                    if (ahead) {
#pragma unroll
                        for (int qq = 0; qq < 8; ++qq) {
                            v[qq * 4 + 0] = __float_as_uint(__uint_as_float(v[qq * 4 + 0]) + rv[qq].x);
                            v[qq * 4 + 1] = __float_as_uint(__uint_as_float(v[qq * 4 + 1]) + rv[qq].y);
                            v[qq * 4 + 2] = __float_as_uint(__uint_as_float(v[qq * 4 + 2]) + rv[qq].z);
                            v[qq * 4 + 3] = __float_as_uint(__uint_as_float(v[qq * 4 + 3]) + rv[qq].w);
                        }
                        if (blk + 2 < n_blk) {   // a block ahead
                            const float4* nxt = reinterpret_cast<const float4*>(slots + slot_floats * (gridDim.x - 2u - first_pos)) +
                                                static_cast<size_t>(blk + 2) * 8 * BM + my_row;
#pragma unroll
                            for (int qq = 0; qq < 8; ++qq) rv[qq] = __ldcg(nxt + qq * BM);
                        }
                        ++pos_from;
                    }
                    for (uint32_t pos = pos_from; pos <= last_pos; ++pos) {
                        const float4* src = reinterpret_cast<const float4*>(slots + slot_floats * (gridDim.x - 1u - pos)) +
                                            static_cast<size_t>(blk) * 8 * BM + my_row;
                        float4 t4[8];
#pragma unroll
                        for (int qq = 0; qq < 8; ++qq) t4[qq] = __ldcg(src + qq * BM);
#pragma unroll
                        for (int qq = 0; qq < 8; ++qq) {
                            const float4 t = t4[qq];
                            v[qq * 4 + 0] = __float_as_uint(__uint_as_float(v[qq * 4 + 0]) + t.x);
                            v[qq * 4 + 1] = __float_as_uint(__uint_as_float(v[qq * 4 + 1]) + t.y);
                            v[qq * 4 + 2] = __float_as_uint(__uint_as_float(v[qq * 4 + 2]) + t.z);
                            v[qq * 4 + 3] = __float_as_uint(__uint_as_float(v[qq * 4 + 3]) + t.w);
                        }
                    }
                }
                if (BAL && !live) continue;
                const uint32_t box = my_staging + bx * BOX_BYTES;
                if (res) {
                    // the store of the block before this one must have read its box, the next one to be loaded
                    if (elect_one()) tma_store_wait_read_n<0>();
                    __syncwarp();
                    request();
                    const bool landed = mbar_wait_lone(smem_u32(&s_res[warp - 4][bx]), bpar);
                    if (!__all_sync(0xFFFFFFFFu, landed)) *abort_flag = 11;
                    ++taken;
                } else {
                    // the store that last read this box must be done with it
                    if (elect_one()) {
                        if (n_box >= 2) tma_store_wait_read_n<1>();
                        else tma_store_wait_read_n<0>();
                    }
                    __syncwarp();
                }
                const uint32_t stage_row = box + lane * 128;
                // Sum, then bias, then shortcut, as in the split-K form's second pass: a plan's schedule does not show in the order of the
                // additions.  (All loads before the first store: the stores are ordered statements, which no later load is moved ahead of.)
                float4 o8[8];
#pragma unroll
                for (int qq = 0; qq < 8; ++qq) {
                    o8[qq] = make_float4(__uint_as_float(v[qq * 4 + 0]), __uint_as_float(v[qq * 4 + 1]), __uint_as_float(v[qq * 4 + 2]),
                                         __uint_as_float(v[qq * 4 + 3]));
                    nm_add4(o8[qq], bias[qq]);
                }
                if (res) {
#pragma unroll
                    for (int qq = 0; qq < 8; ++qq) {
                        float4 x;
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x.x), "=f"(x.y), "=f"(x.z), "=f"(x.w) : "r"(stage_row + ((qq ^ rx) << 4)));
                        nm_add4(o8[qq], x);
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
                    tma_store_2d(box_rows == 32 ? &tm_y : &tm_tail, box, o0 + blk * 32, static_cast<int>(item.ks) * cfg.p_pad + pix0);
                    tma_store_commit();
                }
                if (++bx == n_box) { bx = 0; bpar ^= 1u; }
            }
            if (first >= n_blk) {
                // a single channel block: the second warp of the quadrant only releases the buffer
                if (lane == 0) mbar_arrive(smem_u32(&s_accfree[ab]));
            }
            if (publish) {
                // every lane's stores are ordered before the flag the reading warp acquires
                __threadfence();
                __syncwarp();
                if (lane == 0) st_release_gpu(flags + blockIdx.x * 8u + (warp - 4), 1u);
            }
            if (finish) {
                // this warp was the only reader of its counterparts' flags and has consumed their sums
                __syncwarp();
                if (lane == 0)
                    for (uint32_t pos = first_pos + 1u; pos <= last_pos; ++pos)
                        flags[(gridDim.x - 1u - pos) * 8u + (warp - 4)] = 0u;
            }
        }
        if (aborted(abort_flag)) {   // shortcut boxes still on their way to this CTA's shared memory (bounded)
            for (; taken != asked; ++taken) {
                (void)mbar_wait_polls(smem_u32(&s_res[warp - 4][bx]), bpar, 1u << 16);
                if (++bx == n_box) { bx = 0; bpar ^= 1u; }
            }
        }
        if (elect_one()) tma_store_wait_read();   // shared memory must outlive the stores' reads; the writes complete with the grid
    }

    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort != 0) {
        atomicExch(p.status + 0, static_cast<int>(NM_ERR_TIMEOUT));
        atomicExch(p.status + 1, 40 + s_abort);
        atomicExch(p.status + 2, static_cast<int>(blockIdx.x));
    }
    if (warp == 2) tmem_dealloc(tmem, 512);
}

// Second pass of a split-K plan: y[p][c] = act(sum over splits of partial[s][p][c] + bias[c] + residual[p][c]), the sums in the order of the
// splits.  It is bound by latency (19 MB of sums that are still in the L2 for 6272 x 256 outputs in three ranges): it lets the next kernel start early,
// and with the number of splits and the index type known at compile time every load of an output is in flight at once.  By itself, over 360 pairs
// of layer and split plan, the launch takes 4.3 % less than with a loop that does neither (256 -> 256, 3x3 at 14x14, batch 32, 2:8, three ranges of variant 4
// 18.3 -> 17.7 us); the instances are 2 % of it for two and four splits, 0.3 % for three.  S = 0: any number; I: index type.
template <int S, typename I>
__global__ void __launch_bounds__(256) k_splitk_reduce(const float4* __restrict__ part, int splits, size_t split_stride4, size_t n4, int c_out4,
                                                       const float4* __restrict__ bias, const float4* __restrict__ residual, int relu,
                                                       float4* __restrict__ y)
{
    nmk::pdl_launch_dependents();
    nmk::pdl_wait();   // the partial sums come from the kernel launched just before
    const I step = static_cast<I>(gridDim.x) * blockDim.x, n = static_cast<I>(n4);
    for (I i = blockIdx.x * static_cast<I>(blockDim.x) + threadIdx.x; i < n; i += step) {
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        float4 a;
        if (S > 0) {
            float4 v[S > 0 ? S : 1];
#pragma unroll
            for (int s = 0; s < S; ++s) v[s] = part[i + s * split_stride4];
            const float4 b = bias ? __ldg(bias + i % static_cast<I>(c_out4)) : zero, r = residual ? __ldg(residual + i) : zero;
            a = v[0];
#pragma unroll
            for (int s = 1; s < S; ++s) nm_add4(a, v[s]);
            if (bias) nm_add4(a, b);
            if (residual) nm_add4(a, r);
        } else {
            a = part[i];
            for (int s = 1; s < splits; ++s) nm_add4(a, part[i + s * split_stride4]);
            if (bias) nm_add4(a, __ldg(bias + i % static_cast<I>(c_out4)));
            if (residual) nm_add4(a, __ldg(residual + i));
        }
        if (relu) { a.x = fmaxf(a.x, 0.f); a.y = fmaxf(a.y, 0.f); a.z = fmaxf(a.z, 0.f); a.w = fmaxf(a.w, 0.f); }
        y[i] = a;
    }
}

bool make_cfg(const ConvParams& p, const nm_plan_t* plan, ExpandCfg* cfg)
{
    if (!p.wx || !nmtm::available()) return false;
    // whole 32-channel input blocks, or a pointwise layer whose last block the TMA unit fills up with zeros;
    // output channels in whole float4s (the expanded weights are padded to 32-row blocks)
    const bool pointwise = p.kh == 1 && p.kw == 1;
    if (p.c_in % 32 != 0 && !(pointwise && p.c_in % 4 == 0)) return false;
    if (p.c_out % 4 != 0 || p.wx_rows < p.c_out || p.wx_rows % 32 != 0) return false;
    if (!nmtm::im2col_geometry_ok(p)) return false;
    if (static_cast<long long>(p.batch) * p.h * p.w * p.c_in * 4 < 131072) return false;
    if (p.pixels >= (1ll << 31) - BM) return false;
    int bn = 0;
    if (plan && plan->bn > 0) {
        bn = plan->bn;
    } else {
        for (int cand : {128, 256, 64, 96, 32, 160, 192, 224})
            if (cand <= p.wx_rows && p.wx_rows % cand == 0) { bn = cand; break; }
    }
    if (bn < 32 || bn > 256 || bn % 32 != 0 || p.wx_rows % bn != 0) return false;
    cfg->bn = bn;
    cfg->n_slices = p.wx_rows / bn;
    cfg->sl_shift = (cfg->n_slices & (cfg->n_slices - 1)) == 0 ? __builtin_ctz(static_cast<unsigned>(cfg->n_slices)) : -1;
    cfg->b_bytes = ((bn * 128 + 1023) / 1024) * 1024;
    const int splits = plan && plan->split > 1 ? plan->split : 1;
    const bool balanced = plan && plan->split == -1;
    const int k_blocks = (p.k + 31) / 32;   // the last block of a pointwise layer may be partly zero fill
    if (splits > 8 || k_blocks % splits != 0) return false;
    cfg->ksplit = splits;
    const int blk32 = k_blocks / splits;   // 32-column blocks per work item
    const int kblk = plan && plan->kblk > 0 ? plan->kblk : 1;
    if (kblk > 2 || blk32 % kblk != 0) return false;
    cfg->kblk = kblk;
    cfg->n_sub = blk32 / kblk;
    // one issuer thread unless the plan asks for two (alternate stages, an accumulator each; one accumulator buffer
    // instead of two when both pairs do not fit the 512 columns)
    const int n_iss = plan && plan->issuers > 0 ? plan->issuers : 1;
    if (n_iss < 1 || n_iss > 2) return false;
    cfg->n_iss = n_iss;
    cfg->n_acc = 2 * n_iss * bn <= 512 ? 2 : 1;
    cfg->p_pad = static_cast<int>(((p.pixels + BM - 1) / BM) * BM);
    if (splits > 1 && (!p.splitk || p.splitk_bytes < static_cast<size_t>(splits) * cfg->p_pad * p.c_out * sizeof(float) ||
                       static_cast<long long>(splits) * cfg->p_pad >= (1ll << 31)))
        return false;   // the partial-sum scratch is reserved by nm_autotune
    cfg->boxes = blk32 <= 8 ? 2 : 1;   // long reductions: the epilogue is rare, the ring needs the bytes
    // A weight slice that fits stays resident (plan.split == 1 asks for streaming instead): the ring
    // then holds activations only and is deeper.  Needs one fixed slice per CTA, i.e. a grid that is a
    // multiple of the slice count.
    cfg->wres_bytes = 0;
    cfg->w_res = 0;
    if (splits == 1 && !balanced && !(plan && plan->split == 1) && blk32 * cfg->b_bytes <= WRES_MAX && cfg->n_slices <= nmhost::sm_count()) {
        cfg->w_res = 1;
        cfg->wres_bytes = blk32 * cfg->b_bytes;
        if (cfg->wres_bytes > 64 * 1024) cfg->boxes = 1;   // a large slice: give the output staging's room to the ring
    }
    cfg->flat = pointwise && p.stride_h == 1 && p.stride_w == 1 && p.pad_h == 0 && p.pad_w == 0;
    cfg->rows = BM;
    long long tiles = (p.pixels + BM - 1) / BM;
    if (splits == 1 && !balanced) {
        // fewest pixels per item (in steps of 8) that the same number of rounds covers
        const long long ctas = cfg->w_res ? nmhost::sm_count() / cfg->n_slices * cfg->n_slices : nmhost::sm_count();
        const long long rounds = (tiles * cfg->n_slices + ctas - 1) / ctas;
        const long long most = rounds * ctas / cfg->n_slices;   // pixel tiles that fit into them
        cfg->rows = static_cast<int>(((p.pixels + most - 1) / most + 7) / 8 * 8);
        if (cfg->rows > BM) cfg->rows = BM;
        if (cfg->rows < 32) cfg->rows = 32;   // a whole box; below that the weights cost more than the pixels
        tiles = (p.pixels + cfg->rows - 1) / cfg->rows;
    }
    // Rings.  Both operands are bound by bytes in flight: activations come from HBM, weights (the same for every CTA, twice the
    // bytes) from L2.  A slot holds the item's pixels only, and the weight ring gets as many slots as leave the activation
    // ring one more (at least three where that many of both fit).  1024 -> 256 at 14x14, batch 64 (88-pixel items): 20.2 us with
    // four slots of 16 + 32 KB, 18.8 with 5 + 4, 20.8 with 8 + 3; 256 -> 512 / 2 at 56x56: 39.9 -> 36.0 with 4 + 3, 51 with 2 + 4.
    cfg->a_bytes = (cfg->rows * 128 + 1023) / 1024 * 1024;
    const int a_slot = kblk * cfg->a_bytes, w_slot = cfg->w_res ? 0 : kblk * cfg->b_bytes;
    const int room = 227 * 1024 - 1024 - 2048 - cfg->wres_bytes;   // alignment slack, barriers
    const int asked = plan && plan->stages > 0 ? plan->stages : 0;
    if (p.residual && splits == 1) {
        // as many boxes as leave the ring four (three boxes) or three (two) blocks of 32 columns, or the stages asked for
        const int want = asked * (a_slot + w_slot), block = cfg->a_bytes + (cfg->w_res ? 0 : cfg->b_bytes);
        cfg->boxes = 1;
        for (int b = BOXES_MAX; b >= 2 && cfg->boxes == 1; --b) {
            const int left = room - 8 * b * BOX_BYTES;
            if (left >= (want ? want : (b + 1) * block) && left >= 2 * (a_slot + w_slot)) cfg->boxes = b;
        }
    }
    const int budget = room - 8 * cfg->boxes * BOX_BYTES;
    int na = asked, nw = cfg->w_res ? 0 : asked;
    if (asked == 0) {
        if (!cfg->w_res) {
            auto slots = [&](int n) { return std::min((budget - n * w_slot) / a_slot, NSTAGE_MAX); };
            nw = 2;
            while (slots(nw + 1) >= nw + 2) ++nw;
            if (nw == 2 && slots(3) >= 3) nw = 3;
        }
        na = (budget - nw * w_slot) / a_slot;
        if (na > NSTAGE_MAX) na = NSTAGE_MAX;
        if (n_iss == 2) na &= ~1;
    }
    // (a plan may ask for a single slot; the default is at least two)
    if (na < (asked ? 1 : 2) || na > NSTAGE_MAX || na * a_slot + nw * w_slot > budget) return false;
    if (nw > na) nw = na;
    if (n_iss == 2 && na % 2 != 0) return false;   // two issuers own alternate ring slots
    cfg->stages = na;
    cfg->w_stages = nw;
    cfg->n_work = tiles * cfg->n_slices * splits;
    if (cfg->n_work >= (1ll << 31)) return false;
    // A pointwise layer that reads more than it writes walks its pixels backwards: its input is as a rule the layer before's output, written
    // front to back, and the end of it is what the L2 still holds most of.  By itself (us, forwards and backwards): ResNet-101 at batch 128, 2:8 5155,
    // 5023; ResNet-50 at batch 64, 2:4 1857, 1827; MobileNet-V2's pointwise layers, each on an input of its own, 310, 310.  Only for maps beyond
    // the L2's 126 MB 5118 and 1846: a smaller one shares it with the shortcut and the outputs since.
    cfg->last_tile = pointwise && splits == 1 && !balanced && nm_pointwise_reads_more(p) ? static_cast<int>(tiles) - 1 : -1;
    cfg->balanced = 0;
    if (balanced) {
        // one range per SM; needs at least one (item, stage) unit per CTA and the per-CTA slots + flags in the scratch
        const long long units = cfg->n_work * cfg->n_sub;
        if (units < nmhost::sm_count() || units >= (1ll << 31)) return false;
        if (!p.splitk || p.splitk_bytes < nmhost::expand_balanced_bytes(bn)) return false;
        cfg->balanced = 1;
    }
    return true;
}

}  // namespace

namespace nmhost {

size_t expand_balanced_bytes(int bn)
{
    // per SM: a slot of 128 rows x bn partial sums, and eight flag words (one per epilogue warp)
    return static_cast<size_t>(nmhost::sm_count()) * (static_cast<size_t>(BM) * bn * sizeof(float) + 8 * sizeof(uint32_t));
}

bool expand_plan_ok(const ConvParams& p, const nm_plan_t* plan)
{
    ExpandCfg cfg;
    return make_cfg(p, plan, &cfg);
}

nm_status_t launch_conv_expand(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st)
{
    ExpandCfg cfg;
    if (!make_cfg(p, plan, &cfg))
        return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: the expanded-operand kernel does not take this layer / plan%s",
                    plan && (plan->split > 1 || plan->split == -1) ? " (a split or balanced plan needs scratch: nm_weights_reserve)" : "");
    // a split-K plan stores raw partial sums [split][pixel][channel] in the handle's scratch; bias and
    // activation are applied by the reduction pass
    ConvParams q = p;
    if (cfg.ksplit > 1) {
        q.y = p.splitk;
        q.pixels = static_cast<long long>(cfg.ksplit) * cfg.p_pad;   // rows of the store map
        q.bias = nullptr;
        q.residual = nullptr;
        q.relu = 0;
    }
    alignas(64) CUtensorMap tm_x, tm_y, tm_tail, tm_res;
    if (!(cfg.flat ? nmtm::encode_x_rows(p, cfg.rows, &tm_x) : nmtm::encode_x_im2col(p, cfg.rows, &tm_x)) || !nmtm::encode_y_tiled(q, &tm_y))
        return fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 4)");
    tm_res = tm_y;
    if (q.residual && !nmtm::encode_y_tiled(q, &tm_res, 32, q.residual))
        return fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 4)");
    tm_tail = tm_y;   // an item's last box, when its pixels are no multiple of 32
    if (cfg.rows % 32 != 0 && !nmtm::encode_y_tiled(q, &tm_tail, cfg.rows % 32))
        return fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 4)");
    q.pixels = p.pixels;
    size_t smem = 1024 + cfg.wres_bytes + static_cast<size_t>(cfg.stages) * cfg.kblk * cfg.a_bytes +
                  static_cast<size_t>(cfg.w_stages) * cfg.kblk * cfg.b_bytes + 8 * cfg.boxes * BOX_BYTES;
    if (smem < NM_EXCLUSIVE_SMEM) smem = NM_EXCLUSIVE_SMEM;   // one CTA per SM: it owns all 512 TMEM columns
    using Kernel = void (*)(const ConvParams, const ExpandCfg, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap);
    const Kernel kernel = cfg.balanced ? (cfg.kblk == 2 ? k_conv_expand<2, true> : k_conv_expand<1, true>)
                                       : (cfg.kblk == 2 ? k_conv_expand<2, false> : k_conv_expand<1, false>);
    cudaError_t e = nmhost::ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "cudaFuncSetAttribute (variant 4): %s", cudaGetErrorString(e));
    long long grid = cfg.n_work < nmhost::sm_count() ? cfg.n_work : nmhost::sm_count();
    if (cfg.balanced) grid = nmhost::sm_count();
    if (cfg.w_res) grid = (grid / cfg.n_slices) * cfg.n_slices;   // n_work is a multiple of n_slices, so grid >= n_slices
    e = nmhost::launch_pdl(kernel, static_cast<unsigned>(grid), THREADS, smem, st, q, cfg, tm_x, tm_y, tm_tail, tm_res);
    nmhost::count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "nm_conv2d launch (variant 4): %s", cudaGetErrorString(e));
    if (cfg.ksplit > 1) return launch_splitk_reduce(p, cfg.ksplit, cfg.p_pad, st);
    return NM_OK;
}

nm_status_t launch_splitk_reduce(const ConvParams& p, int splits, int p_pad, cudaStream_t st)
{
    const size_t n4 = static_cast<size_t>(p.pixels) * p.c_out / 4;
    const size_t stride4 = static_cast<size_t>(p_pad) * p.c_out / 4;
    size_t blocks = (n4 + 255) / 256;
    if (blocks > static_cast<size_t>(nmhost::sm_count()) * 8) blocks = static_cast<size_t>(nmhost::sm_count()) * 8;
    const bool small = n4 < (size_t(1) << 31);
    const auto kernel = !small ? k_splitk_reduce<0, size_t> : splits == 2 ? k_splitk_reduce<2, uint32_t> : splits == 3 ? k_splitk_reduce<3, uint32_t> :
                        splits == 4 ? k_splitk_reduce<4, uint32_t> : k_splitk_reduce<0, uint32_t>;
    cudaError_t e = nmhost::launch_pdl(kernel, static_cast<unsigned>(blocks), 256u, 0, st,
                                       reinterpret_cast<const float4*>(p.splitk), splits, stride4, n4, p.c_out / 4,
                                       reinterpret_cast<const float4*>(p.bias), reinterpret_cast<const float4*>(p.residual),
                                       p.relu, reinterpret_cast<float4*>(p.y));
    nmhost::count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "nm_conv2d launch (split-K reduction): %s", cudaGetErrorString(e));
    return NM_OK;
}

size_t expand_splitk_bytes(const ConvParams& p, int splits)
{
    const size_t p_pad = static_cast<size_t>((p.pixels + BM - 1) / BM) * BM;
    return static_cast<size_t>(splits) * p_pad * p.c_out * sizeof(float);
}

}  // namespace nmhost
