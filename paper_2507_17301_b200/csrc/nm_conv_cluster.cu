// Variant 10: cluster kernel — short launches (few images, small maps) as one small tile per CTA, the reduction axis split over
// the CTAs of a thread-block cluster.
//
// A batch-1 layer is a few microseconds of latencies in series, not of bytes or FLOPs: the persistent kernels give it a
// handful of SMs, walk its whole reduction axis on each (72 stages for a 3x3 layer of 256 channels), or split it through
// scratch memory and a second launch.  Here a work item (up to 128 pixels x BN channels, BN = 32, 64 or 128) belongs to a
// cluster of S = 1, 2, 4 or 8 CTAs, each of which
//   * accumulates its contiguous range of 32-column blocks in tensor memory (operands as in variant 4: dense activations
//     by TMA, zero-expanded weights by bulk copy, SS MMA),
//   * sends every run of rows of its partial sums to the CTA that finishes the run (the rows of an item are dealt to the CTAs
//     in S runs): one bulk copy from shared to distributed shared memory each, counted by a barrier there (with remote
//     stores of 16 bytes each, plain or asynchronous, it took 1.3-1.9 us from the accumulator to the last arrival; 0.7 us with
//     the copies, ResNet-50 at batch 1 343 -> 316 us), and
//   * once its own rows are complete adds the S partial sums in the order of the ranges (the result does not depend on
//     timing), adds bias and shortcut, applies the activation and writes whole 128-byte rows to NHWC.
// No scratch memory, no second launch.  A CTA takes a quarter to a half of an SM's shared memory and BN tensor-memory columns, so
// that the next launch's CTAs become resident beside it (programmatic dependent launch): they set up their barriers and
// fetch their first WEIGHT tiles, which no earlier kernel of the stream writes (a handle is complete when the call that
// built it returns), while this launch still runs.
//
// Activations come in one of three forms: plain 2-D rows (pointwise, stride 1), im2col-mode loads (any stride, dilation and
// kernel; inputs of at least 128 KiB), or, for smaller inputs at stride 1, one 4-D box of whole output rows per block and
// tap.  In every form an operand row is an output pixel and the item's pixels are consecutive.
//
//   producer (1 thread), MMA issuer (1 thread), four warps for the reduction and the store; bounded waits.
#include "nm_internal.h"
#include "nm_ptx.cuh"
#include "nm_tmap.cuh"

namespace {

using namespace nmk;

constexpr int THREADS = 192;      // warps: 0 producer, 1 MMA issuer and tensor memory, 2-5 reduction and store
constexpr int NSTAGE_MAX = 12;
constexpr int EPI = 128;          // threads of the reduction

enum LoadForm { ROWS_2D = 0, IM2COL = 1, BOX_4D = 2 };

struct ClusterCfg {
    int bn, n_slices;
    int cs;           // CTAs per cluster = ranges of the reduction axis
    int n_blk;        // 32-column blocks of the reduction axis
    int stages;       // ring depth
    int form;
    int rows;         // operand rows (output pixels) of a full item
    int tiles;        // items along the pixels
    int row_blocks;   // BOX_4D: items per image
    int r_rows;       // BOX_4D: output rows per item
    int a_bytes;      // bytes one activation load delivers
    int b_off;        // offset of the weight tile inside a stage
    int stage_bytes;
    int rps;          // rows a CTA finishes
    int round;        // 1: activations rounded to nearest (inputs that have no im2col form, of less than 128 KiB for instance)
};

__device__ __forceinline__ bool aborted(volatile int* flag) { return *flag != 0; }

__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* tmap, uint32_t bar, int c, int w, int h, int n)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(dst), "l"(tmap), "r"(bar), "r"(c), "r"(w), "r"(h), "r"(n)
        : "memory");
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

// CS: CTAs per cluster; Q4: log2 of the float4s per row (BN / 4).
template <int CS, int Q4>
__global__ void __launch_bounds__(THREADS, 2)
k_conv_cluster(const ConvParams p, const ClusterCfg cfg, const __grid_constant__ CUtensorMap tm_x)
{
    extern __shared__ uint8_t smem_raw[];
    __shared__ uint64_t s_full[NSTAGE_MAX], s_free[NSTAGE_MAX], s_acc, s_part;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;

    const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
    constexpr int BN = 4 << Q4;
    const int NS = cfg.stages;
    const uint32_t ring = (smem_u32(smem_raw) + 1023u) & ~1023u;
    // partial sums of this CTA's rows, [source CTA][row][bn], after the ring and the rows the last stage's MMAs may overread
    const uint32_t part = ring + NS * cfg.stage_bytes + 128u * 128u;
    constexpr uint32_t tmem_cols = BN;
    volatile int* abort_flag = &s_abort;
    const uint32_t rank = cluster_ctarank();

    if (warp == 1) tmem_alloc(smem_u32(&s_tmem), tmem_cols);
    if (tid == 0) {
        for (int i = 0; i < NSTAGE_MAX; ++i) {
            mbar_init(smem_u32(&s_full[i]), 1);
            mbar_init(smem_u32(&s_free[i]), 1);
        }
        mbar_init(smem_u32(&s_acc), 1);
        mbar_init(smem_u32(&s_part), 1);
        mbar_fence_init();
        s_abort = 0;
        tma_prefetch_desc(&tm_x);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    // the item of this cluster and this CTA's range of the reduction axis
    const uint32_t item = blockIdx.x / CS;
    const uint32_t tile = item / static_cast<uint32_t>(cfg.n_slices);
    const int slice = static_cast<int>(item - tile * static_cast<uint32_t>(cfg.n_slices));
    const int c_begin = static_cast<int>(rank) * cfg.n_blk / CS, c_end = (static_cast<int>(rank) + 1) * cfg.n_blk / CS;
    const int hw = p.ho * p.wo;
    long long pix0;
    int count, img = 0, oh0 = 0;   // pixels of the item; BOX_4D: its image and first output row
    if (cfg.form == BOX_4D) {
        img = static_cast<int>(tile / static_cast<uint32_t>(cfg.row_blocks));
        oh0 = static_cast<int>(tile - static_cast<uint32_t>(img) * static_cast<uint32_t>(cfg.row_blocks)) * cfg.r_rows;
        pix0 = static_cast<long long>(img) * hw + static_cast<long long>(oh0) * p.wo;
        count = (p.ho - oh0 < cfg.r_rows ? p.ho - oh0 : cfg.r_rows) * p.wo;
    } else {
        pix0 = static_cast<long long>(tile) * cfg.rows;
        count = p.pixels - pix0 < cfg.rows ? static_cast<int>(p.pixels - pix0) : cfg.rows;
    }

    const int row0 = static_cast<int>(rank) * cfg.rps;   // first row of the item that this CTA finishes
    int my_rows = count - row0;                          // how many of its rows exist
    if (my_rows > cfg.rps) my_rows = cfg.rps;
    if (my_rows < 0) my_rows = 0;
    if (CS > 1) {
        // the barrier knows how many bytes to expect, and every CTA of the cluster has started, before any of them sends
        // (waited for below)
        if (tid == 0) mbar_arrive_expect_tx(smem_u32(&s_part), static_cast<uint32_t>(my_rows) * (BN * 4) * CS);
        asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    }
    pdl_launch_dependents();

    if (warp == 0) {
        // =========================== producer ===========================
        if (elect_one()) {
            const uint32_t w_bytes = static_cast<uint32_t>(BN) * 128u;
            const uint32_t tx = static_cast<uint32_t>(cfg.a_bytes) + w_bytes;
            const size_t w_step = static_cast<size_t>(p.wx_rows) * 32;
            const float* wsrc = p.wx + static_cast<size_t>(c_begin) * w_step + static_cast<size_t>(slice) * BN * 32;
            const int n = c_end - c_begin, first = n < NS ? n : NS;
            // the ring's first weight tiles do not depend on the previous kernel
            for (int i = 0; i < first; ++i) {
                const uint32_t bar = smem_u32(&s_full[i]);
                mbar_arrive_expect_tx(bar, tx);
                bulk_load_1d(ring + i * cfg.stage_bytes + cfg.b_off, wsrc + static_cast<size_t>(i) * w_step, w_bytes, bar);
            }
            int n0 = img, w0 = 0, h0 = 0;
            if (cfg.form == IM2COL) {
                n0 = static_cast<int>(static_cast<uint32_t>(pix0) / static_cast<uint32_t>(hw));
                const int rem = static_cast<int>(static_cast<uint32_t>(pix0) - static_cast<uint32_t>(n0) * static_cast<uint32_t>(hw));
                const int oh = rem / p.wo, ow = rem - oh * p.wo;
                w0 = ow * p.stride_w - p.pad_w;
                h0 = oh * p.stride_h - p.pad_h;
            } else if (cfg.form == BOX_4D) {
                w0 = -p.pad_w;
                h0 = oh0 - p.pad_h;
            }
            int ch = 0, tw = 0, off_w = 0, off_h = 0;
            if (c_begin != 0) {
                const int tap0 = (c_begin * 32) / p.c_in, th = tap0 / p.kw;
                ch = c_begin * 32 - tap0 * p.c_in;
                tw = tap0 - th * p.kw;
                off_w = tw * p.dil_w;
                off_h = th * p.dil_h;
            }
            pdl_wait();
            RingPos rp;
            int issued = 0;
            for (int i = 0; i < n; ++i) {
                if (rp.wrapped && !mbar_wait_lone(smem_u32(&s_free[rp.s]), rp.parity ^ 1u)) *abort_flag = 2;
                if (aborted(abort_flag)) break;
                const uint32_t a_smem = ring + rp.s * cfg.stage_bytes;
                const uint32_t bar = smem_u32(&s_full[rp.s]);
                if (i >= first) {
                    mbar_arrive_expect_tx(bar, tx);
                    bulk_load_1d(a_smem + cfg.b_off, wsrc + static_cast<size_t>(i) * w_step, w_bytes, bar);
                }
                if (cfg.form == ROWS_2D) tma_load_2d(a_smem, &tm_x, bar, ch, static_cast<int>(pix0));
                else if (cfg.form == IM2COL)
                    tma_load_im2col_4d(a_smem, &tm_x, bar, ch, w0, h0, n0, static_cast<uint16_t>(off_w), static_cast<uint16_t>(off_h));
                else tma_load_4d(a_smem, &tm_x, bar, ch, w0 + off_w, h0 + off_h, n0);
                ch += 32;
                if (ch >= p.c_in) {
                    ch = 0;
                    off_w += p.dil_w;
                    if (++tw == p.kw) { tw = 0; off_w = 0; off_h += p.dil_h; }
                }
                rp.advance(NS);
                ++issued;
            }
            if (aborted(abort_flag)) {
                // loads in flight still target this CTA's shared memory: let them land (weight tiles without their activations
                // never complete a barrier; the wait is bounded)
                for (int back = 0; back < NS && back < issued; ++back) {
                    if (rp.s == 0) { rp.s = NS; rp.parity ^= 1u; }
                    --rp.s;
                    (void)mbar_wait(smem_u32(&s_full[rp.s]), rp.parity);
                }
            }
        }
    } else if (warp == 1) {
        // =========================== MMA issuer ===========================
        if (elect_one()) {
            const uint32_t idesc = umma_idesc_tf32(128, BN);
            RingPos rp;
            uint32_t started = 0;
            for (int i = c_begin; i < c_end; ++i) {
                if (!mbar_wait_lone(smem_u32(&s_full[rp.s]), rp.parity)) { *abort_flag = 3; break; }
                tc_fence_after();
                const uint32_t a_smem = ring + rp.s * cfg.stage_bytes;
                const uint64_t adesc = umma_desc_k_sw128(a_smem, 1024), bdesc = umma_desc_k_sw128(a_smem + cfg.b_off, 1024);
#pragma unroll
                for (int kq = 0; kq < 4; ++kq) umma_tf32_ss(tmem, adesc + 2 * kq, bdesc + 2 * kq, idesc, kq > 0 ? 1u : started);
                started = 1u;
                umma_commit(smem_u32(&s_free[rp.s]));
                rp.advance(NS);
            }
            umma_commit(smem_u32(&s_acc));
        }
    }
    __syncwarp();
    if (CS > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // every CTA of the cluster is running
    if (warp >= 2) {
        // =========================== reduction and store ===========================
        // Everything that does not depend on the sums is worked out, and the bias and the first shortcut pieces are loaded, before the
        // accumulator is ready.  A thread's output pieces (16 bytes) lie STEP rows apart in the same channels, so it needs one piece
        // of the bias.  (Fetched piece by piece between the stores, bias and shortcut cost a CTA without a cluster 1.1 us at its end:
        // 192 -> 32 at 28x28, batch 32, 4.9 us.)
        const int e = tid - 64;
        constexpr int STEP = EPI >> Q4;
        // output pieces whose shortcut is fetched together: all of a thread's, up to eight
        constexpr int AHEAD = (1 << Q4) / CS > 8 ? 8 : (1 << Q4) / CS;
        const int c = e & ((1 << Q4) - 1), r0 = e >> Q4, o = slice * BN + c * 4;
        const bool mine = o < p.c_out;
        const size_t at_out = static_cast<size_t>(pix0 + row0 + r0) * p.c_out + o, out_step = static_cast<size_t>(STEP) * p.c_out;
        const float* res = p.residual && mine ? p.residual + at_out : nullptr;
        float* out = p.y + at_out;
        const int q = warp & 3;        // tensor-memory lane quadrant this warp may read
        const int row = q * 32 + lane;
        const int lrow = CS > 1 ? row % cfg.rps : row;
        const uint32_t dst = (CS > 1 ? ring : part) + row * (BN * 4), dst_swz = static_cast<uint32_t>(lrow & 7) << 4;
        const uint32_t src_step = static_cast<uint32_t>(cfg.rps) * (BN * 4);
        // the copies this warp sends: source, destination, barrier there, bytes
        constexpr int SENDS = CS > 4 ? 2 : 1;
        uint32_t send_src[SENDS], send_dst[SENDS], send_bar[SENDS], send_bytes[SENDS];
        if (CS > 1) {
#pragma unroll
            for (int k = 0; k < SENDS; ++k) {
                const int owner = q + 4 * k;
                int rows = owner < CS ? count - owner * cfg.rps : 0;
                if (rows > cfg.rps) rows = cfg.rps;
                send_bytes[k] = rows > 0 ? static_cast<uint32_t>(rows) * (BN * 4) : 0u;
                send_src[k] = ring + owner * src_step;
                send_dst[k] = send_bytes[k] ? mapa_shared(part + rank * src_step, static_cast<uint32_t>(owner)) : 0u;
                send_bar[k] = send_bytes[k] ? mapa_shared(smem_u32(&s_part), static_cast<uint32_t>(owner)) : 0u;
            }
        }
        pdl_wait();   // bias and shortcut are read, and y written, only after the previous kernel
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 bias = p.bias && mine ? __ldg(reinterpret_cast<const float4*>(p.bias + o)) : zero;
        float4 ahead[AHEAD];               // shortcut pieces
        auto fetch = [&](int r) {
#pragma unroll
            for (int k = 0; k < AHEAD; ++k)
                ahead[k] = res && r + k * STEP < my_rows ? __ldg(reinterpret_cast<const float4*>(res + k * out_step)) : zero;
        };
        fetch(r0);
        const bool ok = aborted(abort_flag) || mbar_wait(smem_u32(&s_acc), 0);
        if (!__all_sync(0xFFFFFFFFu, ok)) *abort_flag = 4;
        tc_fence_after();
        // A row of partial sums per thread, into this CTA's own shared memory: over the ring, which is idle now (with one CTA
        // per item straight to where they are added up).  16-byte pieces are XOR-ed with the row inside its run, so that the
        // 32 rows of a warp do not meet in one bank.
#pragma unroll
        for (int blk = 0; blk < BN / 32; ++blk) {
            uint32_t v[32];
            tmem_ld32(tmem + (static_cast<uint32_t>(q * 32) << 16) + blk * 32, v);
            tmem_ld_wait();
            if (row < count) {
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + blk * 128 + ((k << 4) ^ dst_swz)), "r"(v[4 * k]),
                                 "r"(v[4 * k + 1]), "r"(v[4 * k + 2]), "r"(v[4 * k + 3])
                                 : "memory");
            }
        }
        tc_fence_before();
        if (CS > 1) fence_proxy_async();
        asm volatile("bar.sync 1, %0;" ::"n"(EPI) : "memory");
        if (CS > 1) {
            if (elect_one()) {
#pragma unroll
                for (int k = 0; k < SENDS; ++k)
                    if (send_bytes[k]) bulk_copy_cluster(send_dst[k], send_src[k], send_bytes[k], send_bar[k]);
            }
            __syncwarp();
            // every partial sum of this CTA's rows has landed; the limit is a multiple of the other waits', so that a CTA of the
            // cluster that gave up on one of those has sent by then
            const uint32_t bar_own = smem_u32(&s_part);
            const bool landed = mbar_wait_cluster(bar_own, 0) || mbar_wait_cluster(bar_own, 0) || mbar_wait_cluster(bar_own, 0);
            if (!__all_sync(0xFFFFFFFFu, landed)) *abort_flag = 5;
            asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        }
        if (!aborted(abort_flag)) {
            for (int r = r0; r < my_rows; r += AHEAD * STEP) {
                if (r != r0) fetch(r);
#pragma unroll
                for (int k = 0; k < AHEAD; ++k) {
                    const int rk = r + k * STEP;
                    if (rk < my_rows) {
                        const uint32_t at = part + ((rk << Q4) + ((c & ~7) | ((c ^ rk) & 7))) * 16;
                        float4 s[CS];
#pragma unroll
                        for (int i = 0; i < CS; ++i) s[i] = ld_shared_f4(at + i * src_step);
#pragma unroll
                        for (int i = 1; i < CS; ++i) nm_add4(s[0], s[i]);
                        nm_add4(ahead[k], bias);
                        nm_add4(s[0], ahead[k]);
                        if (p.relu) { s[0].x = fmaxf(s[0].x, 0.f); s[0].y = fmaxf(s[0].y, 0.f); s[0].z = fmaxf(s[0].z, 0.f); s[0].w = fmaxf(s[0].w, 0.f); }
                        if (mine) *reinterpret_cast<float4*>(out + k * out_step) = s[0];
                    }
                }
                out += AHEAD * out_step;
                if (res) res += AHEAD * out_step;
            }
        }
    }

    if (CS > 1) {
        // a CTA leaves once every CTA of the cluster has what was sent to it: its copies have then been read
        if (warp < 2) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_abort != 0) {
        atomicExch(p.status + 0, static_cast<int>(NM_ERR_TIMEOUT));
        atomicExch(p.status + 1, 100 + s_abort);
        atomicExch(p.status + 2, static_cast<int>(blockIdx.x));
    }
    if (warp == 1) tmem_dealloc(tmem, tmem_cols);
}

bool make_cfg(const ConvParams& p, const nm_plan_t* plan, ClusterCfg* cfg, size_t* smem)
{
    if (!p.wx || !nmtm::available()) return false;
    const bool pointwise = p.kh == 1 && p.kw == 1;
    if (p.c_in % 32 != 0 && !(pointwise && p.c_in % 4 == 0)) return false;
    if (p.c_out % 4 != 0 || p.pixels >= (1ll << 31) - 128) return false;
    const bool small = static_cast<long long>(p.batch) * p.h * p.w * p.c_in * 4 < 131072;   // no im2col map of so small a tensor
    const bool unit = p.stride_h == 1 && p.stride_w == 1;
    if (pointwise && unit && p.pad_h == 0 && p.pad_w == 0) cfg->form = ROWS_2D;
    else if (!small && nmtm::im2col_geometry_ok(p)) cfg->form = IM2COL;
    else if (unit && p.wo <= 128) cfg->form = BOX_4D;
    else return false;
    cfg->round = small || cfg->form == BOX_4D ? 1 : 0;
    cfg->n_blk = (p.k + 31) / 32;
    cfg->cs = plan && plan->ksplit > 0 ? plan->ksplit : 1;
    if ((cfg->cs != 1 && cfg->cs != 2 && cfg->cs != 4 && cfg->cs != 8) || cfg->n_blk < cfg->cs) return false;
    const int bn = plan && plan->bn > 0 ? plan->bn : 32;
    if ((bn != 32 && bn != 64 && bn != 128) || p.wx_rows % bn != 0) return false;
    cfg->bn = bn;
    cfg->n_slices = p.wx_rows / bn;
    cfg->row_blocks = cfg->r_rows = 0;
    if (cfg->form == BOX_4D) {
        // whole output rows of one image, dealt evenly
        const int most = 128 / p.wo < p.ho ? 128 / p.wo : p.ho;
        cfg->row_blocks = (p.ho + most - 1) / most;
        cfg->r_rows = (p.ho + cfg->row_blocks - 1) / cfg->row_blocks;
        cfg->row_blocks = (p.ho + cfg->r_rows - 1) / cfg->r_rows;
        cfg->rows = cfg->r_rows * p.wo;
        const long long tiles = static_cast<long long>(p.batch) * cfg->row_blocks;
        if (tiles > (1 << 20)) return false;
        cfg->tiles = static_cast<int>(tiles);
    } else {
        // as few items as 128-row tiles allow, of equal size (a multiple of 8 rows): 196 pixels are 2 x 104, not 128 + 68
        const long long tiles = (p.pixels + 127) / 128;
        if (tiles > (1 << 20)) return false;
        cfg->rows = static_cast<int>(((p.pixels + tiles - 1) / tiles + 7) / 8 * 8);
        cfg->tiles = static_cast<int>((p.pixels + cfg->rows - 1) / cfg->rows);
    }
    if (static_cast<long long>(cfg->tiles) * cfg->n_slices * cfg->cs > (1 << 24)) return false;
    cfg->rps = (cfg->rows + cfg->cs - 1) / cfg->cs;
    cfg->a_bytes = cfg->rows * 128;
    // the MMAs read 128 rows: rows past the item's come from the weight tile and the next stage, and the accumulator
    // rows they produce are never read
    cfg->b_off = (cfg->a_bytes + 1023) / 1024 * 1024;
    cfg->stage_bytes = cfg->b_off + bn * 128;
    // Ring: the whole range of a CTA if it fits half an SM, so that two CTAs (of this launch or the next) share one.
    const int range = (cfg->n_blk + cfg->cs - 1) / cfg->cs;
    const int fixed = 1024 + 128 * 128 + cfg->cs * cfg->rps * bn * 4;
    const int budget = 111 * 1024 - fixed;
    int stages = plan && plan->stages > 0 ? plan->stages : (range < NSTAGE_MAX ? range : NSTAGE_MAX);
    if (stages > NSTAGE_MAX) return false;
    while (stages > 1 && stages * cfg->stage_bytes > budget) --stages;
    if (cfg->cs > 1 && stages * cfg->stage_bytes + 128 * 128 < cfg->rows * bn * 4) return false;   // the sums to send lie over the ring
    if (stages * cfg->stage_bytes > budget || (stages < 2 && range > 1)) return false;
    cfg->stages = stages;
    *smem = static_cast<size_t>(fixed) + static_cast<size_t>(stages) * cfg->stage_bytes;
    // The CTAs of a cluster wait for one another, so none of them may be held up in its tensor-memory allocation by a CTA
    // that waits in turn: a CTA takes at least its columns' share of the SM's shared memory (kernels that allocate all 512
    // columns take NM_EXCLUSIVE_SMEM, next to which no CTA of this kernel fits).
    const size_t share = static_cast<size_t>(bn) * (228 * 1024 / 512);
    if (*smem < share) *smem = share;
    if (*smem < NM_BESIDE_EXCLUSIVE) *smem = NM_BESIDE_EXCLUSIVE;
    // Short launches only: with many rounds of CTAs the persistent kernels keep the tensor core busier.
    return static_cast<long long>(cfg->tiles) * cfg->n_slices * cfg->cs <= 12ll * nmhost::sm_count();
}

bool encode_x(const ConvParams& p, const ClusterCfg& cfg, CUtensorMap* tm)
{
    if (cfg.form == IM2COL) return nmtm::encode_x_im2col(p, cfg.rows, tm);
    const bool rows = cfg.form == ROWS_2D;
    // Inputs that have no im2col form (below 128 KiB) are otherwise taken by kernels that round activations to nearest (variants 1 and
    // 2): for them the TMA unit rounds on the way into shared memory (to nearest, ties to even, in no extra time), where the tensor core would truncate.
    // Last map of ResNet-50 at 96 x 96, batch 1, against 64 bits: 3.1e-3 truncated, 1.8e-3 rounded
    // (248 us either way); ResNet-101 at 100 x 100, batch 2, 3:4: 1.5e-2 and 7.7e-3.
    const CUtensorMapDataType type = cfg.round ? CU_TENSOR_MAP_DATA_TYPE_TFLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const cuuint64_t c = static_cast<cuuint64_t>(p.c_in), w = static_cast<cuuint64_t>(p.w), h = static_cast<cuuint64_t>(p.h),
                     n = static_cast<cuuint64_t>(p.batch);
    const cuuint64_t dims2[2] = {c, n * h * w}, dims4[4] = {c, w, h, n};
    const cuuint64_t strides[3] = {c * 4, w * c * 4, h * w * c * 4};
    const cuuint32_t box2[2] = {32, static_cast<cuuint32_t>(cfg.rows)};
    const cuuint32_t box4[4] = {32, static_cast<cuuint32_t>(p.wo), static_cast<cuuint32_t>(cfg.r_rows), 1};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    return nmtm::encoders().tiled(tm, type, rows ? 2 : 4, const_cast<float*>(p.x), rows ? dims2 : dims4, strides,
                                  rows ? box2 : box4, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

namespace {

using Kernel = void (*)(const ConvParams, const ClusterCfg, const CUtensorMap);
template <int CS>
Kernel kernel_of(int bn)
{
    return bn == 32 ? k_conv_cluster<CS, 3> : bn == 64 ? k_conv_cluster<CS, 4> : k_conv_cluster<CS, 5>;
}

}  // namespace

namespace nmhost {

bool cluster_plan_ok(const ConvParams& p, const nm_plan_t* plan)
{
    ClusterCfg cfg;
    size_t smem = 0;
    return make_cfg(p, plan, &cfg, &smem);
}

nm_status_t launch_conv_cluster(const ConvParams& p, const nm_plan_t* plan, cudaStream_t st)
{
    ClusterCfg cfg;
    size_t smem = 0;
    if (!make_cfg(p, plan, &cfg, &smem))
        return fail(NM_ERR_UNSUPPORTED, "nm_conv2d: the cluster kernel does not take this layer / plan");
    alignas(64) CUtensorMap tm_x;
    if (!encode_x(p, cfg, &tm_x)) return fail(NM_ERR_CUDA, "nm_conv2d: tensor-map encoding failed (variant 10)");
    const Kernel kernel = cfg.cs == 1 ? kernel_of<1>(cfg.bn) : cfg.cs == 2 ? kernel_of<2>(cfg.bn) : cfg.cs == 4 ? kernel_of<4>(cfg.bn) : kernel_of<8>(cfg.bn);
    cudaError_t e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "cudaFuncSetAttribute (variant 10): %s", cudaGetErrorString(e));
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(static_cast<unsigned>(cfg.tiles * cfg.n_slices * cfg.cs));
    lc.blockDim = dim3(THREADS);
    lc.dynamicSmemBytes = smem;
    lc.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(cfg.cs);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 2 : 1;
    e = cudaLaunchKernelEx(&lc, kernel, p, cfg, tm_x);
    count_launch(1);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return fail(NM_ERR_CUDA, "nm_conv2d launch (variant 10): %s", cudaGetErrorString(e));
    return NM_OK;
}

}  // namespace nmhost
