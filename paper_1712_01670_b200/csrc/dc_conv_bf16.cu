// Partial convolution on the 5th-generation tensor cores (bf16 in, fp32 accumulate in TMEM).
//
// Section 5, "Reuse", third step: convolve only what the cache did not supply.  The unit of
// work is one dirty 16x8 output tile (128 pixels = the M of one tcgen05.mma) times one block of
// BN output channels.  It is an implicit GEMM: for every kernel tap (ky, kx) and every chunk of
// BK input channels, TMA fetches
//     A: the 16x8 window of the NHWC input map displaced by the tap (a 4-D box; coordinates
//        outside the map are zero-filled, which is the convolution's padding), 128 rows x BK
//     B: BN rows x BK of the weights, which are already K-major as [cout][kh][kw][cin]
// into 128-byte-swizzled shared memory, and one elected thread issues BK/16 tcgen05.mma
// (M = 128, N = BN, K = 16) accumulating into tensor memory.
//
// Warp roles in a CTA of 192 threads (persistent, one CTA per SM):
//     warp 0      TMA producer             (full/empty mbarrier ring of `stages` slots)
//     warp 1      TMEM allocation, MMA issue, tcgen05.commit
//     warps 2-5   epilogue: tcgen05.ld of their 32-lane quadrant, + bias, ReLU, bf16, and a
//                 store predicated on the tile's reuse bitmap (only non-reused pixels are written)
// Two accumulators (2 x BN TMEM columns) let the epilogue of one work item overlap the MMAs of
// the next.  Every mbarrier wait is bounded: on expiry the kernel records DC_ERR_TIMEOUT in the
// status word, all roles leave their loops, tensor memory is freed and the kernel returns.
#include <cuda.h>
#include <stdio.h>
#include <stdlib.h>

#include "dc_common.cuh"
#include "dc_conv_cluster.cuh"
#include "dc_tcgen05.cuh"

namespace {

constexpr int kThreads = 192;          // producer warp, MMA warp, four epilogue warps
constexpr int kThreadsWide = 320;      // ... or eight epilogue warps
static inline int threads_for(int epi_warps) { return 64 + 32 * epi_warps; }
constexpr int kMaxStages = 8;
constexpr unsigned long long kWaitLimitNs = 2000000000ull;   // 2 s

struct TcArgs {
    const float* bias; __nv_bfloat16* out;
    const int32_t* tile_list; const int32_t* tile_count; const uint32_t* masks;
    int Ho, Wo, Co, Ci, kh, kw, sh, sw, ph, pw, relu, tiles_x, tiles_y;
    int BN, NB, BK, kchunks, stages, a_bytes, b_bytes;
    int nb_off;                   // grouped convolution on clusters: first channel block of the group this launch computes
    int nb_group, c_group;        // grouped convolution: channel blocks and input channels of a group (see group_view); ungrouped: all of them
    int MT, nbuf;                 // tiles per work item (1 or 2, sharing one B tile); TMEM accumulator sets (2, or 1 when MT * BN = 512)
    uint32_t idesc, sbo, layout_type;
    uint32_t tmem_cols;           // TMEM columns this CTA allocates: a power of two >= nbuf * MT * BN (256 at most when two CTAs share an SM)
    int32_t* status;
    unsigned long long wait_ns;   // limit of every device-side wait
    int skip_loads;               // failure-detection tests: the producer issues no copy, so the other roles' waits run out
    // flat tiles (tap-by-tap kernel only): row i of tile t is group t * 16 + i, a group being 8 output pixels of one
    // image row, numbered (stream * Ho + y) * gpr + column group; n_groups_all = S * Ho * gpr.  0: 16 x 8 blocks.
    int flat = 0, gpr = 0, gpt = DC_TILE_H, n_groups_all = 0;         // gpt: groups per tile (dc_layer_rt)
    int flat_rows = 0, flat_images = 0;   // > 0: a flat tile is that many whole rows of the stacked streams, whole images (flat_box)
    int epi_warps = 4;            // epilogue warps of the CTA: 4 (192 threads) or 8 (320 threads)
    int early = 0;                // tile list, count and bitmaps are older than the kernel before this one (dc_lists_settled): read before the wait for it
    int slab_order = 0;           // tap-by-tap kernel: the steps in the column-slab kernels' order (see StepOrder)
    // element-wise add of a later layer done here (k_conv_tc<1, true>): add_out = (this layer's output) + add_in (+ ReLU)
    const __nv_bfloat16* add_in = nullptr; __nv_bfloat16* add_out = nullptr; int add_relu = 0;
    int bias_smem = 0;            // > 0: that many bias values (the launch's NB * BN, from channel block nb_off on) are staged in shared memory behind the control block
};

struct SmemCtl {
    unsigned long long full[kMaxStages], empty[kMaxStages], tmem_full[2], tmem_empty[2];
    unsigned long long a_full[4], a_empty[4];     // halo kernel: ring of input patches
    uint32_t tmem_base;
    volatile int abort_flag;
    unsigned long long wait_ns;
    // epilogue staging: per warp 32 pixels x 64 bytes (32 bf16 channels), rows padded to 80 bytes so
    // 16-byte accesses of neighbouring lanes fall in different banks.  Last member: a launch with four epilogue
    // warps asks for (and touches) the first four only, see ctl_bytes().
    __align__(16) uint8_t stage[8][32 * 80];
};
constexpr int kStageBytes = 32 * 80;
// Shared memory the control block takes with `epi_warps` epilogue warps (4 or 8).
__host__ __device__ constexpr size_t ctl_bytes(int epi_warps) { return sizeof(SmemCtl) - (size_t)(8 - epi_warps) * kStageBytes; }

// Bounded wait.  Returns false (and raises the abort flag + status word) when the limit passes
// or another role has already given up.
__device__ __forceinline__ bool mbar_wait(void* bar, uint32_t parity, SmemCtl* ctl, int32_t* status)
{
    return mbar_wait_at(smem_u32(bar), parity, &ctl->abort_flag, &ctl->wait_ns, status);
}
__device__ __forceinline__ bool mbar_wait_a(uint32_t bar, uint32_t parity, SmemCtl* ctl, int32_t* status)
{
    return mbar_wait_at(bar, parity, &ctl->abort_flag, &ctl->wait_ns, status);
}

// From here on the previous kernel's output is read and this kernel's is written.
__device__ __forceinline__ void enter() { dc_pdl_wait(); dc_pdl_release(); }

// The order in which a layer's products are summed.  Every kernel that a layer could be timed with sums in the same one, so that
// the tuner's choice never shows in an output: two caches of one configuration give the same bits.  Layers that the
// column-slab kernels take: 64 channels at a time, kernel columns, kernel rows (a slab holds one column's pixels for all
// rows), 16 channels.  The others: kernel rows, kernel columns, channels.  (What a cluster sums in parts is decided by sizes
// alone: cluster_rule.)
//
// The loop nest of a tap-by-tap producer: the innermost axis is the longest run in which only the channel, the input row and
// the weights' column move, by constants (the producer is one lane: each nested loop's turn costs it).
struct StepOrder {
    int n0, n1, n2, n3, n3_last;                               // turns of the four axes, n3_last in the last turn of the outermost
    int c0, c1, c3;                                            // what a turn adds to the first channel,
    int x1, x2, y1, y2, y3;                                    // to (kx, ky)
    int w0, w1, w2, w3;                                        // and to the column of the weight matrix (taps, then channels)
    __device__ __forceinline__ explicit StepOrder(const TcArgs& a)
    {
        n0 = 1; c0 = c1 = c3 = 0; x1 = x2 = y1 = y2 = y3 = 0; w0 = 0;
        const int row = a.kw * a.Ci;
        if (!a.slab_order) {                                   // kernel rows, kernel columns, channels
            n1 = a.kh; y1 = 1; w1 = row;
            n2 = a.kw; x2 = 1; w2 = a.Ci;
            n3 = n3_last = a.kchunks; c3 = w3 = a.BK;
        } else if (a.BK == 64) {                               // channels, kernel columns, kernel rows
            n1 = a.kchunks; c1 = w1 = 64;
            n2 = a.kw; x2 = 1; w2 = a.Ci;
            n3 = n3_last = a.kh; y3 = 1; w3 = row;
        } else {                                               // 64 channels, kernel columns, kernel rows, channels
            n0 = (a.Ci + 63) / 64; c0 = w0 = 64;
            n1 = a.kw; x1 = 1; w1 = a.Ci;
            n2 = a.kh; y2 = 1; w2 = row;
            n3 = 64 / a.BK; n3_last = (a.Ci - (n0 - 1) * 64) / a.BK; c3 = w3 = a.BK;
        }
    }
    // step(c, kx, ky, w) for every step until it returns false
    template <typename F>
    __device__ __forceinline__ void walk(F&& step) const
    {
        for (int i0 = 0; i0 < n0; ++i0) {
            const int n = i0 + 1 < n0 ? n3 : n3_last;
            for (int i1 = 0; i1 < n1; ++i1)
                for (int i2 = 0; i2 < n2; ++i2) {
                    const int x = i1 * x1 + i2 * x2;
                    int c = i0 * c0 + i1 * c1, y = i1 * y1 + i2 * y2, w = i0 * w0 + i1 * w1 + i2 * w2;
                    for (int i3 = 0; i3 < n; ++i3, c += c3, y += y3, w += w3)
                        if (!step(c, x, y, w)) return;
                }
        }
    }
};

// Copies the launch's bias values behind the control block (all threads; before the set-up's __syncthreads).  The
// epilogue reads 32 of them per step and lane: from shared memory that is eight short broadcast loads, through the
// read-only cache it was a fifth of the time of the layers that the epilogue bounds.
__device__ __forceinline__ void stage_bias(const TcArgs& a, SmemCtl* ctl, int epi_warps)
{
    float* dst = (float*)((uint8_t*)ctl + ctl_bytes(epi_warps));
    const float* src = a.bias + (size_t)a.nb_off * a.BN;
    for (int i = threadIdx.x; i < a.bias_smem; i += blockDim.x) dst[i] = a.nb_off * a.BN + i < a.Co ? __ldg(src + i) : 0.f;
}

// Epilogue warps (4 warps = 128 TMEM lanes = the 128 pixels of a tile): for every work item wait
// for its accumulator, read it 32 columns at a time, add the bias, apply ReLU, round to bf16 and
// store the pixel's channels unless the reuse bitmap says the pixel was filled from the cache.
// epi_warps = 8: two warps per TMEM lane quadrant (warps 2-5 and 6-9), each taking half of the item's channels:
// layers with little accumulation per output (1x1, few input channels) are bound by this read-out.
// first_item / item_stride: the items this CTA (or CTA pair) takes.  tiles_per_group / tile_sub: a group of the tile list
// holds tiles_per_group tiles and this CTA's first one is number tile_sub in it (a pair: 2 and its rank, with a.MT = 1).
// remote_empty: 0, or the shared::cluster address of the pair leader's tmem_empty[0], on which this CTA's epilogue
// threads arrive instead of on their own.
// ADD: the launch visits every tile, and the add that follows is done in the same pass: reused pixels are read back from the output map, where
// the reuse copy has put them; a step's other operands travel while its accumulator is waited for.
template <bool ADD>
__device__ __forceinline__ void epilogue_loop(const TcArgs& a, SmemCtl* ctl, uint32_t tmem_base, int n_items, int n_tiles, int warp, int lane,
                                              int first_item, int item_stride, int tiles_per_group, int tile_sub, uint32_t remote_empty,
                                              int epi_warps = 4)
{
    // the launch's bias values in shared memory (stage_bias), or 0: read through the read-only cache
    const uint32_t bias_s = a.bias_smem > 0 ? smem_u32((const uint8_t*)ctl + ctl_bytes(epi_warps)) : 0u;
    const int per_stream = a.tiles_x * a.tiles_y;
    const int q = warp & 3;                                     // TMEM lane quadrant this warp may read
    // this warp's 32-column steps of an item: all of them, or the lower / upper half
    const int n_steps = a.BN / 32, mid = epi_warps == 8 ? (n_steps + 1) / 2 : n_steps;
    const int c_begin = warp >= 6 ? mid : 0, c_end = warp >= 6 ? n_steps : mid;
    const int m = q * 32 + lane, prow = m / DC_TILE_W, pcol = m % DC_TILE_W;
    const int mword_i = DC_TILE_BIT(prow, pcol) >> 5, mbit = DC_TILE_BIT(prow, pcol) & 31;
    uint32_t acc = 0, acc_ph = 0;
    bool ok = true;
    // the tile index and this pixel's bitmap word of the NEXT item are fetched while the current one is
    // processed: two dependent global loads would otherwise sit on every item's critical path
    int tile_n0 = -1, tile_n1 = -1; uint32_t mask_n0 = 0, mask_n1 = 0;       // scalars: indexed arrays would live in local memory
    auto fetch = [&](int item) {
        if (item >= n_items) return;
        const int idx = (item / a.NB) * tiles_per_group + tile_sub;
        tile_n0 = idx < n_tiles ? __ldcg(a.tile_list + idx) : -1;                  // a pair's second CTA may have no tile in the last group
        mask_n0 = tile_n0 >= 0 ? __ldcg(a.masks + (size_t)tile_n0 * 4 + mword_i) : 0u;
        tile_n1 = (a.MT > 1 && idx + 1 < n_tiles) ? __ldcg(a.tile_list + idx + 1) : -1;   // odd tile count: the last item has one tile
        mask_n1 = tile_n1 >= 0 ? __ldcg(a.masks + (size_t)tile_n1 * 4 + mword_i) : 0u;
    };
    fetch(first_item);
    if (a.early) enter();
    for (int item = first_item; item < n_items && ok; item += item_stride) {
        const int nb = item % a.NB;
        const int tile_c0 = tile_n0, tile_c1 = tile_n1;
        const uint32_t mask_c0 = mask_n0, mask_c1 = mask_n1;
        fetch(item + item_stride);
        auto wait_full = [&]() -> bool {
            ok = mbar_wait(&ctl->tmem_full[acc], acc_ph, ctl, a.status);
            ok = __all_sync(0xffffffffu, ok);
            if (ok) tc_fence_after();
            return ok;
        };
        const float* bias = a.bias + (nb + a.nb_off) * a.BN;
        for (int j = 0; j < a.MT; ++j) {
            const int tile = j == 0 ? tile_c0 : tile_c1;
            if (tile < 0) { if (j == 0 && !wait_full()) return; break; }        // a pair's second CTA without a tile: its turn all the same
            const bool reused = ((j == 0 ? mask_c0 : mask_c1) >> mbit) & 1u;
            bool active, in_map;
            // write-back addressing, once per tile: piece k of this lane is the 16-byte part (lane & 3) of the pixel in
            // tile row q * 4 + k, column lane >> 2 (the warp's 32 pixels are 4 tile rows of 8)
            const size_t row_stride = (size_t)a.Wo * a.Co;
            const size_t ch_off = (size_t)(nb + a.nb_off) * a.BN + (lane & 3) * 8;
            size_t wb_off[4];                                   // element offset of piece k's pixel
            if (a.flat) {
                const int gps = a.Ho * a.gpr;
                const int g = tile * a.gpt + prow, s = g / gps, loc = g - s * gps, y = loc / a.gpr, gx = loc - y * a.gpr;
                in_map = prow < a.gpt && g < a.n_groups_all && gx * DC_TILE_W + pcol < a.Wo;
                active = in_map && !reused;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int gk = tile * a.gpt + q * 4 + k, sk = gk / gps, lk = gk - sk * gps, yk = lk / a.gpr, xk = lk - yk * a.gpr;
                    wb_off[k] = (((size_t)sk * a.Ho + yk) * a.Wo + xk * DC_TILE_W + (lane >> 2)) * a.Co + ch_off;
                }
            } else {
                const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
                const int oy = ty * DC_TILE_H + prow, ox = tx * DC_TILE_W + pcol;
                in_map = oy < a.Ho && ox < a.Wo;
                active = in_map && !reused;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    wb_off[k] = ((size_t)s * a.Ho + ty * DC_TILE_H + q * 4 + k) * row_stride + (size_t)(tx * DC_TILE_W + (lane >> 2)) * a.Co + ch_off;
            }
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (acc * (uint32_t)a.MT + (uint32_t)j) * (uint32_t)a.BN;
            // Each lane owns one pixel (TMEM lane) and gets 32 channels = 64 bytes per step.  Storing them
            // directly would make every warp store touch 32 different lines 16 bytes at a time (half-written
            // sectors); instead the warp stages its 32 x 64 bytes in shared memory and writes them back with
            // 4 lanes per pixel, so each pixel's 64 bytes leave as two whole sectors.
            const unsigned act_mask = __ballot_sync(0xffffffffu, active), map_mask = ADD ? __ballot_sync(0xffffffffu, in_map) : 0u;
            uint4 other[4], old[4];                              // ADD: the step's other operands, and its reused pixels
            auto fetch_add = [&](int c) {
                if constexpr (ADD) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const unsigned bit = c < c_end ? 1u << ((lane >> 2) + 8 * k) : 0u;
                        if (map_mask & bit) other[k] = *(const uint4*)(a.add_in + wb_off[k] + c * 32);
                        if (map_mask & ~act_mask & bit) old[k] = *(const uint4*)(a.out + wb_off[k] + c * 32);
                    }
                }
            };
            const uint32_t stg = smem_u32(ctl->stage[warp - 2]);
            const uint32_t rd = stg + (lane >> 2) * 80 + (lane & 3) * 16, mine = stg + lane * 80;
            fetch_add(c_begin);
            if (j == 0 && !wait_full()) return;                  // the addresses are worked out while the accumulator is
            for (int c = c_begin; c < c_end; ++c) {
                uint32_t r[32];
                tmem_ld32(taddr + c * 32, r);
                // the step's 32 bias values travel while the accumulator read is in flight
                float4 bv[8];
                if (bias_s) {
                    const uint32_t b4 = bias_s + (uint32_t)(nb * a.BN + c * 32) * 4u;
#pragma unroll
                    for (int v = 0; v < 8; ++v) {
                        const uint4 t = lds128(b4 + v * 16);
                        bv[v] = make_float4(__uint_as_float(t.x), __uint_as_float(t.y), __uint_as_float(t.z), __uint_as_float(t.w));
                    }
                } else {
                    const float4* b4 = (const float4*)(bias + c * 32);
#pragma unroll
                    for (int v = 0; v < 8; ++v) bv[v] = __ldg(b4 + v);
                }
                tmem_ld_wait();
                if (a.relu) {
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        sts128(mine + v * 16, bias_pack_bf16<true>(r[v * 8 + 0], r[v * 8 + 1], bv[2 * v].x, bv[2 * v].y),
                               bias_pack_bf16<true>(r[v * 8 + 2], r[v * 8 + 3], bv[2 * v].z, bv[2 * v].w),
                               bias_pack_bf16<true>(r[v * 8 + 4], r[v * 8 + 5], bv[2 * v + 1].x, bv[2 * v + 1].y),
                               bias_pack_bf16<true>(r[v * 8 + 6], r[v * 8 + 7], bv[2 * v + 1].z, bv[2 * v + 1].w));
                } else {
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        sts128(mine + v * 16, bias_pack_bf16<false>(r[v * 8 + 0], r[v * 8 + 1], bv[2 * v].x, bv[2 * v].y),
                               bias_pack_bf16<false>(r[v * 8 + 2], r[v * 8 + 3], bv[2 * v].z, bv[2 * v].w),
                               bias_pack_bf16<false>(r[v * 8 + 4], r[v * 8 + 5], bv[2 * v + 1].x, bv[2 * v + 1].y),
                               bias_pack_bf16<false>(r[v * 8 + 6], r[v * 8 + 7], bv[2 * v + 1].z, bv[2 * v + 1].w));
                }
                __syncwarp();
                const unsigned store = (int)ch_off + c * 32 < a.Co ? act_mask : 0u;     // (a last block that is filled up)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const unsigned bit = 1u << ((lane >> 2) + 8 * k);
                    if constexpr (!ADD) {
                        if (store & bit) *(uint4*)(a.out + wb_off[k] + c * 32) = lds128(rd + k * (8 * 80));
                    } else if (map_mask & bit) {
                        uint4 o = old[k];
                        if (store & bit) {
                            o = lds128(rd + k * (8 * 80));
                            *(uint4*)(a.out + wb_off[k] + c * 32) = o;
                        }
                        *(uint4*)(a.add_out + wb_off[k] + c * 32) = add_bf16x8(o, other[k], a.add_relu);
                    }
                }
                fetch_add(c + 1);
                __syncwarp();
            }
        }
        tc_fence_before();
        if (remote_empty) mbar_arrive_remote(remote_empty + acc * 8u);
        else mbar_arrive_relaxed(&ctl->tmem_empty[acc]);
        if (++acc == (uint32_t)a.nbuf) { acc = 0; acc_ph ^= 1u; }
    }
}

template <int MT, bool ADD>
__global__ void __launch_bounds__(kThreadsWide, 1)
k_conv_tc(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const TcArgs a)
{
    extern __shared__ uint8_t smem_raw[];

    // operand ring at a 1024-byte boundary (the swizzle pattern repeats every 1024 bytes), then control words
    uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = MT * a.a_bytes + a.b_bytes;
    SmemCtl* ctl = (SmemCtl*)(ring + (size_t)a.stages * stage_bytes);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int per_stream = a.tiles_x * a.tiles_y;
    const int kiters = a.kh * a.kw * a.kchunks;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&ctl->tmem_full[i], 1); mbar_init(&ctl->tmem_empty[i], 32u * (uint32_t)a.epi_warps); }
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    stage_bias(a, ctl, a.epi_warps);
    if (warp == 1) {       // up to 512 columns: two accumulators of up to 256 columns
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (!a.early) enter();      // else each role enters once it has its first tile
    const int n_tiles = __ldcg(a.tile_count);
    const int n_items = (n_tiles + MT - 1) / MT * a.NB;     // an item: MT tiles x one block of BN channels; none for this CTA: it only frees its tensor memory

    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
    if (warp == 0) {
        // ---------------- TMA producer ----------------
        RingPos r;
        r.start(smem_u32(ring), (uint32_t)a.stages);
        const uint32_t r0 = r.data, b_at = (uint32_t)(MT * a.a_bytes);
        const StepOrder order(a);
        bool ok = true;
        int ahead = 0;                                              // steps whose weights are on their way already
        // the weights are nobody's output: those of the first item's first steps travel while the previous kernel ends
        auto weights_ahead = [&](uint32_t tx, int row0) -> int {
            if (a.skip_loads) return 0;
            const int n = min(a.stages, kiters);
            int k = 0;
            order.walk([&](int, int, int, int w) {
                if (k == n) return false;
                mbar_expect_tx(full0 + 8u * k, tx);
                tma_load_2d(r0 + k * stage_bytes + b_at, &tmB, w, row0, full0 + 8u * k);
                ++k;
                return true;
            });
            return n;
        };
        if (a.flat && !a.flat_rows && !a.flat_images) {
            // flat tiles: lane l fetches group (l & 15) of tile (l >> 4), one box of 8 pixels per tap and chunk
            const int j = lane >> 4;
            int next = 0;                                       // this lane's tile of the item to come
            auto peek = [&](int item) {
                const int first = item / a.NB * MT;
                if (item < n_items && j < MT) next = __ldcg(a.tile_list + (first + j < n_tiles ? first + j : first));
            };
            peek(blockIdx.x);
            bool entered = !a.early;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const int row0 = (item % a.NB + a.nb_off) * a.BN, tile = next, c_off = item % a.NB / a.nb_group * a.c_group;
                peek(item + gridDim.x);
                int fs = 0, fx = 0, fy = 0; bool fon = false;
                if (j < MT) {
                    const int gps = a.Ho * a.gpr, g = tile * a.gpt + (lane & 15);
                    fon = (lane & 15) < a.gpt && g < a.n_groups_all;                   // the last tile may have fewer groups: their rows stay as they are (never stored)
                    fs = g / gps;
                    const int loc = g - fs * gps, y = loc / a.gpr;
                    fx = (loc - y * a.gpr) * DC_TILE_W * a.sw - a.pw; fy = y * a.sh - a.ph;
                }
                const uint32_t piece = (uint32_t)(a.a_bytes / DC_TILE_H);
                const uint32_t tx = (uint32_t)__popc(__ballot_sync(0xffffffffu, fon)) * piece + (uint32_t)a.b_bytes;
                if (!entered) {
                    if (elect_one()) ahead = weights_ahead(tx, row0);
                    ahead = __reduce_max_sync(0xffffffffu, ahead);
                    enter();
                    entered = true;
                }
                order.walk([&](int c, int kx, int ky, int w) {
                    ok = __all_sync(0xffffffffu, mbar_wait_a(empty0 + r.off, r.phase ^ 1u, ctl, a.status));
                    if (!ok) return false;
                    if (!a.skip_loads) {
                        if (ahead > 0) --ahead;
                        else if (elect_one()) {
                            mbar_expect_tx(full0 + r.off, tx);
                            tma_load_2d(r.data + b_at, &tmB, w, row0, full0 + r.off);
                        }
                        __syncwarp();                                   // the slot is free and its byte count announced: every lane brings its own group
                        if (fon) tma_load_4d(r.data + lane * piece, &tmA, c + c_off, fx + kx, fy + ky, fs, full0 + r.off);
                    }
                    r.next(r0, (uint32_t)a.stages, (uint32_t)stage_bytes);
                    return true;
                });
            }
            if (!entered) enter();
        } else if (elect_one()) {
            int next[MT];                                           // tiles of the item to come
            auto peek = [&](int item) {
                const int first = item / a.NB * MT;
#pragma unroll
                for (int j = 0; j < MT; ++j)                        // an absent second tile repeats the first (never stored)
                    if (item < n_items) next[j] = __ldcg(a.tile_list + (first + j < n_tiles ? first + j : first));
            };
            peek(blockIdx.x);
            const uint32_t tx = (uint32_t)(MT * a.a_bytes / DC_TILE_H * a.gpt + a.b_bytes);
            int row0 = 0, c_off = 0, sN[MT], xb[MT], yb[MT];
            auto place = [&](int item) {                            // where the item's boxes lie
                if (item >= n_items) return;
                const int nb = item % a.NB;
                row0 = (nb + a.nb_off) * a.BN; c_off = nb / a.nb_group * a.c_group;
#pragma unroll
                for (int j = 0; j < MT; ++j) {
                    const int tile = next[j];
                    const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx_ = t - ty * a.tiles_x;
                    sN[j] = s; xb[j] = tx_ * DC_TILE_W * a.sw - a.pw; yb[j] = ty * DC_TILE_H * a.sh - a.ph;
                    if (a.flat_rows) { sN[j] = xb[j] = 0; yb[j] = tile * a.flat_rows * a.sh; }
                    if (a.flat_images) { sN[j] = tile * a.flat_images; xb[j] = -a.pw; yb[j] = -a.ph; }
                }
            };
            place(blockIdx.x);
            if (a.early) {
                if ((int)blockIdx.x < n_items) ahead = weights_ahead(tx, row0);
                enter();
            }
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                peek(item + gridDim.x);
                order.walk([&](int c, int kx, int ky, int w) {
                    ok = mbar_wait_a(empty0 + r.off, r.phase ^ 1u, ctl, a.status);
                    if (!ok) return false;
                    if (!a.skip_loads) {
                        if (ahead > 0) --ahead;
                        else {
                            mbar_expect_tx(full0 + r.off, tx);
                            tma_load_2d(r.data + b_at, &tmB, w, row0, full0 + r.off);
                        }
#pragma unroll
                        for (int j = 0; j < MT; ++j)
                            tma_load_4d(r.data + j * a.a_bytes, &tmA, c + c_off, xb[j] + kx, yb[j] + ky, sN[j], full0 + r.off);
                    }
                    r.next(r0, (uint32_t)a.stages, (uint32_t)stage_bytes);
                    return true;
                });
                place(item + gridDim.x);
            }
        }
        __syncwarp();
        // on an abort: give the copies already issued a bounded chance to land before the CTA exits
        if (__any_sync(0xffffffffu, !ok)) {
            const unsigned long long t0 = now_ns();
            while (now_ns() - t0 < 2000000ull) { }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (a.early) enter();
        // Descriptors differ from slot to slot in their address bits alone.
        if (elect_one()) {
            const uint64_t dconst = umma_desc(0, a.sbo, a.layout_type);
            const uint32_t d_hi = (uint32_t)(dconst >> 32), r0 = (uint32_t)dconst + (smem_u32(ring) >> 4);
            const uint32_t stage_lo = (uint32_t)stage_bytes >> 4, a_lo = (uint32_t)a.a_bytes >> 4;
            const int ksteps = a.BK / 16;                           // 16 bf16 = 32 bytes = 2 descriptor units
            RingPos r;
            r.start(r0, (uint32_t)a.stages);
            uint32_t acc = 0, acc_ph = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)(MT * a.BN);
                ok = mbar_wait(&ctl->tmem_empty[acc], acc_ph ^ 1u, ctl, a.status);
                tc_fence_after();
                uint32_t accumulate = 0;
                for (int k = 0; k < kiters && ok; ++k) {
                    ok = mbar_wait_a(full0 + r.off, r.phase, ctl, a.status);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int j = 0; j < MT; ++j)
                        umma_chunk(d_tmem + j * a.BN, r.data + j * a_lo, d_hi, 2u, r.data + MT * a_lo, d_hi, 2u, a.idesc, accumulate, ksteps);
                    accumulate = 1;
                    umma_commit_at(empty0 + r.off);                    // frees the slot when these MMAs retire
                    r.next(r0, (uint32_t)a.stages, stage_lo);
                }
                if (ok) umma_commit(&ctl->tmem_full[acc]);
                if (++acc == (uint32_t)a.nbuf) { acc = 0; acc_ph ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ----------------
        epilogue_loop<ADD>(a, ctl, tmem_base, n_items, n_tiles, warp, lane, blockIdx.x, gridDim.x, a.MT, 0, 0u, a.epi_warps);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// Few input channels (cin <= 8, e.g. the first layer on RGB): the channels are padded to 8
// (16 bytes per pixel) and the kernel taps are laid side by side along K: K = taps * 8, padded to
// a multiple of 16.  Operands use the unswizzled core-matrix layout.  ONE TMA box per tile brings the
// (16 + kh - 1) x (8 + kw - 1) input patch as pixels of 16 bytes; the rows of tap (ky, kx) are the
// patch pixels starting at (ky * PW + kx), one patch row (PW x 16 bytes) between 8-row groups, so
// every tap is read in place, and one tcgen05.mma (K = 16) consumes two taps whose pixel offsets
// differ by the descriptor's leading-dimension offset.  The packed weights ([K/8][cout][8]) stay
// in shared memory for the whole kernel.  A whole work item is one pipeline stage.
// ---------------------------------------------------------------------------------------------
struct TcSmallArgs {
    TcArgs t;                     // shared fields (BN = cout, NB = 1)
    const __nv_bfloat16* wpacked; // [kblocks][cout][8]
    int kblocks;                  // K / 8 (even); taps = kh * kw real ones, the rest zero
    int w_bytes;                  // kblocks * cout * 16
    int PW, PH, stage_bytes;      // input patch per tile: (8 + kw - 1) x (16 + kh - 1) pixels of 16 bytes, + pad
};

__global__ void __launch_bounds__(kThreadsWide, 1)
k_conv_tc_smallc(const __grid_constant__ CUtensorMap tmA, const TcSmallArgs sa)
{
    extern __shared__ uint8_t smem_raw[];
    const TcArgs& a = sa.t;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint8_t* wsm = base;                                        // packed weights
    uint8_t* ring = wsm + ((sa.w_bytes + 127) & ~127);
    SmemCtl* ctl = (SmemCtl*)(ring + (size_t)a.stages * sa.stage_bytes);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int per_stream = a.tiles_x * a.tiles_y;
    const int taps = a.kh * a.kw;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&ctl->tmem_full[i], 1); mbar_init(&ctl->tmem_empty[i], 32u * (uint32_t)a.epi_warps); }
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
    }
    // weights into shared memory; zero the ring once: each slot ends in a pad that no TMA box fills but
    // the last (zero-weight) K block reads, and 0 x garbage could be NaN
    for (int i = threadIdx.x; i < sa.w_bytes / 16; i += blockDim.x)
        ((uint4*)wsm)[i] = __ldg((const uint4*)sa.wpacked + i);
    for (int i = threadIdx.x; i < a.stages * sa.stage_bytes / 16; i += blockDim.x)
        ((uint4*)ring)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to TMA / MMA
    stage_bias(a, ctl, a.epi_warps);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (!a.early) enter();      // else each role enters once it has its first tile
    const int n_items = __ldcg(a.tile_count);

    if (warp == 0) {
        if (elect_one()) {                                      // producer: one patch per item
            RingPos r;
            r.start(smem_u32(ring), (uint32_t)a.stages);
            const uint32_t r0 = r.data, full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            bool ok = true;
            int tile_next = __ldcg(a.tile_list + blockIdx.x);   // fetched one item ahead: off the critical path
            if (a.early) enter();
            for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
                const int tile = tile_next;
                if (item + (int)gridDim.x < n_items) tile_next = __ldcg(a.tile_list + item + gridDim.x);
                const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
                ok = mbar_wait_a(empty0 + r.off, r.phase ^ 1u, ctl, a.status);
                if (!ok) break;
                if (!a.skip_loads) {
                    mbar_expect_tx(full0 + r.off, (uint32_t)(sa.PW * sa.PH * 16));
                    tma_load_4d(r.data, &tmA, 0, tx * DC_TILE_W - a.pw, ty * DC_TILE_H - a.ph, s, full0 + r.off);
                }
                r.next(r0, (uint32_t)a.stages, (uint32_t)sa.stage_bytes);
            }
            if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (a.early) enter();
        if (elect_one()) {                                      // MMA issuer
            const uint32_t b_lbo = (uint32_t)a.Co * 16u;
            const uint64_t bconst = umma_desc(smem_u32(wsm), 128, 0, b_lbo);
            const uint64_t hi = umma_desc(0, (uint32_t)sa.PW * 16u, 0, 0);     // SBO = one patch row; LBO added per K step
            RingPos r;
            r.start(smem_u32(ring) >> 4, (uint32_t)a.stages);
            const uint32_t r0 = r.data, stage_lo = (uint32_t)sa.stage_bytes >> 4, full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]);
            uint32_t acc = 0, acc_ph = 0;
            for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
                if (!(mbar_wait(&ctl->tmem_empty[acc], acc_ph ^ 1u, ctl, a.status) && mbar_wait_a(full0 + r.off, r.phase, ctl, a.status))) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)a.BN;
                // K step kk covers taps 2kk and 2kk+1: two 16-byte pixel columns of the patch, `lbo` apart
                int tap = 0, ky = 0, kx = 0;
                for (int kk = 0; kk < sa.kblocks / 2; ++kk) {
                    const uint32_t off0 = (uint32_t)(ky * sa.PW + kx);
                    if (++kx == a.kw) { kx = 0; ++ky; }
                    ++tap;
                    uint32_t off1 = off0 + 1;                      // past the last tap: any finite data (its weights are zero)
                    if (tap < taps) { off1 = (uint32_t)(ky * sa.PW + kx); if (++kx == a.kw) { kx = 0; ++ky; } }
                    ++tap;
                    const uint64_t adesc = hi + (r.data + off0) + ((uint64_t)(off1 - off0) << 16);
                    umma_f16(d_tmem, adesc, bconst + (uint64_t)(kk * ((2 * b_lbo) >> 4)), a.idesc, kk != 0);
                }
                umma_commit_at(empty0 + r.off);
                umma_commit(&ctl->tmem_full[acc]);
                r.next(r0, (uint32_t)a.stages, stage_lo);
                if (++acc == 2u) { acc = 0; acc_ph ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        epilogue_loop<false>(a, ctl, tmem_base, n_items, n_items, warp, lane, blockIdx.x, gridDim.x, 1, 0, 0u, a.epi_warps);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// Input-patch reuse ("halo") variant for stride-1 k x k convolutions with cin a multiple of 16.
// k_conv_tc fetches the 16x8 input window once per kernel tap (9 x 16 KB for 3x3); here the
// (16 + kh - 1) x (8 + kw - 1) patch is fetched ONCE per 64-channel chunk and every tap reads it
// in place.  That needs an operand layout whose rows may start at any patch pixel: the
// unswizzled core-matrix layout with the patch stored as 8 planes (one per 8 channels = 16
// bytes) of [patch row][patch column] pixels.  A tile is 8 pixels wide, so the 8 rows of one
// operand group are the 8 consecutive pixels of one image row, and groups are one patch row
// (PW x 16 bytes) apart: SBO = PW * 16, LBO = plane size, start = plane + (ky * PW + kx) * 16.
// Weights are pre-packed per (channel block, tap, chunk) as the MMA reads them (k_pack_halo) and
// arrive with one plain bulk copy each.
// ---------------------------------------------------------------------------------------------
struct TcHaloArgs {
    TcArgs t;
    const __nv_bfloat16* wpacked;    // [NB][taps][kchunks][BN][64], swizzled (k_pack_halo)
    int PW, PH, plane_bytes, patch_bytes, a_stages;
    int k_last;                      // K steps of 16 channels in the last chunk (4 unless the channels are no multiple of 64)
};

// SLAB = false: the A side of a 64-channel chunk is one (16 + kh - 1) x (8 + kw - 1) patch in eight 16-byte planes
//               (unswizzled core matrices), read in place by every tap.
// SLAB = true:  the A side of a (chunk, kx) pair is one column slab: the (16 + kh - 1) x 8 pixels of the tile's
//               columns displaced by kx, 128 bytes (64 channels) per pixel, 128-byte swizzled.  The eight pixels of
//               a tile row are one 1024-byte swizzle atom, so tap (ky, kx) is the slab from atom ky on: a plain
//               K-major tile.  kw loads of whole 128-byte rows per chunk instead of kh * kw (tap by tap) or eight
//               loads of 16-byte rows (patch).  ha.patch_bytes then holds the bytes of one slab.
template <int MT, bool SLAB>
__global__ void __launch_bounds__(kThreadsWide, 1)
k_conv_tc_halo(const __grid_constant__ CUtensorMap tmA, const TcHaloArgs ha)
{
    extern __shared__ uint8_t smem_raw[];
    const TcArgs& a = ha.t;
    constexpr uintptr_t kAlign = 1023;                        // swizzle atoms start on 1024-byte boundaries
    uint8_t* aring = (uint8_t*)(((uintptr_t)smem_raw + kAlign) & ~kAlign);
    const int a_slot = MT * ha.patch_bytes;
    uint8_t* bring = aring + (size_t)ha.a_stages * a_slot;
    SmemCtl* ctl = (SmemCtl*)(bring + (size_t)a.stages * a.b_bytes);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int per_stream = a.tiles_x * a.tiles_y;
    const int taps = a.kh * a.kw;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&ctl->tmem_full[i], 1); mbar_init(&ctl->tmem_empty[i], 32u * (uint32_t)a.epi_warps); }
        for (int i = 0; i < 4; ++i) { mbar_init(&ctl->a_full[i], 1); mbar_init(&ctl->a_empty[i], 1); }
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
    }
    stage_bias(a, ctl, a.epi_warps);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (!a.early) enter();      // else each role enters once it has its first tile
    const int n_tiles = __ldcg(a.tile_count);
    const int n_items = (n_tiles + MT - 1) / MT * a.NB;

    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), a_full0 = smem_u32(&ctl->a_full[0]), a_empty0 = smem_u32(&ctl->a_empty[0]);
    if (warp == 0) {
        // ---------------- producer: patches by TMA, weights by bulk copy ----------------
        if (elect_one()) {
            RingPos ra, rb;
            ra.start(smem_u32(aring), (uint32_t)ha.a_stages); rb.start(smem_u32(bring), (uint32_t)a.stages);
            const uint32_t a0 = ra.data, b0 = rb.data;
            const size_t tap_stride = (size_t)a.kchunks * a.b_bytes;             // packed weights: one tap further
            bool ok = true;
            int next[MT];                                                        // tiles of the item to come
            auto peek = [&](int item) {
                const int first = item / a.NB * MT;
#pragma unroll
                for (int j = 0; j < MT; ++j)                                     // an absent second tile repeats the first (never stored)
                    if (item < n_items) next[j] = __ldcg(a.tile_list + (first + j < n_tiles ? first + j : first));
            };
            peek(blockIdx.x);
            int ahead = 0;                                                       // weight tiles on their way already
            if (a.early) {
                // the weights are nobody's output: the first item's first tiles travel while the previous kernel ends
                if ((int)blockIdx.x < n_items && !a.skip_loads) {
                    const uint8_t* w = (const uint8_t*)ha.wpacked + (size_t)((int)blockIdx.x % a.NB + a.nb_off) * taps * tap_stride;
                    const int n = min(a.stages, a.kchunks * taps);
                    for (int cc = 0, kx = 0, ky = 0; ahead < n; ++ahead) {
                        mbar_expect_tx(full0 + 8u * ahead, (uint32_t)a.b_bytes);
                        bulk_copy(b0 + ahead * a.b_bytes, w + (ky * a.kw + kx) * tap_stride + (size_t)cc * a.b_bytes, (uint32_t)a.b_bytes, full0 + 8u * ahead);
                        if (++ky == a.kh) { ky = 0; if (++kx == a.kw) { kx = 0; ++cc; } }
                    }
                }
                enter();
            }
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const int nb = item % a.NB, c_off = nb / a.nb_group * a.c_group;
                int sN[MT], xb[MT], yb[MT];
#pragma unroll
                for (int j = 0; j < MT; ++j) {
                    const int tile = next[j];
                    const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
                    sN[j] = s; xb[j] = tx * DC_TILE_W - a.pw; yb[j] = ty * DC_TILE_H - a.ph;
                }
                peek(item + gridDim.x);
                const uint8_t* w_item = (const uint8_t*)ha.wpacked + (size_t)(nb + a.nb_off) * taps * tap_stride;
                for (int cc = 0; cc < a.kchunks && ok; ++cc) {
                    for (int kx = 0; kx < (SLAB ? a.kw : 1) && ok; ++kx) {
                        ok = mbar_wait_a(a_empty0 + ra.off, ra.phase ^ 1u, ctl, a.status);
                        if (!ok) break;
                        if (!a.skip_loads) {
                            if (SLAB) {
                                mbar_expect_tx(a_full0 + ra.off, (uint32_t)(MT * ha.patch_bytes));
#pragma unroll
                                for (int j = 0; j < MT; ++j)
                                    tma_load_4d(ra.data + j * ha.patch_bytes, &tmA, c_off + cc * 64, xb[j] + kx, yb[j], sN[j], a_full0 + ra.off);
                            } else {
                                mbar_expect_tx(a_full0 + ra.off, (uint32_t)(MT * 8 * ha.PW * ha.PH * 16));
#pragma unroll
                                for (int j = 0; j < MT; ++j)
                                    for (int g = 0; g < 8; ++g)
                                        tma_load_4d(ra.data + j * ha.patch_bytes + g * ha.plane_bytes, &tmA, c_off + cc * 64 + g * 8, xb[j], yb[j], sN[j], a_full0 + ra.off);
                            }
                        }
                        ra.next(a0, (uint32_t)ha.a_stages, (uint32_t)a_slot);
                        // the weight tiles that go with this A stage: all taps, column by column (patch), or the taps of column kx (slab)
                        const uint8_t* w = w_item + kx * tap_stride + (size_t)cc * a.b_bytes;
                        const size_t w_step = a.kw * tap_stride;
                        const int n_t = SLAB ? a.kh : taps;
                        for (int t = 0, ky = 0; t < n_t; ++t) {
                            // a tile sent ahead: its slot was free, and may have been used and freed again by now (no wait for it)
                            if (ahead > 0) --ahead;
                            else {
                                ok = mbar_wait_a(empty0 + rb.off, rb.phase ^ 1u, ctl, a.status);
                                if (!ok) break;
                                if (!a.skip_loads) {
                                    mbar_expect_tx(full0 + rb.off, (uint32_t)a.b_bytes);
                                    bulk_copy(rb.data, w, (uint32_t)a.b_bytes, full0 + rb.off);
                                }
                            }
                            w += w_step;
                            if (!SLAB && ++ky == a.kh) { ky = 0; w -= a.kh * w_step - tap_stride; }      // the next column's first row
                            rb.next(b0, (uint32_t)a.stages, (uint32_t)a.b_bytes);
                        }
                    }
                }
            }
            if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (a.early) enter();
        if (elect_one()) {
            // A: patch planes (rows PW * 16 bytes apart, planes along K), or a 128-byte swizzled K-major slab; weights: 128-byte
            // swizzled, K-major.  Descriptors differ from slot to slot in their lower halves alone.
            const uint64_t aconst = SLAB ? umma_desc(0, 1024, 2) : umma_desc(0, (uint32_t)ha.PW * 16u, 0, (uint32_t)ha.plane_bytes);
            const uint64_t bconst = umma_desc(0, 1024, 2);
            const uint32_t a_hi = (uint32_t)(aconst >> 32), b_hi = (uint32_t)(bconst >> 32);
            const uint32_t a0 = (uint32_t)aconst + (smem_u32(aring) >> 4), b0 = (uint32_t)bconst + (smem_u32(bring) >> 4);
            const uint32_t a_slot_lo = (uint32_t)a_slot >> 4, patch_lo = (uint32_t)ha.patch_bytes >> 4, b_lo = (uint32_t)a.b_bytes >> 4;
            const uint32_t a_kstep = SLAB ? 2u : (uint32_t)(2 * ha.plane_bytes) >> 4;    // 16 channels further along K
            RingPos ra, rb;
            ra.start(a0, (uint32_t)ha.a_stages); rb.start(b0, (uint32_t)a.stages);
            uint32_t acc = 0, acc_ph = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)(MT * a.BN);
                ok = mbar_wait(&ctl->tmem_empty[acc], acc_ph ^ 1u, ctl, a.status);
                tc_fence_after();
                uint32_t accumulate = 0;
                for (int cc = 0; cc < a.kchunks && ok; ++cc) {
                    const int n_kk = cc + 1 < a.kchunks ? 4 : ha.k_last;
                    for (int ax = 0; ax < (SLAB ? a.kw : 1) && ok; ++ax) {     // A stages of this chunk: one patch, or kw slabs
                        ok = mbar_wait_a(a_full0 + ra.off, ra.phase, ctl, a.status);
                        // patch: taps column by column at (ky * PW + kx) * 16 bytes; slab ax: taps (ky, ax) at ky atoms of 1024 bytes
                        uint32_t at = ra.data;
                        int ky = 0;
                        const int n_t = SLAB ? a.kh : taps;
                        for (int t = 0; t < n_t && ok; ++t) {
                            ok = mbar_wait_a(full0 + rb.off, rb.phase, ctl, a.status);
                            if (!ok) break;
                            tc_fence_after();
#pragma unroll
                            for (int j = 0; j < MT; ++j)
                                umma_chunk(d_tmem + j * a.BN, at + j * patch_lo, a_hi, a_kstep, rb.data, b_hi, 2u, a.idesc, accumulate, n_kk);
                            accumulate = 1;
                            umma_commit_at(empty0 + rb.off);
                            rb.next(b0, (uint32_t)a.stages, b_lo);
                            if (SLAB) at += 64u;
                            else if (++ky == a.kh) { ky = 0; at += 1u - (uint32_t)((a.kh - 1) * ha.PW); } else at += (uint32_t)ha.PW;
                        }
                        if (ok) umma_commit_at(a_empty0 + ra.off);             // the A stage is free once its taps retire
                        ra.next(a0, (uint32_t)ha.a_stages, a_slot_lo);
                    }
                }
                if (ok) umma_commit(&ctl->tmem_full[acc]);
                if (++acc == (uint32_t)a.nbuf) { acc = 0; acc_ph ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        epilogue_loop<false>(a, ctl, tmem_base, n_items, n_tiles, warp, lane, blockIdx.x, gridDim.x, a.MT, 0, 0u, a.epi_warps);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
}

// ---------------------------------------------------------------------------------------------
// CTA pairs (tcgen05.mma.cta_group::2): the column-slab scheme with one 256-row tile pair per work item.
// Wide layers are bound by their weights: per 64-channel chunk a tile needs 54 KB of input slabs but 288 KB of
// weights at 256 output channels.  Here the two CTAs of a cluster (two SMs of one TPC) take one tile each and HALF of
// the item's output channels' weights each; one MMA instruction, issued by the leader (rank 0), reads both CTAs'
// operands (M = 256: 128 rows from each CTA's slab; N = BN: BN / 2 columns from each CTA's weight tile) and
// accumulates into both CTAs' tensor memory (each holds its own tile's 128 rows x BN columns).  Per tile the weight
// traffic into an SM halves, and the accumulators stay double buffered (2 x BN <= 512 columns per CTA).
//
// Every load is a plain per-CTA TMA load into the CTA's own shared memory (no multicast anywhere); the loads of the
// second CTA report their bytes to the leader's barrier (cta_group::2 form of the load), because the leader's MMA
// thread is the only consumer.  Barriers: full / a_full / tmem_empty live in the leader and collect both CTAs;
// empty / a_empty / tmem_full exist in each CTA and are signalled in both by the leader's tcgen05.commit.
// ---------------------------------------------------------------------------------------------
// loads into this CTA's shared memory whose bytes are counted on the barrier at shared::cluster address `bar` (the leader's)
__device__ __forceinline__ void tma_load_4d_pair(uint32_t dst, const CUtensorMap* tm, int c0, int c1, int c2, int c3, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                 ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int c0, int c1, uint32_t bar)
{
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
// arrives, once the MMAs issued so far have retired, on the barrier at this offset in both CTAs of the pair
__device__ __forceinline__ void umma_commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}

// ha.t.BN: output channels per item (both CTAs together); ha.t.b_bytes: one CTA's weight tile (BN / 2 rows of 128 bytes);
// tmW: the packed weights [2 NB][taps][kchunks][BN / 2][64] seen as rows of 128 bytes.
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_conv_tc_pair(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmW, const TcHaloArgs ha)
{
    extern __shared__ uint8_t smem_raw[];
    const TcArgs& a = ha.t;
    const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
    const uint32_t rank = cluster_rank();
    const bool leader = rank == 0;
    uint8_t* aring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int a_slot = ha.patch_bytes;                        // one slab
    uint8_t* bring = aring + (size_t)ha.a_stages * a_slot;
    SmemCtl* ctl = (SmemCtl*)(bring + (size_t)a.stages * a.b_bytes);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int per_stream = a.tiles_x * a.tiles_y;
    const int taps = a.kh * a.kw;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&ctl->tmem_full[i], 1); mbar_init(&ctl->tmem_empty[i], 256); }
        for (int i = 0; i < 4; ++i) { mbar_init(&ctl->a_full[i], 1); mbar_init(&ctl->a_empty[i], 1); }
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmW) : "memory");
    }
    stage_bias(a, ctl, 4);
    if (warp == 1) {                                          // the same warp in both CTAs: tensor memory of the pair
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                       // both CTAs' barriers exist before either is signalled from outside
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (!a.early) enter();      // else each role enters once it has its first tile
    const int n_tiles = __ldcg(a.tile_count);
    const int n_items = (n_tiles + 1) / 2 * a.NB;

    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), a_full0 = smem_u32(&ctl->a_full[0]), a_empty0 = smem_u32(&ctl->a_empty[0]);
    if (warp == 0) {
        // ---------------- producer: this CTA's slab and its half of the weights ----------------
        if (elect_one()) {
            const uint32_t lead_a_full = map_to_cta(&ctl->a_full[0], 0), lead_full = map_to_cta(&ctl->full[0], 0);   // the leader's barriers
            RingPos ra, rb;
            ra.start(smem_u32(aring), (uint32_t)ha.a_stages); rb.start(smem_u32(bring), (uint32_t)a.stages);
            const uint32_t a0 = ra.data, b0 = rb.data;
            const int rows_per_tile = a.b_bytes >> 7;             // weight rows of 128 bytes in one CTA's tile
            bool ok = true;
            int next = 0;                                         // the tile of the item to come
            auto peek = [&](int item) {
                const int first = item / a.NB * 2, idx = first + (int)rank;
                if (item < n_items) next = __ldcg(a.tile_list + (idx < n_tiles ? idx : first));   // an absent second tile repeats the first (never stored)
            };
            peek(pair);
            if (a.early) enter();
            for (int item = pair; item < n_items && ok; item += n_pairs) {
                const int nb = item % a.NB, tile = next;
                peek(item + n_pairs);
                const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
                const int xb = tx * DC_TILE_W - a.pw, yb = ty * DC_TILE_H - a.ph;
                const int row_step = a.kw * a.kchunks * rows_per_tile;              // packed weights: one kernel row further
                for (int cc = 0; cc < a.kchunks && ok; ++cc) {
                    for (int kx = 0; kx < a.kw && ok; ++kx) {
                        ok = mbar_wait_a(a_empty0 + ra.off, ra.phase ^ 1u, ctl, a.status);
                        if (!ok) break;
                        if (!a.skip_loads) {
                            if (leader) mbar_expect_tx(a_full0 + ra.off, (uint32_t)(2 * ha.patch_bytes));
                            tma_load_4d_pair(ra.data, &tmA, cc * 64, xb + kx, yb, s, lead_a_full + ra.off);
                        }
                        ra.next(a0, (uint32_t)ha.a_stages, (uint32_t)a_slot);
                        int row = (((nb * 2 + (int)rank) * taps + kx) * a.kchunks + cc) * rows_per_tile;
                        for (int t2 = 0; t2 < a.kh; ++t2, row += row_step) {
                            ok = mbar_wait_a(empty0 + rb.off, rb.phase ^ 1u, ctl, a.status);
                            if (!ok) break;
                            if (!a.skip_loads) {
                                if (leader) mbar_expect_tx(full0 + rb.off, (uint32_t)(2 * a.b_bytes));
                                tma_load_2d_pair(rb.data, &tmW, 0, row, lead_full + rb.off);
                            }
                            rb.next(b0, (uint32_t)a.stages, (uint32_t)a.b_bytes);
                        }
                    }
                }
            }
            if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer: an elected lane of the leader issues for both CTAs ----------------
        if (a.early) enter();
        if (leader && elect_one()) {
            const uint64_t dconst = umma_desc(0, 1024, 2);            // slabs and weights: 128-byte swizzled, K-major
            const uint32_t d_hi = (uint32_t)(dconst >> 32), a0 = (uint32_t)dconst + (smem_u32(aring) >> 4), b0 = (uint32_t)dconst + (smem_u32(bring) >> 4);
            const uint32_t a_slot_lo = (uint32_t)a_slot >> 4, b_lo = (uint32_t)a.b_bytes >> 4;
            RingPos ra, rb;
            ra.start(a0, (uint32_t)ha.a_stages); rb.start(b0, (uint32_t)a.stages);
            uint32_t acc = 0, acc_ph = 0;
            bool ok = true;
            for (int item = pair; item < n_items && ok; item += n_pairs) {
                const uint32_t d_tmem = tmem_base + acc * (uint32_t)a.BN;
                ok = mbar_wait(&ctl->tmem_empty[acc], acc_ph ^ 1u, ctl, a.status);
                tc_fence_after();
                uint32_t accumulate = 0;
                for (int cc = 0; cc < a.kchunks && ok; ++cc) {
                    const int n_kk = cc + 1 < a.kchunks ? 4 : ha.k_last;
                    for (int ax = 0; ax < a.kw && ok; ++ax) {
                        ok = mbar_wait_a(a_full0 + ra.off, ra.phase, ctl, a.status);
                        for (int t = 0; t < a.kh && ok; ++t) {               // tap (t, ax): the slab from swizzle atom t on
                            ok = mbar_wait_a(full0 + rb.off, rb.phase, ctl, a.status);
                            if (!ok) break;
                            tc_fence_after();
                            umma_chunk_pair(d_tmem, ra.data + (uint32_t)t * 64u, d_hi, 2u, rb.data, d_hi, 2u, a.idesc, accumulate, n_kk);
                            accumulate = 1;
                            umma_commit_pair(empty0 + rb.off);
                            rb.next(b0, (uint32_t)a.stages, b_lo);
                        }
                        if (ok) umma_commit_pair(a_empty0 + ra.off);
                        ra.next(a0, (uint32_t)ha.a_stages, a_slot_lo);
                    }
                }
                if (ok) umma_commit_pair(smem_u32(&ctl->tmem_full[acc]));
                if (++acc == 2u) { acc = 0; acc_ph ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: this CTA's tile; the accumulator is handed back on the leader's barrier ----------------
        const uint32_t remote_empty = map_to_cta(&ctl->tmem_empty[0], 0);
        epilogue_loop<false>(a, ctl, tmem_base, n_items, n_tiles, warp, lane, pair, n_pairs, 2, (int)rank, remote_empty);
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync_all();                                       // neither CTA frees tensor memory or leaves while the other may still use it
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
}

// weights [cout][taps][cin] -> [NB][taps][kchunks] tiles of BN rows (output channels) x 64 channels, zeros beyond the last
// channel.  A tile lies in memory as the MMA reads it from shared memory, K-major with 128-byte swizzle: the 16-byte piece
// k8 of row n is at piece k8 ^ (n & 7) of that row, so that a plain bulk copy brings it in place.  (Unswizzled core
// matrices, the layout before, cost the MMAs shared-memory time.)
// rows: output channels filled up to whole blocks.
__global__ void k_pack_halo(const __nv_bfloat16* w, int cout, int rows, int taps, int cin, int BN, __nv_bfloat16* out)
{
    const int kchunks = (cin + 63) / 64;
    const size_t total = (size_t)rows * taps * kchunks * 64;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i;
        const int e = (int)(r & 7); r >>= 3;
        const int piece = (int)(r & 7); r >>= 3;
        const int n = (int)(r % BN); r /= BN;
        const int cc = (int)(r % kchunks); r /= kchunks;
        const int tap = (int)(r % taps); const int nb = (int)(r / taps);
        const int ch = cc * 64 + (piece ^ (n & 7)) * 8 + e;
        out[i] = ch < cin && nb * BN + n < cout ? w[((size_t)(nb * BN + n) * taps + tap) * cin + ch] : __float2bfloat16(0.f);
    }
}

// [S][H][W][C] -> [S][H][W][8] with zero padding, C <= 8
__global__ void k_pad_channels8(const __nv_bfloat16* in, size_t pixels, int C, __nv_bfloat16* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < pixels; i += (size_t)gridDim.x * blockDim.x) {
        unsigned short v[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const unsigned short* p = (const unsigned short*)in + i * C;
        for (int c = 0; c < C; ++c) v[c] = p[c];
        ((uint4*)out)[i] = make_uint4(v[0] | ((uint32_t)v[1] << 16), v[2] | ((uint32_t)v[3] << 16),
                                      v[4] | ((uint32_t)v[5] << 16), v[6] | ((uint32_t)v[7] << 16));
    }
}

// [S][H][W][C] -> [S][H][W][16] with zero padding, C < 16
__global__ void k_pad_channels16(const __nv_bfloat16* in, size_t pixels, int C, __nv_bfloat16* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < pixels; i += (size_t)gridDim.x * blockDim.x) {
        unsigned short v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = 0;
        const unsigned short* p = (const unsigned short*)in + i * C;
        for (int c = 0; c < C; ++c) v[c] = p[c];
        ((uint4*)out)[2 * i] = make_uint4(v[0] | ((uint32_t)v[1] << 16), v[2] | ((uint32_t)v[3] << 16),
                                          v[4] | ((uint32_t)v[5] << 16), v[6] | ((uint32_t)v[7] << 16));
        ((uint4*)out)[2 * i + 1] = make_uint4(v[8] | ((uint32_t)v[9] << 16), v[10] | ((uint32_t)v[11] << 16),
                                              v[12] | ((uint32_t)v[13] << 16), v[14] | ((uint32_t)v[15] << 16));
    }
}

// weights [cout][taps][cin] -> [cout][taps][16], channels beyond cin zero
__global__ void k_pack_pad16(const __nv_bfloat16* w, size_t cout_taps, int cin, __nv_bfloat16* out)
{
    const size_t total = cout_taps * 16;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t ct = i >> 4; const int ch = (int)(i & 15);
        out[i] = ch < cin ? w[ct * cin + ch] : __float2bfloat16(0.f);
    }
}

// weights [cout][taps][cin] -> [kblocks][cout][8]: block j holds tap j (cin real channels, rest zero)
__global__ void k_pack_smallc(const __nv_bfloat16* w, int cout, int taps, int cin, int kblocks, __nv_bfloat16* out)
{
    const int total = kblocks * cout * 8;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const int e = i & 7, n = (i >> 3) % cout, j = (i >> 3) / cout;
        out[i] = (j < taps && e < cin) ? w[((size_t)n * taps + j) * cin + e] : __float2bfloat16_rn(0.f);
    }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (EncodeTiledFn)p;
        cudaGetLastError();
    }
    return fn;
}

// Tensor maps are encoded once per (base address, operand scheme, channel block) and kept with the layer: in steady
// state a launch finds its maps in these slots.  A new base or scheme (the tuner's trials, a caller's own buffers in
// dc_conv_partial) replaces a slot.
static_assert(sizeof(CUtensorMap) == 128, "dc_tm_slot stores a CUtensorMap");
static CUtensorMap* tm_find(dc_tm_slot* slots, int n, int* next, const void* base, int code, int bn, bool* hit)
{
    for (int i = 0; i < n; ++i)
        if (slots[i].valid && slots[i].base == base && slots[i].code == code && slots[i].bn == bn) {
            *hit = true;
            return (CUtensorMap*)slots[i].map;
        }
    int k = 0;
    if (n > 1) { k = *next % n; *next = (k + 1) % n; }
    slots[k].valid = true; slots[k].base = base; slots[k].code = code; slots[k].bn = bn;
    *hit = false;
    return (CUtensorMap*)slots[k].map;
}
static void tm_drop(dc_tm_slot* slots, int n, const CUtensorMap* m)
{
    for (int i = 0; i < n; ++i) if ((const CUtensorMap*)slots[i].map == m) slots[i].valid = false;
}

// Two CTAs may share an SM when each needs at most 256 TMEM columns; each then gets half the operand-ring budget.
// Layers with few output channels or a short K are bound by the epilogue (TMEM -> registers -> global), and a
// second resident CTA doubles the epilogue warps per SM.
static uint32_t tmem_cols_for(int nbuf, int mt, int bn)
{
    uint32_t need = (uint32_t)(nbuf * mt * bn), cols = 32;
    while (cols < need) cols <<= 1;
    return cols;
}
// Operand-ring bytes of a CTA that has its SM alone: 200 KB, or 182 KB while the cache's matcher runs beside the
// inference (dc_lookahead_frame): with 182 KB a convolution CTA leaves room for one CTA of the block search (32 KB) on
// its SM, which then works in the tensor-core kernel's idle issue slots instead of waiting for a free SM.  Set per
// launch from the cache's state.
static thread_local int t_ring_kb = 200;
static thread_local int t_epi_warps = 4;      // the layer's tuned epilogue width, honoured by launches with one CTA per SM
static int epi_warps_for(int ctas) { return t_epi_warps == 8 && ctas != 2 ? 8 : 4; }
static thread_local int t_bias_bytes = 0;     // the launch's bias values staged in shared memory (0: too many, read from global memory)
static int bias_bytes_for(const dc_layer_desc& group) { return group.cout * 4 <= 16384 ? (group.cout * 4 + 15) & ~15 : 0; }
// eight epilogue warps stage twice as much, and every CTA keeps its bias values: the rings give that up
static int ring_budget(int ctas)
{
    const int n = ctas == 2 ? 2 : 1;
    return (t_ring_kb * 1024 - (epi_warps_for(ctas) == 8 ? 4 * kStageBytes : 0) - n * t_bias_bytes) / n;
}

// Every launch waits at most kWaitLimitNs on the device.  dc_debug_stall_next_conv (below) arms the next launch
// only: its producer issues no copy and its waits run out after the given time.
static void set_wait_limit(dc_cache* c, TcArgs& a)
{
    a.wait_ns = kWaitLimitNs; a.skip_loads = 0;
    if (c->debug_stall_ms > 0) {
        a.wait_ns = (unsigned long long)c->debug_stall_ms * 1000000ull;
        a.skip_loads = 1;
        c->debug_stall_ms = 0;
    }
}

// A grouped convolution (AlexNet's layers 2, 4, 5) is `groups` independent convolutions, each from its own slice of
// the input channels to its own slice of the output channels.  One launch does them all: a block of output channels belongs to one
// group, and the producer takes its pixels from that group's first channel on (c_group).  The weights [cout][kh][kw][cin / groups] need
// no slicing.  A chunk that reaches beyond the group's last channel brings the next group's, which no MMA reads (whole steps of
// 16 channels).  AlexNet grouped, 96 streams: with a launch per group, each with a last round of its own, 363 us a pass, 342 so.  On clusters, for few
// tiles, a launch per group (nb_off).  This is the layer as one group sees it.
static int n_groups(const dc_layer_desc& d) { return d.groups > 1 ? d.groups : 1; }
// Output channels come in blocks of 32.  An ungrouped layer whose channels do not is seen with them filled up (weight rows beyond the last
// are zeros, by the loads or by k_pack_halo; the epilogue stores what exists): 32 -> 16 channels at 64 x 80, 16 streams, 27 us on
// the CUDA cores, 7 here; the error against 64-bit sums is the same, 1.6485e-3, nearly all of it the rounding to bf16.  Single
// output pixels stay with k_dense, and with more than 4096 channels the bias is not staged.
static dc_layer_desc group_view(const dc_layer_desc& d)
{
    dc_layer_desc g = d;
    g.cin = d.cin / n_groups(d); g.cout = d.cout / n_groups(d); g.groups = 1;
    if (n_groups(d) == 1 && d.cout % 32 != 0 && d.cout % 8 == 0 && d.cout <= 4096 && d.out_h * d.out_w > 1) g.cout = dc_div_up(d.cout, 32) * 32;
    return g;
}

// The output channels of a launch: all groups'.
static dc_layer_desc all_groups(const dc_layer_desc& d)
{
    dc_layer_desc g = group_view(d);
    g.cout *= n_groups(d);
    return g;
}

// Elements from one input pixel, and one input row, to the next.  A block map whose kernel columns were merged into channels
// (dc_conv_s2d.cu) has windows of several pixels as its pixels: they overlap.
struct InPitch { cuuint64_t px, row; };
static InPitch in_pitch(const dc_layer_rt& L, int cin)
{
    InPitch p = {(cuuint64_t)cin, (cuuint64_t)L.in_w * cin};
    if (L.s2d_s) { p.px = (cuuint64_t)L.s2d_cs; p.row = (cuuint64_t)L.s2d_ws * L.s2d_cs; }
    return p;
}

struct TcPlan { int BK, BN, NB, MT, nbuf, stages, a_bytes, b_bytes; CUtensorMapSwizzle swz; uint32_t layout_type, sbo; size_t smem; };

bool make_plan(const dc_layer_desc& d, TcPlan& p, int want_mt = 0, int want_bn = 0, int ctas = 1)
{
    if (d.kind != DC_CONV) return false;
    if (d.sh < 1 || d.sw < 1 || DC_TILE_W * d.sw > 256 || DC_TILE_H * d.sh > 256) return false;   // TMA box limit
    if (d.cin % 64 == 0) { p.BK = 64; p.swz = CU_TENSOR_MAP_SWIZZLE_128B; p.layout_type = 2; }
    else if (d.cin % 32 == 0) { p.BK = 32; p.swz = CU_TENSOR_MAP_SWIZZLE_64B; p.layout_type = 4; }
    else if (d.cin % 16 == 0) { p.BK = 16; p.swz = CU_TENSOR_MAP_SWIZZLE_32B; p.layout_type = 6; }
    else return false;
    p.BN = 0;
    for (int bn = 256; bn >= 32; bn -= 32) if (d.cout % bn == 0) { p.BN = bn; break; }
    if (!p.BN) return false;
    if (want_bn > 0) {                                           // a tuned choice: must divide cout like the default
        if (want_bn % 32 != 0 || want_bn > 256 || d.cout % want_bn != 0) return false;
        p.BN = want_bn;
    }
    p.NB = d.cout / p.BN;
    p.a_bytes = DC_TILE_PX * p.BK * 2;
    p.b_bytes = p.BN * p.BK * 2;
    p.sbo = 8 * p.BK * 2;
    if (p.b_bytes % 1024 != 0) return false;                    // keep every operand tile on a swizzle-pattern boundary
    // two tiles share each B tile: halves the weight traffic per FLOP; 512 TMEM columns hold
    // MT * BN * nbuf accumulator columns
    p.MT = want_mt > 0 ? want_mt : 1;
    p.nbuf = p.MT * p.BN * 2 <= 512 ? 2 : 1;
    if (ctas == 2 && tmem_cols_for(p.nbuf, p.MT, p.BN) > 256) return false;
    int st = ring_budget(ctas) / (p.MT * p.a_bytes + p.b_bytes);
    p.stages = st > kMaxStages ? kMaxStages : st;
    if (p.stages < 2) return false;
    p.smem = (size_t)p.stages * (p.MT * p.a_bytes + p.b_bytes) + ctl_bytes(epi_warps_for(ctas)) + t_bias_bytes + 1024;
    return true;
}

// Channels that are no multiple of 64 (AlexNet's 96, or 48 per group): the last chunk's missing channels are zero-filled by
// the loads, the packed weights have zeros there, and the chunk's K steps without a channel are left out.
struct HaloPlan { int BN, NB, PW, PH, plane_bytes, patch_bytes, b_bytes, kchunks, k_last; };

bool halo_ok(const dc_layer_desc& d, HaloPlan& h, int want_bn = 0)
{
    if (d.kind != DC_CONV || d.sh != 1 || d.sw != 1 || d.cin % 16 != 0 || d.kh * d.kw < 2 || d.kh > 5 || d.kw > 5) return false;
    h.BN = 0;
    for (int bn = 256; bn >= 32; bn -= 32) if (d.cout % bn == 0) { h.BN = bn; break; }
    if (!h.BN) return false;
    if (want_bn > 0) {                                           // a tuned choice: must divide cout like the default
        if (want_bn % 32 != 0 || want_bn > 256 || d.cout % want_bn != 0) return false;
        h.BN = want_bn;
    }
    h.NB = d.cout / h.BN;
    h.PW = DC_TILE_W + d.kw - 1; h.PH = DC_TILE_H + d.kh - 1;
    h.plane_bytes = (h.PW * h.PH * 16 + 127) & ~127;       // TMA destinations are 128-byte aligned
    h.patch_bytes = 8 * h.plane_bytes;
    h.b_bytes = h.BN * 128;
    h.kchunks = (d.cin + 63) / 64; h.k_last = (d.cin - (h.kchunks - 1) * 64 + 15) / 16;
    return true;
}

bool smallc_ok(const dc_layer_desc& d)
{
    return d.kind == DC_CONV && d.sh == 1 && d.sw == 1 && d.cin <= 8 && d.cout % 32 == 0 && d.cout <= 256 &&
           d.kh * d.kw <= 64;
}

// Few input channels with a stride or a large kernel (e.g. 11 x 11 stride 4 on RGB): the channels are padded
// to 16 and the layer runs on the tap-by-tap kernel as a 16-channel convolution (K = taps x 16; the padded
// products are zeros).  Far more tensor work than needed, still many times faster than the CUDA-core kernel.
dc_layer_desc padded16(const dc_layer_desc& d) { dc_layer_desc e = d; e.cin = 16; return e; }
bool pad16_ok(const dc_layer_desc& d)
{
    TcPlan p;
    return d.kind == DC_CONV && d.cin < 16 && !make_plan(d, p) && !smallc_ok(d) && make_plan(padded16(d), p);
}

}  // namespace

int dc_conv_bf16_supported(const dc_cache* c, int layer)
{
    TcPlan p;
    if (getenv("DC_NO_TENSOR_CORES")) return 0;
    if (c->cfg.dtype != DC_BF16 || encode_fn() == nullptr) return 0;
    if (n_groups(c->L[layer].d) > 1) {                            // per group: the tap-by-tap kernel or the patch / slab kernels
        const dc_layer_desc g = group_view(c->L[layer].d);
        return make_plan(g, p) && (g.cin * 2) % 16 == 0;          // a group's first channel must be 16-byte aligned for its tensor map
    }
    return make_plan(group_view(c->L[layer].d), p) || smallc_ok(c->L[layer].d) || pad16_ok(c->L[layer].d);
}

// The first convolution of a bfloat16 cache reads a rearranged copy of its input: the block map (strided layers) or the
// pixels with their channels padded to eight (few-channel kernel).
bool dc_conv_takes_frame(const dc_cache* c, int layer)
{
    const dc_layer_rt& L = c->L[layer];
    TcPlan p;
    if (c->cfg.dtype != DC_BF16 || L.d.kind != DC_CONV || !dc_conv_bf16_supported(c, layer)) return false;
    return L.s2d_s ? L.s2d_cin == 3 : n_groups(L.d) == 1 && L.d.cin == 3 && smallc_ok(L.d) && !make_plan(L.d, p) && L.in_padded != nullptr;
}

// The weights of the patch, slab and pair kernels are packed by channel blocks, so another block width needs another packing
// (of the same size).  Happens while the tuner tries widths, and once more for its final choice before the cache is ready; a
// launch that finds the packing changed under it (`changed`) must not read the weights ahead of its turn.
static int pack_halo(dc_cache* c, dc_layer_rt& L, int bn, bool* changed)
{
    *changed = L.halo_bn != bn;
    if (!*changed) return DC_OK;
    const int taps = L.d.kh * L.d.kw, cin = L.d.cin / n_groups(L.d), rows = group_view(L.d).cout * n_groups(L.d);
    const size_t n = (size_t)rows * taps * ((cin + 63) / 64) * 64;
    int grid = (int)((n + 255) / 256); if (grid > c->num_sms * 8) grid = c->num_sms * 8;
    k_pack_halo<<<grid, 256, 0, c->stream>>>((const __nv_bfloat16*)L.weight, L.d.cout, rows, taps, cin, bn, (__nv_bfloat16*)L.weight_halo);
    DC_CUDA(cudaGetLastError());
    L.halo_bn = bn;
    return DC_OK;
}

// Normal layers need no repacking ([cout][kh][kw][cin] is already K-major); few-channel layers
// get their tap-major packed copy and a buffer for the channel-padded input.
int dc_pack_weights_bf16(dc_cache* c, int layer)
{
    dc_layer_rt& L = c->L[layer];
    TcPlan p;
    HaloPlan h;
    const dc_layer_desc dg = group_view(L.d);                     // the layer itself when it is not grouped
    if (halo_ok(dg, h)) {
        // [cout][taps][cin / groups]: channel blocks never straddle a group (BN divides cout / groups)
        const size_t n = (size_t)dg.cout * n_groups(L.d) * L.d.kh * L.d.kw * h.kchunks * 64;
        DC_CUDA(cudaMalloc(&L.weight_halo, n * 2));
        c->bytes += n * 2;
        bool changed;
        const int rc = pack_halo(c, L, h.BN, &changed);
        if (rc != DC_OK) return rc;
    }
    if (n_groups(L.d) > 1) return DC_OK;                          // grouped layers use the kernels above only
    if (pad16_ok(L.d)) {
        const size_t cout_taps = (size_t)L.d.cout * L.d.kh * L.d.kw;
        const size_t wbytes = cout_taps * 16 * 2, pbytes = (size_t)c->S * L.in_h * L.in_w * 32;
        DC_CUDA(cudaMalloc(&L.weight_packed, wbytes));
        DC_CUDA(cudaMalloc(&L.in_padded, pbytes));
        c->bytes += wbytes + pbytes;
        L.k_packed = L.d.kh * L.d.kw * 16;
        k_pack_pad16<<<dc_div_up((int)(cout_taps * 16), 256), 256, 0, c->stream>>>((const __nv_bfloat16*)L.weight, cout_taps, L.d.cin,
                                                                                   (__nv_bfloat16*)L.weight_packed);
        DC_CUDA(cudaGetLastError());
        return DC_OK;
    }
    if (make_plan(dg, p) || !smallc_ok(L.d)) return DC_OK;
    const int taps = L.d.kh * L.d.kw, kblocks = (taps + 1) / 2 * 2;
    const size_t wbytes = (size_t)kblocks * L.d.cout * 16, pbytes = (size_t)c->S * L.in_h * L.in_w * 16;
    DC_CUDA(cudaMalloc(&L.weight_packed, wbytes));
    DC_CUDA(cudaMalloc(&L.in_padded, pbytes));
    c->bytes += wbytes + pbytes;
    L.k_packed = kblocks * 8;
    k_pack_smallc<<<dc_div_up(kblocks * L.d.cout * 8, 256), 256, 0, c->stream>>>((const __nv_bfloat16*)L.weight, L.d.cout, taps,
                                                                               L.d.cin, kblocks, (__nv_bfloat16*)L.weight_packed);
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

static int launch_smallc(dc_cache* c, int layer, const void* in, void* out, const int32_t* tile_list,
                         const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const dc_layer_desc& d = L.d;
    EncodeTiledFn enc = encode_fn();
    if (!enc || !L.weight_packed) return DC_ERR_CUDA;
    const size_t pixels = (size_t)c->S * L.in_h * L.in_w;
    const int PW = DC_TILE_W + d.kw - 1, PH = DC_TILE_H + d.kh - 1;
    bool hit;
    CUtensorMap* tmAp = tm_find(L.tm_a, 4, &L.tm_next, L.in_padded, 7, 0, &hit);
    if (!hit) {
        cuuint64_t dims[4] = {8, (cuuint64_t)L.in_w, (cuuint64_t)L.in_h, (cuuint64_t)c->S};
        cuuint64_t strides[3] = {16, (cuuint64_t)L.in_w * 16, (cuuint64_t)L.in_h * L.in_w * 16};
        cuuint32_t box[4] = {8, (cuuint32_t)PW, (cuuint32_t)PH, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(tmAp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, L.in_padded, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            tm_drop(L.tm_a, 4, tmAp);
            return DC_ERR_CUDA;
        }
    }
    const CUtensorMap& tmA = *tmAp;
    TcSmallArgs sa;
    TcArgs& a = sa.t;
    a.bias = L.bias; a.out = (__nv_bfloat16*)out; a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks;
    a.Ho = d.out_h; a.Wo = d.out_w; a.Co = d.cout; a.Ci = d.cin; a.kh = d.kh; a.kw = d.kw; a.sh = 1; a.sw = 1;
    a.ph = d.ph; a.pw = d.pw; a.relu = d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.BN = d.cout; a.NB = 1; a.nb_off = 0; a.MT = 1; a.nbuf = 2; a.BK = 16; a.kchunks = 1; a.a_bytes = 0; a.b_bytes = 0; a.sbo = 128; a.layout_type = 0;
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(d.cout >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    a.status = c->status;
    a.early = dc_lists_settled(c);
    set_wait_limit(c, a);
    sa.wpacked = (const __nv_bfloat16*)L.weight_packed;
    sa.kblocks = L.k_packed / 8;
    sa.w_bytes = sa.kblocks * d.cout * 16;
    sa.PW = PW; sa.PH = PH;
    sa.stage_bytes = (PW * PH * 16 + 128 + 127) & ~127;          // patch + a readable pad behind its last pixel
    const int stage_bytes = sa.stage_bytes;
    const int ctas = L.tc_ctas == 2 && tmem_cols_for(2, 1, d.cout) <= 256 ? 2 : 1;
    a.tmem_cols = tmem_cols_for(2, 1, d.cout);
    int st = (ring_budget(ctas) - sa.w_bytes) / stage_bytes;
    a.stages = st > kMaxStages ? kMaxStages : st;
    if (a.stages < 2) return DC_ERR_CONFIG;
    a.epi_warps = epi_warps_for(ctas);
    a.bias_smem = t_bias_bytes ? d.cout : 0;
    const size_t smem = (size_t)a.stages * stage_bytes + ((sa.w_bytes + 127) & ~127) + ctl_bytes(a.epi_warps) + t_bias_bytes + 256;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) {
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_smallc, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    }
    int grid_pad = (int)((pixels + 255) / 256); if (grid_pad > c->num_sms * 8) grid_pad = c->num_sms * 8;
    int items = max_tiles < 1 ? 1 : max_tiles;
    int grid = items > c->num_sms * ctas ? c->num_sms * ctas : items;
    dc_prof_scope ps(c, DC_ST_CONV);
    if (in) DC_CUDA(dc_launch_pdl(k_pad_channels8, dim3((unsigned)grid_pad), 256, 0, c->stream, (const __nv_bfloat16*)in, pixels, (int)d.cin, (__nv_bfloat16*)L.in_padded));
    DC_CUDA(dc_launch_pdl(k_conv_tc_smallc, dim3((unsigned)(grid)), threads_for(a.epi_warps), smem, c->stream, tmA, sa));
    c->launches += in ? 2 : 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

static int launch_halo(dc_cache* c, int layer, int mt, bool slab, const void* in, void* out, const int32_t* tile_list,
                       const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const dc_layer_desc d = group_view(L.d);                      // what one group computes; L.d itself when ungrouped
    const int cin_all = L.d.cin, cout_all = L.d.cout;
    HaloPlan h;
    EncodeTiledFn enc = encode_fn();
    if (!enc || !L.weight_halo || !halo_ok(d, h, L.tc_bn)) return DC_ERR_CONFIG;
    bool repacked;
    const int prc = pack_halo(c, L, h.BN, &repacked);
    if (prc != DC_OK) return prc;
    const int G = n_groups(L.d);
    bool hit;
    CUtensorMap* tmAp = tm_find(L.tm_a, 4, &L.tm_next, in, slab ? 5 : 3, 0, &hit);
    if (!hit) {
        cuuint64_t dims[4] = {(cuuint64_t)cin_all, (cuuint64_t)L.in_w, (cuuint64_t)L.in_h, (cuuint64_t)c->S};
        const InPitch ip = in_pitch(L, cin_all);
        cuuint64_t strides[3] = {ip.px * 2, ip.row * 2, (cuuint64_t)L.in_h * ip.row * 2};
        cuuint32_t box[4] = {8, (cuuint32_t)h.PW, (cuuint32_t)h.PH, 1};
        if (slab) { box[0] = 64; box[1] = DC_TILE_W; }            // a column slab: 64 channels x 8 pixels x PH rows
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(tmAp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(in), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, slab ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            tm_drop(L.tm_a, 4, tmAp);
            return DC_ERR_CUDA;
        }
    }
    const CUtensorMap& tmA = *tmAp;
    TcHaloArgs ha;
    TcArgs& a = ha.t;
    a.bias = L.bias; a.out = (__nv_bfloat16*)out; a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks;
    a.Ho = d.out_h; a.Wo = d.out_w; a.Co = cout_all; a.Ci = d.cin; a.kh = d.kh; a.kw = d.kw; a.sh = 1; a.sw = 1;
    a.ph = d.ph; a.pw = d.pw; a.relu = d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.BN = h.BN; a.NB = h.NB * G; a.nb_off = 0; a.nb_group = h.NB; a.c_group = d.cin; a.BK = 64; a.kchunks = h.kchunks; a.MT = mt; a.nbuf = mt * h.BN * 2 <= 512 ? 2 : 1;
    a.a_bytes = 0; a.b_bytes = h.b_bytes; a.sbo = 128; a.layout_type = 0;
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(h.BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    a.status = c->status;
    a.early = repacked ? 0 : dc_lists_settled(c);                  // the producer sends for its first weights early
    set_wait_limit(c, a);
    ha.wpacked = (const __nv_bfloat16*)L.weight_halo;
    ha.k_last = h.k_last;
    ha.PW = h.PW; ha.PH = h.PH; ha.plane_bytes = h.plane_bytes;
    ha.patch_bytes = slab ? h.PH * DC_TILE_W * 128 : h.patch_bytes;
    // patch ring: as deep as leaves at least 3 weight stages (a small-K item is one patch, so depth = items in flight)
    a.tmem_cols = tmem_cols_for(a.nbuf, mt, h.BN);
    const int ctas = L.tc_ctas == 2 && a.tmem_cols <= 256 ? 2 : 1;
    const int budget = ring_budget(ctas);
    ha.a_stages = 2;
    for (int as = 4; as > 2; --as)
        if (budget - as * mt * ha.patch_bytes >= 3 * h.b_bytes) { ha.a_stages = as; break; }
    const int a_total = ha.a_stages * mt * ha.patch_bytes;
    int st = (budget - a_total) / h.b_bytes;
    a.stages = st > kMaxStages ? kMaxStages : st;
    if (a.stages < 2) return DC_ERR_CONFIG;
    a.epi_warps = epi_warps_for(ctas);
    a.bias_smem = t_bias_bytes ? d.cout * G : 0;
    const size_t smem = (size_t)a_total + (size_t)a.stages * h.b_bytes + ctl_bytes(a.epi_warps) + t_bias_bytes + 1280;
    if (smem > 227 * 1024) return DC_ERR_CONFIG;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) {
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_halo<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_halo<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_halo<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_halo<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    }
    long long items = (long long)(((max_tiles < 1 ? 1 : max_tiles) + mt - 1) / mt) * a.NB;
    int grid = items > c->num_sms * ctas ? c->num_sms * ctas : (int)items;
    dc_prof_scope ps(c, DC_ST_CONV);
    if (slab) {
        if (mt == 2) DC_CUDA(dc_launch_pdl(k_conv_tc_halo<2, true>, dim3((unsigned)(grid)), threads_for(a.epi_warps), smem, c->stream, tmA, ha));
        else DC_CUDA(dc_launch_pdl(k_conv_tc_halo<1, true>, dim3((unsigned)(grid)), threads_for(a.epi_warps), smem, c->stream, tmA, ha));
    } else {
        if (mt == 2) DC_CUDA(dc_launch_pdl(k_conv_tc_halo<2, false>, dim3((unsigned)(grid)), threads_for(a.epi_warps), smem, c->stream, tmA, ha));
        else DC_CUDA(dc_launch_pdl(k_conv_tc_halo<1, false>, dim3((unsigned)(grid)), threads_for(a.epi_warps), smem, c->stream, tmA, ha));
    }
    c->launches += 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

// The CTA-pair kernel takes stride-1 layers with cin a multiple of 16 (the column-slab conditions) whose output
// channels divide into blocks of 256 or 128 (half a block per CTA).
static bool pair_ok(const dc_layer_desc& d, int& bn)
{
    HaloPlan h;
    if (n_groups(d) > 1 || !halo_ok(d, h)) return false;
    bn = d.cout % 256 == 0 ? 256 : (d.cout % 128 == 0 ? 128 : 0);
    return bn != 0;
}

static int launch_pair(dc_cache* c, int layer, const void* in, void* out, const int32_t* tile_list,
                       const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const dc_layer_desc& d = L.d;
    EncodeTiledFn enc = encode_fn();
    int bn = 0;
    HaloPlan h;
    if (!enc || !L.weight_halo || !pair_ok(d, bn) || !halo_ok(d, h)) return DC_ERR_CONFIG;
    const int half = bn / 2, taps = d.kh * d.kw, kchunks = h.kchunks;
    bool repacked;                                               // weights grouped by half blocks: [2 NB][taps][kchunks][half][64], read after the wait
    const int prc = pack_halo(c, L, half, &repacked);
    if (prc != DC_OK) return prc;
    const int PH = DC_TILE_H + d.kh - 1;
    bool hit_a, hit_b;
    CUtensorMap* tmAp = tm_find(L.tm_a, 4, &L.tm_next, in, 5, 0, &hit_a);     // the column-slab map of the single-CTA kernel
    if (!hit_a) {
        cuuint64_t dims[4] = {(cuuint64_t)d.cin, (cuuint64_t)L.in_w, (cuuint64_t)L.in_h, (cuuint64_t)c->S};
        const InPitch ip = in_pitch(L, d.cin);
        cuuint64_t strides[3] = {ip.px * 2, ip.row * 2, (cuuint64_t)L.in_h * ip.row * 2};
        cuuint32_t box[4] = {64, DC_TILE_W, (cuuint32_t)PH, 1};
        cuuint32_t estr[4] = {1, 1, 1, 1};
        if (enc(tmAp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(in), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            tm_drop(L.tm_a, 4, tmAp);
            return DC_ERR_CUDA;
        }
    }
    const int b_bytes = half * 128;                              // one CTA's weight tile: half rows of 64 channels
    CUtensorMap* tmWp = tm_find(&L.tm_b, 1, nullptr, L.weight_halo, 7, half, &hit_b);
    if (!hit_b) {                                                // the packed weights as rows of 128 bytes; a box is one tile
        const cuuint64_t rows = (cuuint64_t)d.cout * taps * kchunks;
        cuuint64_t dims[2] = {64, rows};
        cuuint64_t strides[1] = {128};
        cuuint32_t box[2] = {64, (cuuint32_t)(b_bytes / 128)};
        cuuint32_t estr[2] = {1, 1};
        if (enc(tmWp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, L.weight_halo, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
            tm_drop(&L.tm_b, 1, tmWp);
            return DC_ERR_CUDA;
        }
    }
    TcHaloArgs ha;
    TcArgs& a = ha.t;
    a.bias = L.bias; a.out = (__nv_bfloat16*)out; a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks;
    a.Ho = d.out_h; a.Wo = d.out_w; a.Co = d.cout; a.Ci = d.cin; a.kh = d.kh; a.kw = d.kw; a.sh = 1; a.sw = 1;
    a.ph = d.ph; a.pw = d.pw; a.relu = d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.BN = bn; a.NB = d.cout / bn; a.nb_off = 0; a.BK = 64; a.kchunks = kchunks; a.MT = 1; a.nbuf = 2;
    a.a_bytes = 0; a.b_bytes = b_bytes; a.sbo = 128; a.layout_type = 0;
    // instruction descriptor: D = f32, A = B = bf16, both K-major, N = bn, M = 256 (128 rows in each CTA)
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
    a.status = c->status;
    a.early = dc_lists_settled(c);
    set_wait_limit(c, a);
    a.tmem_cols = tmem_cols_for(2, 1, bn);
    ha.wpacked = (const __nv_bfloat16*)L.weight_halo;
    ha.k_last = h.k_last;
    ha.PW = DC_TILE_W; ha.PH = PH; ha.plane_bytes = 0;
    ha.patch_bytes = PH * DC_TILE_W * 128;                       // one slab
    const int budget = ring_budget(1);
    ha.a_stages = 2;
    for (int as = 4; as > 2; --as)
        if (budget - as * ha.patch_bytes >= 4 * b_bytes) { ha.a_stages = as; break; }
    int st = (budget - ha.a_stages * ha.patch_bytes) / b_bytes;
    a.stages = st > kMaxStages ? kMaxStages : st;
    if (a.stages < 2) return DC_ERR_CONFIG;
    a.bias_smem = t_bias_bytes ? d.cout : 0;
    const size_t smem = (size_t)ha.a_stages * ha.patch_bytes + (size_t)a.stages * b_bytes + ctl_bytes(4) + t_bias_bytes + 1280;
    if (smem > 227 * 1024) return DC_ERR_CONFIG;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device))
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    const long long items = (long long)(((max_tiles < 1 ? 1 : max_tiles) + 1) / 2) * a.NB;
    const int max_pairs = c->num_sms / 2;                        // one CTA per SM, a pair per TPC
    const int pairs = items > max_pairs ? max_pairs : (int)items;
    dc_prof_scope ps(c, DC_ST_CONV);
    DC_CUDA(dc_launch_pdl(k_conv_tc_pair, dim3((unsigned)(2 * pairs)), kThreads, smem, c->stream, *tmAp, *tmWp, ha));
    c->launches += 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

static int launch_group(dc_cache* c, int layer, int grp, const void* in, void* out, const int32_t* tile_list,
                        const int32_t* tile_count, const uint32_t* masks, int max_tiles);

int dc_launch_conv_bf16(dc_cache* c, int layer, const void* in, void* out, const int32_t* tile_list,
                        const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    const int G = n_groups(c->L[layer].d);
    t_ring_kb = c->overlap_mode ? 182 : 200;
    t_bias_bytes = bias_bytes_for(all_groups(c->L[layer].d));
    // eight epilogue warps take the registers that the block search of the next frame needs to stay resident beside
    // this kernel: while that overlap is in use the CTA keeps to four
    t_epi_warps = c->L[layer].tc_ew == 8 && !c->overlap_mode ? 8 : 4;
    for (int grp = 0; grp < (c->L[layer].tc_cs > 0 ? G : 1); ++grp) {        // clusters: one launch per group
        int rc = launch_group(c, layer, grp, in, out, tile_list, tile_count, masks, max_tiles);
        if (rc == DC_ERR_CONFIG && t_ring_kb != 200) {            // the layer's tuned shape needs the full rings: it gets them
            t_ring_kb = 200;
            rc = launch_group(c, layer, grp, in, out, tile_list, tile_count, masks, max_tiles);
        }
        if (rc != DC_OK) return rc;
    }
    return DC_OK;
}

// Flat tiles that come as one box, where they took 16, one per group.
// rows: a 1 x 1 layer whose rows are 1, 2, 4, 8 or 16 groups.  The streams' rows lie one under another, so a tile is 16, 8, 4, 2 or 1 whole
// rows of that stack (columns beyond the row's end are zeros).  images: a small map under a larger kernel.  A tile is as many whole
// images as fit (gpt groups); the box displaced by a tap is cut at every image's edges.
// 128 streams, 7 x 7: 512 -> 2048 28 -> 20 us, 2048 -> 512 25 -> 16, 3 x 3 512 -> 512 50 -> 28 (128 tiles, then 56 and 64).
struct FlatBox { int rows, images; };
static FlatBox flat_box(const dc_layer_rt& L, const dc_layer_desc& d)
{
    FlatBox f = {0, 0};
    if (!L.flat || L.s2d_s || DC_TILE_W * L.gpr * d.sw > 256) return f;          // TMA box limit
    const int rows = DC_TILE_H / L.gpr;
    if (d.kh == 1 && d.kw == 1) {
        if (d.ph == 0 && d.pw == 0 && L.in_h == d.out_h * d.sh && DC_TILE_H % L.gpr == 0 && rows * d.sh <= 256) f.rows = rows;
    } else if (L.gpt % (d.out_h * L.gpr) == 0 && d.out_h * d.sh <= 256) f.images = L.gpt / (d.out_h * L.gpr);
    return f;
}

// Tensor maps of the tap-by-tap kernels: the input (16 x 8 windows, or single row pieces for flat tiles) and the weights.
static int generic_maps(dc_cache* c, dc_layer_rt& L, const dc_layer_desc& d, const TcPlan& p, const void* in, const void* weights, int cin_all, int cout_all,
                        CUtensorMap** map_a, CUtensorMap** map_b)
{
    EncodeTiledFn enc = encode_fn();
    if (!enc) return DC_ERR_CUDA;
    bool hit_a, hit_b;
    const FlatBox fb = flat_box(L, d);
    CUtensorMap* tmAp = tm_find(L.tm_a, 4, &L.tm_next, in, L.tc_cs > 0 ? 10 : fb.rows || fb.images ? 9 : L.flat ? 8 : 1, 0, &hit_a);
    CUtensorMap* tmBp = tm_find(&L.tm_b, 1, nullptr, weights, 1, p.BN, &hit_b);
    if (!hit_a) {   // input map [S][Hi][Wi][Ci] bf16; box = BK channels x 16 columns x 8 rows x 1 stream
        cuuint64_t dims[4] = {(cuuint64_t)(L.tc_cs > 0 ? d.cin : cin_all), (cuuint64_t)L.in_w, (cuuint64_t)L.in_h, (cuuint64_t)c->S};
        const InPitch ip = in_pitch(L, cin_all);
        cuuint64_t strides[3] = {ip.px * 2, ip.row * 2, (cuuint64_t)L.in_h * ip.row * 2};
        // a strided convolution reads every sw-th column / sh-th row: the box spans TW * sw x TH * sh input
        // pixels and the traversal strides pick TW x TH of them
        // (flat tiles: one image row of 8 pixels per box)
        cuuint32_t box[4] = {(cuuint32_t)p.BK, (cuuint32_t)(DC_TILE_W * d.sw), (cuuint32_t)(L.flat ? 1 : DC_TILE_H * d.sh), 1};
        cuuint32_t estr[4] = {1, (cuuint32_t)d.sw, (cuuint32_t)(L.flat ? 1 : d.sh), 1};
        if (fb.rows) { dims[2] *= (cuuint64_t)c->S; dims[3] = 1; }
        if (fb.images) box[3] = (cuuint32_t)fb.images;
        if (fb.rows || fb.images) { box[1] *= (cuuint32_t)L.gpr; box[2] = (cuuint32_t)((fb.rows ? fb.rows : d.out_h) * d.sh); estr[2] = (cuuint32_t)d.sh; }
        if (enc(tmAp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(in), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, p.swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) { tm_drop(L.tm_a, 4, tmAp); tm_drop(&L.tm_b, 1, tmBp); return DC_ERR_CUDA; }
    }
    if (!hit_b) {   // weights [cout][K] bf16, K = kh * kw * cin
        const cuuint64_t K = (cuuint64_t)d.kh * d.kw * d.cin;
        cuuint64_t dims[2] = {K, (cuuint64_t)cout_all};               // every group's rows; a launch reads its own (nb_off)
        cuuint64_t strides[1] = {K * 2};
        cuuint32_t box[2] = {(cuuint32_t)p.BK, (cuuint32_t)p.BN};
        cuuint32_t estr[2] = {1, 1};
        if (enc(tmBp, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(weights), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, p.swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) { tm_drop(&L.tm_b, 1, tmBp); return DC_ERR_CUDA; }
    }
    *map_a = tmAp; *map_b = tmBp;
    return DC_OK;
}

// Few tiles: one cluster of L.tc_cs CTAs per tile and block of L.tc_bn channels.
static bool cluster_plan(const dc_layer_desc& d, int bn, int cs, TcPlan& p)
{
    if (bn != 32 && bn != 64) return false;
    t_ring_kb = 200; t_epi_warps = 4; t_bias_bytes = 0;
    if (!make_plan(d, p, 1, bn, 1)) return false;
    const int kiters = d.kh * d.kw * (d.cin / p.BK);
    if (kiters < cs) return false;
    const int most = dc_div_up(kiters, cs);
    p.stages = most < kClusterStages ? most : kClusterStages;
    while (p.stages > 1 && dc_cluster_smem(p.stages, p.a_bytes, p.b_bytes, p.BN) > 227 * 1024) --p.stages;
    return p.stages >= 2 || most == 1;
}

// Do the clusters of a layer with every tile dirty run at the same time?
static bool cluster_fits(const dc_cache* c, const dc_layer_rt& L, const dc_layer_desc& d, int bn, int cs)
{
    TcPlan p;
    if (d.cout % bn != 0 || !cluster_plan(d, bn, cs, p)) return false;
    const long long clusters = (long long)L.tiles_x * L.tiles_y * c->S * (d.cout / bn);
    return clusters <= dc_cluster_wave(c->device, cs, dc_cluster_smem(p.stages, p.a_bytes, p.b_bytes, p.BN));
}

// How many CTAs a layer's clusters have, 0: it stays on the other kernels.  By sizes alone: a cluster sums in parts, so a choice
// by timing would show in the outputs.  Measured with `steps` of 64 channels, the fastest other kernel against clusters of 2 /
// 4 / 8 (us a launch): 72 steps, 1 tile 18.9 against 13.4 / 8.8 / 8.2; 36 steps, 2 tiles 12.4, 9.4 / 6.8 / 7.3; 16 steps 7.9, 7.0 / 5.8 /
// 6.1; 9 steps 6.5, 7.1 / 7.2 / 9.2; 4 steps 5.0, 6.1.  They pay while one wave holds them (54 steps in twos: 72 clusters 14.2
// against 16.1, 96 clusters 25.7 against 16.5); twos, the last resort, need a longer reduction (27 steps 19.8 against 20.4, 18
// steps 9.4 against 8.5, 25 steps 25.9 against 18.6).  Over the layers of the trunks at 1 to 128 streams the rule's choice takes
// 0.3 % longer than the fastest one of each layer.
static int cluster_rule(const dc_cache* c, const dc_layer_rt& L, const dc_layer_desc& d)
{
    if (L.d.cout % 32 != 0) return 0;                             // its finish knows whole blocks alone
    const int steps = d.kh * d.kw * ((d.cin + 63) / 64);
    const struct { int cs, steps; } take[3] = {{8, 48}, {4, 16}, {2, 26}};
    for (const auto& t : take)
        if (steps >= t.steps && (cluster_fits(c, L, d, 32, t.cs) || cluster_fits(c, L, d, 64, t.cs))) return t.cs;
    return 0;
}

static int launch_cluster(dc_cache* c, int layer, int grp, const void* in, void* out, const int32_t* tile_list,
                          const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const dc_layer_desc d = group_view(L.d);
    TcPlan p;
    if (!cluster_plan(d, L.tc_bn, L.tc_cs, p)) return DC_ERR_CONFIG;
    in = (const uint8_t*)in + (size_t)grp * d.cin * 2;
    CUtensorMap *tmAp, *tmBp;
    const int rc = generic_maps(c, L, d, p, in, L.weight, L.d.cin, L.d.cout, &tmAp, &tmBp);
    if (rc != DC_OK) return rc;
    dc_cluster_args a;
    a.bias = L.bias; a.out = (__nv_bfloat16*)out; a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks;
    a.Ho = d.out_h; a.Wo = d.out_w; a.Co = L.d.cout; a.Ci = d.cin; a.kh = d.kh; a.kw = d.kw; a.sh = d.sh; a.sw = d.sw;
    a.ph = d.ph; a.pw = d.pw; a.relu = d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.BN = p.BN; a.NB = p.NB; a.BK = p.BK; a.kchunks = d.cin / p.BK; a.stages = p.stages; a.a_bytes = p.a_bytes; a.b_bytes = p.b_bytes;
    a.nb_off = grp * p.NB; a.CS = L.tc_cs;
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    a.sbo = p.sbo; a.layout_type = p.layout_type; a.tmem_cols = tmem_cols_for(1, 1, p.BN);
    a.status = c->status;
    TcArgs w;
    set_wait_limit(c, w);
    a.wait_ns = w.wait_ns; a.skip_loads = w.skip_loads; a.early = dc_lists_settled(c);
    a.add_in = (const __nv_bfloat16*)c->add_in; a.add_out = (__nv_bfloat16*)c->add_out; a.add_relu = c->add_relu;
    dc_prof_scope ps(c, DC_ST_CONV);
    c->launches += 1;
    return dc_launch_cluster_kernel(c, *tmAp, *tmBp, a, max_tiles);
}

static int launch_group(dc_cache* c, int layer, int grp, const void* in, void* out, const int32_t* tile_list,
                        const int32_t* tile_count, const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    if (L.tc_cs > 0) return launch_cluster(c, layer, grp, in, out, tile_list, tile_count, masks, max_tiles);
    if (L.flat && L.tc_mt > 2) return DC_ERR_CONFIG;              // flat tiles exist in the tap-by-tap kernel only
    if (L.tc_mt == 7) return launch_pair(c, layer, in, out, tile_list, tile_count, masks, max_tiles);
    if (L.tc_mt >= 5) return launch_halo(c, layer, L.tc_mt - 4, true, in, out, tile_list, tile_count, masks, max_tiles);
    if (L.tc_mt >= 3) return launch_halo(c, layer, L.tc_mt - 2, false, in, out, tile_list, tile_count, masks, max_tiles);
    const bool grouped = n_groups(L.d) > 1;
    const bool pad16 = !grouped && pad16_ok(L.d) && L.weight_packed && L.in_padded;
    const dc_layer_desc d = pad16 ? padded16(L.d) : group_view(L.d);
    const int cin_all = pad16 ? 16 : L.d.cin, cout_all = L.d.cout;
    const void* weights = pad16 ? L.weight_packed : L.weight;
    if (pad16) {
        const size_t pixels = (size_t)c->S * L.in_h * L.in_w;
        int grid_pad = (int)((pixels + 255) / 256); if (grid_pad > c->num_sms * 8) grid_pad = c->num_sms * 8;
        dc_prof_scope ps(c, DC_ST_CONV);
        DC_CUDA(dc_launch_pdl(k_pad_channels16, dim3((unsigned)grid_pad), 256, 0, c->stream, (const __nv_bfloat16*)in, pixels, (int)L.d.cin, (__nv_bfloat16*)L.in_padded));
        c->launches += 1;
        in = L.in_padded;
    }
    const int G = n_groups(L.d);
    TcPlan p;
    int ctas = L.tc_ctas == 2 ? 2 : 1;
    if (ctas == 2 && !make_plan(d, p, L.tc_mt, L.tc_bn, 2)) ctas = 1;
    if (!make_plan(d, p, L.tc_mt, L.tc_bn, ctas)) {
        if (smallc_ok(d)) return launch_smallc(c, layer, in, out, tile_list, tile_count, masks, max_tiles);
        return DC_ERR_CONFIG;
    }
    CUtensorMap *tmAp, *tmBp;
    const int rc = generic_maps(c, L, d, p, in, weights, cin_all, cout_all, &tmAp, &tmBp);
    if (rc != DC_OK) return rc;
    const CUtensorMap& tmA = *tmAp;
    const CUtensorMap& tmB = *tmBp;
    TcArgs a;
    a.bias = L.bias; a.out = (__nv_bfloat16*)out; a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks;
    a.Ho = d.out_h; a.Wo = d.out_w; a.Co = cout_all; a.Ci = d.cin; a.kh = d.kh; a.kw = d.kw; a.sh = d.sh; a.sw = d.sw;
    a.ph = d.ph; a.pw = d.pw; a.relu = d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.BN = p.BN; a.NB = p.NB * G; a.nb_off = 0; a.nb_group = p.NB; a.c_group = d.cin; a.BK = p.BK; a.kchunks = d.cin / p.BK; a.stages = p.stages; a.MT = p.MT; a.nbuf = p.nbuf;
    a.a_bytes = p.a_bytes; a.b_bytes = p.b_bytes; a.sbo = p.sbo; a.layout_type = p.layout_type;
    a.tmem_cols = tmem_cols_for(p.nbuf, p.MT, p.BN);
    // instruction descriptor: D = f32, A = B = bf16, both K-major, N = BN, M = 128
    a.idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.BN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
    a.status = c->status;
    a.flat = L.flat; a.gpr = L.gpr; a.n_groups_all = c->S * d.out_h * L.gpr; a.gpt = L.flat ? L.gpt : DC_TILE_H;
    a.flat_rows = flat_box(L, d).rows; a.flat_images = flat_box(L, d).images;
    a.epi_warps = epi_warps_for(ctas);
    a.bias_smem = t_bias_bytes ? d.cout * G : 0;
    a.slab_order = L.weight_halo != nullptr;
    a.add_in = (const __nv_bfloat16*)c->add_in; a.add_out = (__nv_bfloat16*)c->add_out; a.add_relu = c->add_relu;
    a.early = dc_lists_settled(c);
    set_wait_limit(c, a);
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) {
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        DC_CUDA(cudaFuncSetAttribute(k_conv_tc<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    }
    long long items = (long long)(((max_tiles < 1 ? 1 : max_tiles) + p.MT - 1) / p.MT) * a.NB;
    int grid = items > c->num_sms * ctas ? c->num_sms * ctas : (int)items;
    dc_prof_scope ps(c, DC_ST_CONV);
    if (a.add_out && p.MT != 1) return DC_ERR_CONFIG;
    if (a.add_out) DC_CUDA(dc_launch_pdl(k_conv_tc<1, true>, dim3((unsigned)(grid)), threads_for(a.epi_warps), p.smem, c->stream, tmA, tmB, a));
    else if (p.MT == 2) DC_CUDA(dc_launch_pdl(k_conv_tc<2, false>, dim3((unsigned)(grid)), threads_for(a.epi_warps), p.smem, c->stream, tmA, tmB, a));
    else DC_CUDA(dc_launch_pdl(k_conv_tc<1, false>, dim3((unsigned)(grid)), threads_for(a.epi_warps), p.smem, c->stream, tmA, tmB, a));
    c->launches += 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

// Does the layer's kernel take the add that follows it along?  On clusters always; tap by tap with one tile per item where every tile of
// the layer has an SM: there a launch is a chain of latencies and the add one more of them (ResNet-50, one stream: 365 -> 346 us a frame).  With more
// tiles than that the add as a kernel of its own, which reads half of its operand from L2, is the faster one.
bool dc_conv_takes_add(const dc_cache* c, int layer)
{
    const dc_layer_rt& L = c->L[layer];
    if (L.tc_cs > 0) return true;
    TcPlan p;
    if (c->cfg.dtype != DC_BF16 || !dc_conv_bf16_supported(c, layer) || n_groups(L.d) > 1 || L.s2d_s || L.d.cin < 16 || L.d.cout % 32 != 0 || L.tc_mt != 1) return false;
    const int ctas = L.tc_ctas == 2 ? 2 : 1;
    t_ring_kb = 200; t_epi_warps = L.tc_ew == 8 ? 8 : 4; t_bias_bytes = bias_bytes_for(L.d);
    return make_plan(L.d, p, 1, L.tc_bn, ctas) && (long long)dc_layer_tiles(c, L) * p.NB <= c->num_sms;
}

// Picks, per convolution layer, the operand scheme and the work-item shape (tiles per item x channels per block)
// by timing the candidates once on the layer's own buffers with every tile dirty.  All candidates of a layer sum in the same
// order (StepOrder; cluster_rule decides whether a layer's candidates are the clusters of one size or the other kernels), so
// the choice changes no bit of an output.  Called by dc_cache_create (which may synchronise).
int dc_conv_bf16_autotune(dc_cache* c, int layer, const void* in)
{
    dc_layer_rt& L = c->L[layer];
    TcPlan p;
    if (c->cfg.dtype != DC_BF16 || !encode_fn() || getenv("DC_NO_TENSOR_CORES")) return DC_OK;
    const bool grouped = n_groups(L.d) > 1;
    if (grouped && !dc_conv_bf16_supported(c, layer)) return DC_OK;
    const dc_layer_desc de = !grouped && pad16_ok(L.d) ? padded16(L.d) : group_view(L.d);
    const bool generic = make_plan(de, p);
    if (!generic && (grouped || !smallc_ok(L.d))) return DC_OK;
    if (getenv("DC_CONV_NO_TUNE")) return DC_OK;
    cudaEvent_t e0, e1;
    DC_CUDA(cudaEventCreate(&e0));
    DC_CUDA(cudaEventCreate(&e1));
    float best = 1e30f; int best_mt = L.tc_mt, best_bn = L.tc_bn, best_ctas = 1, best_flat = 0, best_ew = 4, best_cs = 0;
    c->list_mark = -1;                                                // the list of all tiles
    constexpr int kTuneReps = 6;                                      // timed launches per candidate, after one untimed
    // the GPU may have been idle: bring the clocks up before the first candidate is timed
    for (int rep = 0; rep < 12; ++rep)
        if (dc_launch_conv_bf16(c, layer, in, L.map[0], L.all_list, dc_all_count(c, layer), c->zero_masks, dc_layer_tiles(c, L)) != DC_OK) break;
    const bool verbose = getenv("DC_VERBOSE") != nullptr;
    // times the launch the current L.tc_* fields select; keeps it when it is the fastest so far
    // DC_CONV_SCHEME=<code> (diagnostics, tests): only candidates of that operand scheme are timed, so the scheme runs
    // wherever it can (1, 2 tap by tap; 3, 4 patch; 5, 6 column slabs; the second of each pair with two tiles per item;
    // 7 column slabs on CTA pairs; 8, 9 tap by tap on flat tiles; 10 tap by tap on clusters)
    const int only = getenv("DC_CONV_SCHEME") ? atoi(getenv("DC_CONV_SCHEME")) : 0;
    // DC_CONV_BLOCK=<channels> likewise: only candidates with blocks of so many output channels
    const int only_bn = getenv("DC_CONV_BLOCK") ? atoi(getenv("DC_CONV_BLOCK")) : 0;
    auto trial = [&](const char* what) {
        if (only_bn > 0 && generic && L.tc_bn != only_bn) return;
        if (only > 0 && generic && (L.tc_cs > 0 ? 10 : L.flat ? L.tc_mt + 7 : L.tc_mt) != only) return;
        int rc = DC_OK;
        for (int rep = 0; rep < kTuneReps + 1 && rc == DC_OK; ++rep) {
            if (rep == 1) cudaEventRecord(e0, c->stream);
            rc = dc_launch_conv_bf16(c, layer, in, L.map[0], L.all_list, dc_all_count(c, layer), c->zero_masks, dc_layer_tiles(c, L));
        }
        cudaEventRecord(e1, c->stream);
        if (rc != DC_OK || cudaEventSynchronize(e1) != cudaSuccess) { cudaGetLastError(); return; }
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (verbose) fprintf(stderr, "libdeepcache: layer %d: %s, tiles/item code %d, %d channels per block, %d CTA(s) per SM, %d epilogue warps, clusters of %d: %.4f ms\n",
                             layer, what, L.flat ? L.tc_mt + 7 : L.tc_mt, L.tc_bn, L.tc_ctas, L.tc_ew, L.tc_cs, ms / kTuneReps);
        if (ms < best) { best = ms; best_mt = L.tc_mt; best_bn = L.tc_bn; best_ctas = L.tc_ctas; best_flat = L.flat; best_ew = L.tc_ew; best_cs = L.tc_cs; }
    };
    // clusters of CTAs sum in parts, so their size follows from the layer's sizes; the other kernels are then not timed
    const bool may_cluster = generic && !(de.cin < 16) && L.d.cout % 32 == 0 && L.d.cin == de.cin * n_groups(L.d);
    const int cs = may_cluster && (only == 0 || only == 10) ? cluster_rule(c, L, de) : 0;
    // one CTA per SM with four or eight epilogue warps, or two CTAs per SM with four each
    for (int shape = 0; shape < 3 && cs == 0; ++shape) {
        const int ctas = shape == 2 ? 2 : 1;
        L.tc_ctas = ctas; L.tc_ew = shape == 1 ? 8 : 4;
        t_epi_warps = L.tc_ew;                                        // make_plan below sizes the rings for it
        t_bias_bytes = bias_bytes_for(!grouped && pad16_ok(L.d) ? de : all_groups(L.d));
        if (!generic) {                                               // few input channels: one kernel shape, 1 or 2 CTAs per SM
            if (ctas == 2 && tmem_cols_for(2, 1, L.d.cout) > 256) continue;
            trial("few-channel kernel");
            continue;
        }
        const int default_bn = p.BN;
        for (int bn = default_bn; (bn >= 64 || bn == default_bn) && bn >= default_bn / 2; bn -= 32) {
            if (de.cout % bn != 0) continue;
            for (int mt = 1; mt <= 2; ++mt) {
                TcPlan q;
                if (!make_plan(de, q, mt, bn, ctas)) continue;
                L.tc_mt = mt; L.tc_bn = bn;
                trial("tap-by-tap kernel");
                // flat tiles where the 16 x 8 blocks leave a good part of their pixels outside the map
                if (L.d.cout % 32 == 0 && (L.tiles_flat * 20 <= L.tiles_x * L.tiles_y * c->S * 19 || only >= 8)) {
                    L.flat = 1;
                    trial("tap-by-tap kernel, flat tiles");
                    L.flat = 0;
                }
            }
        }
        // few tiles: narrow blocks, while every item has an SM, spread the epilogue (a launch is then a chain of latencies, and of its 5 us
        // 2.7 were four steps of 32 channels with the add that follows: ResNet-50, one stream, 325 us a frame, 300 so)
        for (int bn = 64; bn >= 32 && shape == 0; bn -= 32) {
            TcPlan q;
            if (2 * bn >= default_bn || de.cout % bn != 0 || (long long)dc_layer_tiles(c, L) * (L.d.cout / bn) > c->num_sms || !make_plan(de, q, 1, bn, ctas)) continue;
            L.tc_mt = 1; L.tc_bn = bn;
            trial("tap-by-tap kernel, narrow blocks");
        }
        HaloPlan h0;
        if (L.weight_halo && halo_ok(de, h0)) {
            for (int bn = h0.BN; (bn >= 64 || bn == h0.BN) && bn >= h0.BN / 2; bn -= 32) {
                HaloPlan h;
                if (!halo_ok(de, h, bn)) continue;
                for (int mt = 1; mt <= 2; ++mt) {                      // tc_mt 3 / 4: patch-reuse kernel with 1 / 2 tiles per item
                    if (ctas == 2 && tmem_cols_for(mt * h.BN * 2 <= 512 ? 2 : 1, mt, h.BN) > 256) continue;
                    L.tc_bn = bn;
                    if (bn == h0.BN) { L.tc_mt = mt + 2; trial("patch-reuse kernel"); }
                    L.tc_mt = mt + 4;                                   // tc_mt 5 / 6: column slabs with 1 / 2 tiles per item
                    trial("column-slab kernel");
                }
            }
        }
    }
    {
        int pbn = 0;
        if (cs == 0 && generic && L.weight_halo && pair_ok(L.d, pbn)) {   // tc_mt 7: a CTA pair per two tiles (cta_group::2)
            L.tc_mt = 7; L.tc_bn = pbn; L.tc_ctas = 1; L.tc_ew = 4;
            trial("CTA-pair kernel");
        }
    }
    if (cs > 0 || (may_cluster && only == 10)) {                      // asked for where the rule has none: any size (diagnostics)
        L.tc_mt = 1; L.tc_ctas = 1; L.tc_ew = 4;
        for (int bn = 32; bn <= 64; bn += 32)
            for (int k = cs > 0 ? cs : 2; k <= (cs > 0 ? cs : 8); k *= 2) {
                TcPlan q;
                if (de.cout % bn != 0 || !cluster_plan(de, bn, k, q) || (cs > 0 && !cluster_fits(c, L, de, bn, k))) continue;
                L.tc_bn = bn; L.tc_cs = k;
                trial("cluster kernel");
            }
        L.tc_cs = 0;
    }
    L.tc_mt = best_mt; L.tc_bn = best_bn; L.tc_ctas = best_ctas; L.flat = best_flat; L.tc_ew = best_ew; L.tc_cs = best_cs;
    cudaEventDestroy(e0); cudaEventDestroy(e1);
    if (L.tc_mt >= 3 && L.tc_cs == 0) {                               // packed for the choice before any frame is launched
        bool changed;
        const int rc = pack_halo(c, L, L.tc_mt == 7 ? L.tc_bn / 2 : L.tc_bn, &changed);
        if (rc != DC_OK) return rc;
    }
    c->launches = 0; c->list_mark = DC_LISTS_FRESH;
    if (verbose) fprintf(stderr, "libdeepcache: layer %d: chose code %d, %d channels per block, %d CTA(s) per SM, %d epilogue warps, clusters of %d (%.4f ms)\n",
                         layer, best_flat ? best_mt + 7 : best_mt, best_bn, best_ctas, best_ew, best_cs, best / kTuneReps);
    return DC_OK;
}

// Failure detection without a fault (not part of the public header: tests declare it themselves).  The next
// tensor-core convolution launch of this cache issues none of its operand copies and bounds its waits by wait_ms
// instead of 2 s: the MMA and epilogue roles find nothing arriving, give up, record DC_ERR_TIMEOUT in the status
// word, free their tensor memory and the kernel returns normally.  No copy and no MMA is in flight when they leave.
// (Cluster kernel: one CTA of each cluster issues none; the others finish their part and store nothing.)
// The launch after it is an ordinary one.
extern "C" int dc_debug_stall_next_conv(dc_cache* c, int wait_ms)
{
    if (!c || wait_ms < 1 || wait_ms > 1000) return DC_ERR_ARG;
    c->debug_stall_ms = wait_ms;
    return DC_OK;
}
