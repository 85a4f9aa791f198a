// Partial convolution of few tiles: the reduction of one output tile split over a cluster of CTAs.
//
// With one stream a deep layer has one to four 128-pixel tiles and a reduction of thousands: the persistent kernels of
// dc_conv_bf16.cu then run on a handful of SMs, each walking all taps and channels alone (512 -> 512, 3x3 at 7x7: 4 CTAs,
// 72 steps, 32 us).  Here a work item - one tile, a narrow block of BN = 32 or 64 output channels - belongs to a cluster of
// CS = 2, 4 or 8 CTAs.  Each takes 1 / CS of the (tap, channel chunk) steps, operands and MMA as in the tap-by-tap kernel;
// the partial sums meet through distributed shared memory: CTA r finishes pixels r * 128 / CS ..., and every CTA writes its
// sums of those pixels into r's shared memory; after one cluster barrier each CTA adds its CS copies in rank order,
// without touching the others again.  The weights do not depend on any kernel before, so their loads start before the
// wait for the previous layer.
// What bounds it: the chain of latencies of one item (tile list, one TMA round trip, the cluster barrier), and no longer
// the length of the reduction.
//
// An element-wise add that follows (a residual block's end) can be done in the same pass over the tile: reused pixels
// are read back from the output map, where the reuse copy has put them.  Such a launch visits every tile.
#include "dc_conv_cluster.cuh"
#include "dc_tcgen05.cuh"

namespace {

constexpr int kThreadsCl = 192;               // producer warp, MMA warp, four accumulator warps

struct CtlCl {
    unsigned long long full[kClusterStages], empty[kClusterStages], done;
    uint32_t tmem_base;
    volatile int abort_flag;
    unsigned long long wait_ns;
};

__device__ __forceinline__ bool cl_wait(uint32_t bar, uint32_t parity, CtlCl* ctl, int32_t* status)
{
    return mbar_wait_at(bar, parity, &ctl->abort_flag, &ctl->wait_ns, status);
}
// Leaves word of an abort in every CTA of the cluster (after the first cluster barrier, before the second).
__device__ __forceinline__ void abort_cluster(const CtlCl* ctl, int cs)
{
    for (int r = 0; r < cs; ++r)
        asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(map_to_cta((const void*)&ctl->abort_flag, (uint32_t)r)), "r"(1) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t addr, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
// padded row of partial sums: 16-byte accesses of neighbouring lanes fall in different banks
__host__ __device__ constexpr int red_pitch(int BN) { return BN + 4; }

__global__ void __launch_bounds__(kThreadsCl, 1) k_conv_cluster(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const dc_cluster_args a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = a.a_bytes + a.b_bytes;
    float* red = (float*)(ring + (size_t)a.stages * stage_bytes);            // [CS][128 / CS][BN + 4]: this CTA's pixels, from every CTA
    CtlCl* ctl = (CtlCl*)(red + 128 * red_pitch(a.BN));
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank(), item = blockIdx.x / a.CS, nb = item % a.NB, idx = item / a.NB;
    const int kiters = a.kh * a.kw * a.kchunks;
    const int k0 = rank * kiters / a.CS, nk = (rank + 1) * kiters / a.CS - k0;
    const bool skip_loads = a.skip_loads && rank == 0;           // failure-detection tests: one CTA of the cluster gets no operands

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 2); mbar_init(&ctl->empty[i], 1); }   // weights and pixels arrive apart
        mbar_init(&ctl->done, 1);
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(a.tmem_cols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");    // waited for before another CTA's shared memory is written
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), ring0 = smem_u32(ring);
    const int tap0 = k0 / a.kchunks, cc0 = k0 - tap0 * a.kchunks;
    const int w_row = (nb + a.nb_off) * a.BN, early = nk < a.stages ? nk : a.stages;
    auto load_weights = [&](int tap, int cc, uint32_t off, uint32_t slot) {
        mbar_expect_tx(full0 + off, (uint32_t)a.b_bytes);
        tma_load_2d(slot + a.a_bytes, &tmB, tap * a.Ci + cc * a.BK, w_row, full0 + off);
    };
    if (warp == 0 && !skip_loads && elect_one()) {
        int tap = tap0, cc = cc0;
        for (int it = 0; it < early; ++it) {
            load_weights(tap, cc, 8u * it, ring0 + it * stage_bytes);
            if (++cc == a.kchunks) { cc = 0; ++tap; }
        }
    }
    __syncwarp();
    // the previous kernel's output is read, and this one's written, only after the wait; the tile list and the bitmaps too,
    // unless they are older than that kernel
    if (!a.early) { dc_pdl_wait(); dc_pdl_release(); }
    const int n_tiles = __ldcg(a.tile_count);
    const int listed = __ldcg(a.tile_list + idx);     // inside the list's length whatever the count
    const bool present = idx < n_tiles;
    const int tile = present ? listed : 0;

    // this tile's pixels: pixel m is column m % 8 of tile row m / 8
    const int per_stream = a.tiles_x * a.tiles_y;
    const int ts = tile / per_stream, t_in = tile - ts * per_stream, ty = t_in / a.tiles_x, tx = t_in - ty * a.tiles_x;
    // What thread u finishes: 8 channels of one of this CTA's pixels.  The first unit's operands are fetched now, beside
    // the loads and MMAs.
    const int rows = 128 / a.CS, per_px = a.BN / 8, units = present ? rows * per_px : 0;
    struct Unit { size_t at; uint4 other; float4 b0, b1; bool in_map, active; };
    auto unit_of = [&](int u) -> Unit {
        Unit n;
        const int pr = u / per_px, c8 = u - pr * per_px, m = rank * rows + pr, row = m / DC_TILE_W, col = m % DC_TILE_W;
        const int y = ty * DC_TILE_H + row, x = tx * DC_TILE_W + col;
        n.in_map = y < a.Ho && x < a.Wo;
        n.active = n.in_map && !((__ldcg(a.masks + (size_t)tile * 4 + (row >> 2)) >> (8 * (row & 3) + col)) & 1u);
        const int ch = (nb + a.nb_off) * a.BN + c8 * 8;
        n.at = (((size_t)ts * a.Ho + y) * a.Wo + x) * a.Co + ch;
        n.b0 = __ldg((const float4*)(a.bias + ch)); n.b1 = __ldg((const float4*)(a.bias + ch + 4));
        return n;
    };
    auto fetch_other = [&](Unit& n) { if (n.in_map && a.add_out) n.other = *(const uint4*)(a.add_in + n.at); };
    Unit mine = {};
    if ((int)threadIdx.x < units) mine = unit_of(threadIdx.x);
    if (a.early) { dc_pdl_wait(); dc_pdl_release(); }
    fetch_other(mine);

    if (warp == 0) {
        // ---------------- producer ----------------
        bool ok = true;
        if (!present) {
            // the weights are on their way: let them land before this CTA's shared memory is given up
            if (lane == 0 && !skip_loads)
                for (int it = 0; it < early && ok; ++it) { mbar_arrive(&ctl->full[it]); ok = cl_wait(full0 + 8u * it, 0, ctl, a.status); }
        } else if (!skip_loads) {
            if (elect_one()) {
                const int fx = tx * DC_TILE_W * a.sw - a.pw, fy = ty * DC_TILE_H * a.sh - a.ph;
                RingPos r;
                r.start(ring0, (uint32_t)a.stages);
                int cc = cc0, ky = tap0 / a.kw, kx = tap0 - ky * a.kw;
                for (int it = 0; it < nk; ++it) {
                    if (it >= a.stages) {
                        ok = cl_wait(empty0 + r.off, r.phase ^ 1u, ctl, a.status);
                        if (!ok) break;
                        load_weights(ky * a.kw + kx, cc, r.off, r.data);
                    }
                    mbar_expect_tx(full0 + r.off, (uint32_t)a.a_bytes);
                    tma_load_4d(r.data, &tmA, cc * a.BK, fx + kx, fy + ky, ts, full0 + r.off);
                    if (++cc == a.kchunks) { cc = 0; if (++kx == a.kw) { kx = 0; ++ky; } }
                    r.next(ring0, (uint32_t)a.stages, (uint32_t)stage_bytes);
                }
            }
        }
        // on an abort: give the copies already issued a bounded chance to land before the CTA exits
        if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (present && elect_one()) {
            const uint64_t dconst = umma_desc(0, a.sbo, a.layout_type);
            const uint32_t d_hi = (uint32_t)(dconst >> 32), r0 = (uint32_t)dconst + (ring0 >> 4);
            const uint32_t stage_lo = (uint32_t)stage_bytes >> 4, a_lo = (uint32_t)a.a_bytes >> 4;
            const int ksteps = a.BK / 16;
            RingPos r;
            r.start(r0, (uint32_t)a.stages);
            for (int it = 0; it < nk; ++it) {
                if (!cl_wait(full0 + r.off, r.phase, ctl, a.status)) break;
                tc_fence_after();
                umma_chunk(tmem_base, r.data, d_hi, 2u, r.data + a_lo, d_hi, 2u, a.idesc, (uint32_t)(it != 0), ksteps);
                if (it + a.stages < nk) umma_commit_at(empty0 + r.off);
                if (it + 1 == nk) umma_commit(&ctl->done);
                r.next(r0, (uint32_t)a.stages, stage_lo);
            }
        }
        __syncwarp();
    } else if (present) {
        // ---------------- partial sums to the CTA that finishes the pixel ----------------
        const int q = warp & 3, m = q * 32 + lane;                   // tensor-memory lane quadrant of this warp, its pixel
        const int owner = m / rows;
        const uint32_t dst = map_to_cta(red + (rank * rows + m - owner * rows) * red_pitch(a.BN), (uint32_t)owner);
        bool ok = cl_wait(smem_u32(&ctl->done), 0, ctl, a.status);
        ok = __all_sync(0xffffffffu, ok);
        asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        if (ok) {
            tc_fence_after();
            for (int c = 0; c < a.BN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + c * 32, r);
                tmem_ld_wait();
#pragma unroll
                for (int v = 0; v < 8; ++v) st_remote(dst + c * 128 + v * 16, r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
            }
        }
        tc_fence_before();
    }
    if (warp < 2 || !present) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");   // (the accumulator warps have waited)
    // a CTA that gave up has not sent its sums: no CTA of the cluster stores anything then
    if (ctl->abort_flag != 0) abort_cluster(ctl, a.CS);
    cluster_sync_all();                      // this CTA's pixels have arrived from every CTA
    const bool dead = ctl->abort_flag != 0;
    if (!dead) {
        // ---------------- this CTA's pixels: sums from all ranks, bias, ReLU, bf16, store ----------------
        for (int u = threadIdx.x; u < units; u += kThreadsCl) {
            if (u != (int)threadIdx.x) { mine = unit_of(u); fetch_other(mine); }
            if (!mine.in_map || (!mine.active && !a.add_out)) continue;
            uint4 o;
            if (mine.active) {
                const float* p = red + (u / per_px) * red_pitch(a.BN) + (u % per_px) * 8;
                float4 s0 = *(const float4*)p, s1 = *(const float4*)(p + 4);
                for (int r = 1; r < a.CS; ++r) {
                    p += rows * red_pitch(a.BN);
                    const float4 p0 = *(const float4*)p, p1 = *(const float4*)(p + 4);
                    s0.x += p0.x; s0.y += p0.y; s0.z += p0.z; s0.w += p0.w;
                    s1.x += p1.x; s1.y += p1.y; s1.z += p1.z; s1.w += p1.w;
                }
                float v[8] = {s0.x + mine.b0.x, s0.y + mine.b0.y, s0.z + mine.b0.z, s0.w + mine.b0.w,
                              s1.x + mine.b1.x, s1.y + mine.b1.y, s1.z + mine.b1.z, s1.w + mine.b1.w};
                if (a.relu) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = fmaxf(v[k], 0.f);
                }
                __nv_bfloat162 h[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) h[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                o = *(const uint4*)h;
                *(uint4*)(a.out + mine.at) = o;
            } else {
                o = *(const uint4*)(a.out + mine.at);                // filled from the cache
            }
            if (a.add_out) *(uint4*)(a.add_out + mine.at) = add_bf16x8(o, mine.other, a.add_relu);
        }
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(a.tmem_cols) : "memory");
    }
}

}  // namespace

size_t dc_cluster_smem(int stages, int a_bytes, int b_bytes, int BN)
{
    return (size_t)stages * (a_bytes + b_bytes) + (size_t)128 * red_pitch(BN) * 4 + sizeof(CtlCl) + 1024;
}

static cudaLaunchConfig_t cluster_config(cudaLaunchAttribute* attr, int ctas, int cs, size_t smem, cudaStream_t stream)
{
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)cs; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctas); cfg.blockDim = dim3(kThreadsCl); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cfg;
}

static cudaError_t cluster_smem_opt_in(int device)
{
    static dc_once_per_device attr_set;
    return attr_set.first(device) ? cudaFuncSetAttribute(k_conv_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) : cudaSuccess;
}

int dc_cluster_wave(int device, int cs, size_t smem)
{
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_config(attr, cs, cs, smem, nullptr);
    int n = 0;
    if (cluster_smem_opt_in(device) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, k_conv_cluster, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
    return n;
}

int dc_launch_cluster_kernel(dc_cache* c, const CUtensorMap& tmA, const CUtensorMap& tmB, const dc_cluster_args& a, int tiles)
{
    DC_CUDA(cluster_smem_opt_in(c->device));
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = cluster_config(attr, (tiles < 1 ? 1 : tiles) * a.NB * a.CS, a.CS, dc_cluster_smem(a.stages, a.a_bytes, a.b_bytes, a.BN), c->stream);
    cfg.numAttrs = g_dc_pdl ? 2 : 1;
    DC_CUDA(cudaLaunchKernelEx(&cfg, k_conv_cluster, tmA, tmB, a));
    return DC_OK;
}
