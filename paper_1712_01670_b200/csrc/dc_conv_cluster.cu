// Partial convolution of few tiles: the reduction of one output tile split over a cluster of CTAs.
//
// With one stream a deep layer has one to four 128-pixel tiles and a reduction of thousands: the persistent kernels of
// dc_conv_bf16.cu then run on a handful of SMs, each walking all taps and channels alone (512 -> 512, 3x3 at 7x7: 4 CTAs,
// 72 steps, 32 us).  Here a work item - one tile, a narrow block of BN = 32 or 64 output channels - belongs to a cluster of
// CS = 2, 4 or 8 CTAs.  Each takes 1 / CS of the (tap, channel chunk) steps, operands and MMA as in the tap-by-tap kernel;
// the partial sums meet through distributed shared memory: every CTA leaves its 128 x BN floats in its own shared
// memory, and after a cluster barrier finishes 128 / CS of the pixels from all CS copies, in rank order.  The weights do not
// depend on any kernel before, so their loads start before the wait for the previous layer.
// What bounds it: the chain of latencies of one item (tile list, one TMA round trip, the cluster barrier, the remote
// reads), about 4 us, and no longer the length of the reduction.
//
// An element-wise add that follows (a residual block's end) can be done in the same pass over the tile: reused pixels
// are read back from the output map, where the reuse copy has put them.  Such a launch visits every tile; a tile without
// a pixel to compute skips its loads and MMAs.
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

// Bounded wait, as in dc_conv_bf16.cu.
__device__ __forceinline__ bool cl_wait(void* bar, uint32_t parity, CtlCl* ctl, int32_t* status)
{
    if (mbar_try(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try(bar, parity)) return true;
        if ((spin & 255u) == 0) {
            if (ctl->abort_flag) return false;
            if (now_ns() - t0 > ctl->wait_ns) {
                ctl->abort_flag = 1;
                atomicExch(status, (int)DC_ERR_TIMEOUT);
                return false;
            }
        }
    }
}
__device__ __forceinline__ float4 ld_remote(uint32_t addr)
{
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}
// padded row of partial sums: 16-byte accesses of neighbouring lanes fall in different banks
__host__ __device__ constexpr int red_pitch(int BN) { return BN + 4; }

__global__ void __launch_bounds__(kThreadsCl, 1) k_conv_cluster(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const dc_cluster_args a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* ring = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int stage_bytes = a.a_bytes + a.b_bytes;
    float* red = (float*)(ring + (size_t)a.stages * stage_bytes);            // [128][BN + 4]
    CtlCl* ctl = (CtlCl*)(red + 128 * red_pitch(a.BN));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = (int)cluster_rank(), item = blockIdx.x / a.CS, nb = item % a.NB, idx = item / a.NB;
    const int kiters = a.kh * a.kw * a.kchunks;
    const int k0 = rank * kiters / a.CS, nk = (rank + 1) * kiters / a.CS - k0;

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
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    auto load_weights = [&](int it) {
        const int st = it % a.stages, tap = (k0 + it) / a.kchunks, cc = (k0 + it) - tap * a.kchunks;
        mbar_expect_tx(&ctl->full[st], (uint32_t)a.b_bytes);
        tma_load_2d(ring + (size_t)st * stage_bytes + a.a_bytes, &tmB, tap * a.Ci + cc * a.BK, (nb + a.nb_off) * a.BN, &ctl->full[st]);
    };
    const int early = nk < a.stages ? nk : a.stages;
    if (warp == 0 && lane == 0 && !a.skip_loads)
        for (int it = 0; it < early; ++it) load_weights(it);
    dc_pdl_wait();                           // the previous kernel's output, the tile list and its count are read from here on
    dc_pdl_release();
    const int n_tiles = *a.tile_count;
    const int listed = a.tile_list[idx];     // inside the list's length whatever the count
    const bool present = idx < n_tiles;
    const int tile = present ? listed : 0;

    // this tile's pixels: pixel m is column m % 8 of tile row m / 8
    const int gps = a.Ho * a.gpr, per_stream = a.tiles_x * a.tiles_y;
    int ts = 0, ty = 0, tx = 0;
    if (!a.flat) { ts = tile / per_stream; const int t = tile - ts * per_stream; ty = t / a.tiles_x; tx = t - ty * a.tiles_x; }
    auto locate = [&](int row, int& s, int& y, int& x0) -> bool {             // tile row -> stream, map row, first column
        if (a.flat) {
            const int g = tile * DC_TILE_H + row;
            if (g >= a.n_groups_all) return false;
            s = g / gps;
            const int loc = g - s * gps;
            y = loc / a.gpr; x0 = (loc - y * a.gpr) * DC_TILE_W;
            return true;
        }
        s = ts; y = ty * DC_TILE_H + row; x0 = tx * DC_TILE_W;
        return y < a.Ho;
    };
    // which pixels of a tile row have to be computed
    auto todo_of = [&](int row) -> uint32_t {
        int s, y, x0;
        if (!locate(row, s, y, x0)) return 0u;
        uint32_t m = ~(a.masks[(size_t)tile * 4 + (row >> 2)] >> (8 * (row & 3))) & 0xffu;
        if (a.Wo - x0 < DC_TILE_W) m &= (1u << (a.Wo - x0)) - 1u;
        return m;
    };
    const bool work = present && __any_sync(0xffffffffu, todo_of(lane & 15) != 0);    // the same in all warps of the cluster

    if (warp == 0) {
        // ---------------- producer ----------------
        bool ok = true;
        if (!work) {
            // the weights are on their way: let them land before this CTA's shared memory is given up
            if (lane == 0 && !a.skip_loads)
                for (int it = 0; it < early && ok; ++it) { mbar_arrive(&ctl->full[it]); ok = cl_wait(&ctl->full[it], 0, ctl, a.status); }
        } else if (!a.skip_loads) {
            // 16 x 8 tile: lane 0 brings the window of a tap; flat tiles: lane l brings row piece l
            int fs = 0, fx = 0, fy = 0;
            bool fon = !a.flat && lane == 0;
            if (a.flat) {
                int y, x0;
                fon = lane < DC_TILE_H && locate(lane, fs, y, x0);
                if (fon) { fx = x0 * a.sw - a.pw; fy = y * a.sh - a.ph; }
            } else {
                fs = ts; fx = tx * DC_TILE_W * a.sw - a.pw; fy = ty * DC_TILE_H * a.sh - a.ph;
            }
            const int piece = a.flat ? a.a_bytes / DC_TILE_H : 0;
            const uint32_t a_tx = a.flat ? (uint32_t)__popc(__ballot_sync(0xffffffffu, fon)) * (uint32_t)piece : (uint32_t)a.a_bytes;
            for (int it = 0; it < nk && ok; ++it) {
                const int st = it % a.stages, tap = (k0 + it) / a.kchunks, cc = (k0 + it) - tap * a.kchunks, ky = tap / a.kw, kx = tap - ky * a.kw;
                if (lane == 0) {
                    if (it >= a.stages) {
                        ok = cl_wait(&ctl->empty[st], (uint32_t)(it / a.stages - 1) & 1u, ctl, a.status);
                        if (ok) load_weights(it);
                    }
                    if (ok) mbar_expect_tx(&ctl->full[st], a_tx);
                }
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (ok && fon) tma_load_4d(ring + (size_t)st * stage_bytes + (size_t)lane * piece, &tmA, cc * a.BK, fx + kx, fy + ky, fs, &ctl->full[st]);
            }
        }
        // on an abort: give the copies already issued a bounded chance to land before the CTA exits
        if (!ok && lane == 0) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (lane == 0 && work) {
            const uint64_t dconst = umma_desc(0, a.sbo, a.layout_type);
            const uint32_t ring_lo = smem_u32(ring) >> 4, stage_lo = (uint32_t)stage_bytes >> 4, a_lo = (uint32_t)a.a_bytes >> 4;
            const int ksteps = a.BK / 16;
            bool ok = true;
            for (int it = 0; it < nk && ok; ++it) {
                const int st = it % a.stages;
                ok = cl_wait(&ctl->full[st], (uint32_t)(it / a.stages) & 1u, ctl, a.status);
                if (!ok) break;
                tc_fence_after();
                const uint64_t adesc = dconst + (ring_lo + (uint32_t)st * stage_lo), bdesc = adesc + a_lo;
                for (int kk = 0; kk < ksteps; ++kk) umma_f16(tmem_base, adesc + 2 * kk, bdesc + 2 * kk, a.idesc, (uint32_t)((it | kk) != 0));
                if (it + a.stages < nk) umma_commit(&ctl->empty[st]);
            }
            if (ok) umma_commit(&ctl->done);
        }
        __syncwarp();
    } else if (work) {
        // ---------------- partial sums to shared memory ----------------
        const int q = warp & 3, m = q * 32 + lane;                   // tensor-memory lane quadrant of this warp, its pixel
        const bool ok = cl_wait(&ctl->done, 0, ctl, a.status);
        if (__all_sync(0xffffffffu, ok)) {
            tc_fence_after();
            const uint32_t dst = smem_u32(red + m * red_pitch(a.BN));
            for (int c = 0; c < a.BN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + c * 32, r);
                tmem_ld_wait();
#pragma unroll
                for (int v = 0; v < 8; ++v) sts128(dst + c * 128 + v * 16, r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
            }
        }
        tc_fence_before();
    }
    cluster_sync_all();                      // every CTA's sums are in its shared memory
    const bool dead = ctl->abort_flag != 0;  // an aborted launch's sums are not valid: nothing is stored
    if (present && !dead && (work || a.add_out)) {
        // ---------------- this CTA's pixels: sums of all ranks, bias, ReLU, bf16, store ----------------
        const int rows = 128 / a.CS, per_px = a.BN / 8;
        uint32_t base[8];
#pragma unroll
        for (int r = 0; r < 8; ++r) base[r] = map_to_cta(red, (uint32_t)(r < a.CS ? r : 0));
        for (int u = threadIdx.x; u < rows * per_px; u += kThreadsCl) {
            const int pr = u / per_px, c8 = u - pr * per_px, m = rank * rows + pr, row = m / DC_TILE_W, col = m % DC_TILE_W;
            int s, y, x0;
            if (!locate(row, s, y, x0) || x0 + col >= a.Wo) continue;
            const bool active = (todo_of(row) >> col) & 1u;
            if (!active && !a.add_out) continue;
            const int ch = (nb + a.nb_off) * a.BN + c8 * 8;
            const size_t at = (((size_t)s * a.Ho + y) * a.Wo + x0 + col) * a.Co + ch;
            uint4 o;
            if (active) {
                float v[8];
                const float4 b0 = __ldg((const float4*)(a.bias + ch)), b1 = __ldg((const float4*)(a.bias + ch + 4));
                float4 p0[8], p1[8];
                const uint32_t off = (uint32_t)(m * red_pitch(a.BN) + c8 * 8) * 4u;
#pragma unroll
                for (int r = 0; r < 8; ++r)
                    if (r < a.CS) { p0[r] = ld_remote(base[r] + off); p1[r] = ld_remote(base[r] + off + 16); }
                float4 s0 = p0[0], s1 = p1[0];
#pragma unroll
                for (int r = 1; r < 8; ++r)
                    if (r < a.CS) {
                        s0.x += p0[r].x; s0.y += p0[r].y; s0.z += p0[r].z; s0.w += p0[r].w;
                        s1.x += p1[r].x; s1.y += p1[r].y; s1.z += p1[r].z; s1.w += p1[r].w;
                    }
                v[0] = s0.x + b0.x; v[1] = s0.y + b0.y; v[2] = s0.z + b0.z; v[3] = s0.w + b0.w;
                v[4] = s1.x + b1.x; v[5] = s1.y + b1.y; v[6] = s1.z + b1.z; v[7] = s1.w + b1.w;
                if (a.relu) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = fmaxf(v[k], 0.f);
                }
                __nv_bfloat162 h[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) h[k] = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
                o = *(const uint4*)h;
                *(uint4*)(a.out + at) = o;
            } else {
                o = *(const uint4*)(a.out + at);                     // filled from the cache
            }
            if (a.add_out) {
                const uint4 w = *(const uint4*)(a.add_in + at);
                const uint32_t x[4] = {o.x, o.y, o.z, o.w}, z[4] = {w.x, w.y, w.z, w.w};
                uint32_t r[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {                        // fp32 sum, one rounding to bf16 (as the add layer's own kernel)
                    float lo = __uint_as_float(x[k] << 16) + __uint_as_float(z[k] << 16);
                    float hi = __uint_as_float(x[k] & 0xffff0000u) + __uint_as_float(z[k] & 0xffff0000u);
                    if (a.add_relu) { lo = fmaxf(lo, 0.f); hi = fmaxf(hi, 0.f); }
                    const __nv_bfloat162 t = __floats2bfloat162_rn(lo, hi);
                    r[k] = *(const uint32_t*)&t;
                }
                *(uint4*)(a.add_out + at) = make_uint4(r[0], r[1], r[2], r[3]);
            }
        }
    }
    cluster_sync_all();                      // nobody leaves while its sums may still be read
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

int dc_launch_cluster_kernel(dc_cache* c, const CUtensorMap& tmA, const CUtensorMap& tmB, const dc_cluster_args& a, int tiles)
{
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) DC_CUDA(cudaFuncSetAttribute(k_conv_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((tiles < 1 ? 1 : tiles) * a.NB * a.CS)); cfg.blockDim = dim3(kThreadsCl); cfg.stream = c->stream;
    cfg.dynamicSmemBytes = dc_cluster_smem(a.stages, a.a_bytes, a.b_bytes, a.BN);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)a.CS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = g_dc_pdl ? 2 : 1;
    DC_CUDA(cudaLaunchKernelEx(&cfg, k_conv_cluster, tmA, tmB, a));
    return DC_OK;
}
