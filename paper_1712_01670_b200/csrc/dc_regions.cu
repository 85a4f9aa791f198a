// Region propagation (Section 5, Table 2) and the reuse step of the cache-aware convolution
// (Section 5, "Reuse": copy cached regions, build the bitmap, list what is left to compute).
//
//   k_propagate      four lanes per (stream, rectangle slot) walk the layer table in order and
//                    leave the rectangle's image after every layer; a vanished rectangle is all zeros.
//   k_classify_copy  one warp per 16x8 output tile: lanes test the stream's rectangles against
//                    the tile, OR their coverage into a 128-bit bitmap, the warp copies each
//                    covered row span from the cached map with bulk copies (global -> shared ->
//                    global through the copy engine, no registers), and tiles that still hold
//                    uncovered pixels are appended to the layer's dirty list.
#include "dc_common.cuh"

namespace {

__device__ __forceinline__ int floor_div(int a, int b)
{
    int q = a / b, r = a - q * b;
    return (r != 0 && ((r < 0) != (b < 0))) ? q - 1 : q;
}
__device__ __forceinline__ int ceil_div(int a, int b) { return -floor_div(-a, b); }

// Sliding window on one axis: output o reads [o s - p, o s - p + k - 1]; reusable iff that lies
// inside [x, x + w).  First = ceil((x + p) / s) as printed in Table 2; last = floor((x + w - k + p) / s).
__device__ __forceinline__ void erode_axis(int x, int w, int k, int s, int p, int& xo, int& wo)
{
    if (s == 1) { xo = x + p; wo = w - k + 1; return; }
    int first = ceil_div(x + p, s), last = floor_div(x + w - k + p, s);
    xo = first; wo = last - first + 1;
}
// Area resize n_in -> n_out: output o averages [floor(o n_in / n_out), ceil((o + 1) n_in / n_out) - 1].
__device__ __forceinline__ void resize_axis(int x, int w, int n_in, int n_out, int& xo, int& wo)
{
    int first, last;
    if (n_in <= 32768 && n_out <= 32768 && (unsigned)x <= 32768u && (unsigned)w <= 32768u) {      // the products fit 32 bits
        first = (int)(((unsigned)x * (unsigned)n_out + (unsigned)n_in - 1u) / (unsigned)n_in);
        last = (int)((unsigned)(x + w) * (unsigned)n_out / (unsigned)n_in) - 1;
    } else {
        first = (int)(((long long)x * n_out + n_in - 1) / n_in);
        last = (int)(((long long)(x + w) * n_out) / n_in) - 1;
    }
    xo = first; wo = last - first + 1;
}

__device__ __forceinline__ dc_region empty_region() { dc_region e = {0, 0, 0, 0, 0, 0}; return e; }

// A layer as propagation sees it, the fields of the horizontal axis and of the vertical one side by side.
// axis[]: {c1, c2, sh, simple}.  The rule of a sliding window whose strides are powers of two (convolutions, pooling; LRN is one at stride 1,
// ReLU one of a single pixel) is, on either axis, first = (x + c1) >> sh, last = (x + w + c2) >> sh.  simple: such a window on the layer
// before.
// links: {in0, in1, kind, until}; kind: kWindow or the layer's; until: the last layer that reads this one's rectangle, kept (later than the
// next one), and at least the last layer that reads the frame's.
// rule[]: for the rules that are no such window: {kernel, stride, padding, -}, resize {input, output, -, -}.
constexpr int kWindow = -1;
constexpr int kLanes = 4;                                  // lanes per rectangle
constexpr size_t kWalkBytes = 160 * 1024;                  // shared memory for the rectangles of a batch at all layers
struct __align__(16) PropLayer { int4 axis[2], links, rule[2]; };

// A lane's share of a rectangle: where it starts and how long it is on one axis, in the frame (lanes 0: x, 1: y of the four) or in the
// cached map (2: x, 3: y).  The two shares of an axis have the same length.  A vanished rectangle is all zeros.
struct Span { int at, len; };

__device__ __forceinline__ Span window_rule(int4 ax, Span a)
{
    Span o;
    o.at = (a.at + ax.x) >> ax.z;
    o.len = ((a.at + a.len + ax.y) >> ax.z) - o.at + 1;
    return o;
}
// The same for every other layer, the same one in all lanes of the warp.
__device__ Span general_rule(const PropLayer& L, int lane, Span a, Span b)
{
    const unsigned all = 0xffffffffu;
    const int4 z = L.rule[lane & 1];
    Span o = {0, 0};
    switch (L.links.z) {
    case kWindow: o = window_rule(L.axis[lane & 1], a); break;
    case DC_CONV: case DC_MAXPOOL: erode_axis(a.at, a.len, z.x, z.y, z.z, o.at, o.len); break;
    case DC_RESIZE_AREA: resize_axis(a.at, a.len, z.x, z.y, o.at, o.len); break;
    case DC_ADD: case DC_CONCAT: {
        // the overlapped region; both inputs must agree on the displacement, on both axes
        const int da = __shfl_xor_sync(all, a.at, 2) - a.at, db = __shfl_xor_sync(all, b.at, 2) - b.at;
        const unsigned same = __ballot_sync(all, da == db) >> (lane & ~3);
        o.at = max(a.at, b.at);
        o.len = (same & 3u) == 3u && b.len > 0 ? min(a.at + a.len, b.at + b.len) - o.at : 0;
        break;
    }
    case DC_FC: break;
    default: o = a;
    }
    return o;
}

// The CTAs of a stream take batches of as many rectangles as have room in shared memory at all layers, in turns where there are more batches.
// First the walk, four lanes per rectangle: the two axes of the rectangle and of its cached image, which only meet where their
// lengths are compared.  It leaves its rectangles in shared memory and does nothing else, because what bounds it is the chain of a lane's
// instructions from layer to layer.  A warp whose rectangles have all vanished, those that later layers read too, stops.  Then all warps write
// the table and the lists.
// us for ResNet-50's 71 layers, one stream: a thread per rectangle that also wrote the table and asked for its places in the lists layer
// by layer 26, so 11.
// alive, live: how many rectangles are left at each layer and stream, and these alone, in any order (they are disjoint): most of a
// frame's erode within a few layers, and the reuse step tests every tile against all it is given.
// FRAME: the rectangles of a frame: lists and counts are wanted, the counters of the reuse step are zeroed; table (every slot at every layer) or
// NULL.  SHARED: several CTAs per stream; where a frame's rectangles are more than a batch, they ask for their places in the lists in `places` ([n_layers][S], then a ticket per
// stream), and the last of them moves the counts to `alive` and leaves zeros behind.  Else a caller's list: out, n_out, or NULL: copies of layers out_begin .. layer_end - 1 and of the counts.
// walkers: threads that walk (a multiple of 32); dynamic shared memory: 8 * layer_end * walkers bytes.
template <bool FRAME, bool SHARED>
__global__ void __launch_bounds__(1024) k_propagate(const PropLayer* layers, int layer_end, int n_layers, int S, int max_regions, int walkers,
                                                   const dc_region* in, const int32_t* n_in, dc_region* table, dc_region* live, int32_t* alive, int32_t* reuse_px,
                                                   int32_t* dirty_count, int32_t* places, dc_region* out, int out_begin, int32_t* n_out)
{
    __shared__ PropLayer sl[DC_MAX_LAYERS];
    __shared__ int32_t count[DC_MAX_LAYERS], end_of[32], last;   // end_of: per walking warp, the layer at which it stopped
    extern __shared__ __align__(16) int32_t at_all[];      // [layer_end][walkers], then the lengths likewise
    const unsigned all = 0xffffffffu;
    const int s = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, per_batch = walkers / kLanes;
    int32_t* const len_all = at_all + layer_end * walkers;
    for (int i = tid; i < layer_end * (int)(sizeof(PropLayer) / 16); i += nt) ((int4*)sl)[i] = __ldg((const int4*)layers + i);
    if (tid < DC_MAX_LAYERS) count[tid] = 0;
    dc_pdl_wait();
    dc_pdl_release();
    const int n = min(n_in[s], max_regions);              // a caller's count beyond the table is cut, never written
    // a caller's list has zeros behind its rectangles
    const int rows = !FRAME && out ? max_regions : n;
    const size_t layer_stride = (size_t)S * max_regions;
    const bool out_aligned = (uintptr_t)out % 8 == 0;     // a caller's array may lie at any word
    const bool shared_lists = SHARED && n > per_batch;
    if (SHARED && blockIdx.y > 0 && (int)blockIdx.y * per_batch >= n) return;
    for (int first = blockIdx.y * per_batch; first < rows; first += gridDim.y * per_batch) {
        const int i = first + tid / kLanes;
        Span r0 = {0, 0};
        if (tid < walkers && i < n) {
            const int32_t* r = (const int32_t*)(in + (size_t)s * max_regions + i);
            r0.at = r[lane & 2 ? 4 + (lane & 1) : lane & 1]; r0.len = r[2 + (lane & 1)];
        }
        __syncthreads();                                   // the layer table; the batch before has been written
        if (tid < walkers) {
            const int group = lane & ~3, axis = lane & 1;
            int l = 0, until = sl[0].links.w;
            int32_t* at = at_all + tid; int32_t* len = len_all + tid;
            Span a = r0;
            unsigned living = __ballot_sync(all, a.len > 0);
            int4 ax = sl[0].axis[axis];
            // no later layer reads what is left, or nothing is left at all
            for (; l < layer_end && (living != 0 || l <= until); ++l, at += walkers, len += walkers) {
                const int4 ax1 = ax;
                const int until1 = sl[l].links.w;
                ax = sl[min(l + 1, layer_end - 1)].axis[axis];
                Span o;
                if (ax1.w) o = window_rule(ax1, a);
                else {
                    const PropLayer& L = sl[l];
                    auto fetch = [&](int from) -> Span {
                        if (from == l - 1 && l > 0) return a;
                        if (from < 0) return r0;
                        return Span{at_all[from * walkers + tid], len_all[from * walkers + tid]};
                    };
                    const Span b = L.links.z == DC_ADD || L.links.z == DC_CONCAT ? fetch(L.links.y) : Span{0, 0};
                    a = fetch(L.links.x);
                    o = general_rule(L, lane, a, b);
                }
                // the cached side on its own; smaller size wins; nothing is left unless something is on both axes
                o.len = min(o.len, __shfl_xor_sync(all, o.len, 2));
                const unsigned some = __ballot_sync(all, o.len > 0 && a.len > 0);
                living = some & (some >> 1) & 0x11111111u;
                const bool on = (living >> group) & 1u;
                a.at = on ? o.at : 0; a.len = on ? o.len : 0;
                *at = a.at; *len = a.len;
                if (living) until = max(until, until1);
            }
            if (lane == 0) end_of[warp] = l;
        }
        __syncthreads();
        const int here = min(per_batch, rows - first), runs = (here + 31) >> 5;
        // rectangle k of the batch at layer l
        auto fetch = [&](int l, int k, int2& at, int2& len, int2& src) {
            at = len = src = make_int2(0, 0);
            if (k < here && l < end_of[k >> 3]) {
                const int32_t* p = at_all + l * walkers + k * kLanes;
                at = *(const int2*)p; src = *(const int2*)(p + 2);
                len = *(const int2*)(len_all + l * walkers + k * kLanes);
            }
        };
        auto put = [](dc_region* to, int2 at, int2 len, int2 src) { int2* t = (int2*)to; t[0] = at; t[1] = len; t[2] = src; };    // 8-byte aligned
        if constexpr (FRAME) {
            // a layer per warp, a rectangle per lane
            for (int l = warp; l < layer_end; l += nt >> 5) {
                const size_t row = l * layer_stride + (size_t)s * max_regions;
                int listed = count[l];
                int2 at, len, src;
                if (shared_lists) {
                    int total = 0;
                    for (int k0 = 0; k0 < here; k0 += 32) { fetch(l, k0 + lane, at, len, src); total += __popc(__ballot_sync(all, len.x > 0)); }
                    if (lane == 0 && total) listed = atomicAdd(&places[l * S + s], total);
                    listed = __shfl_sync(all, listed, 0);
                }
                for (int k0 = 0; k0 < here; k0 += 32) {
                    const int k = k0 + lane;
                    fetch(l, k, at, len, src);
                    if (table && k < here) put(table + row + first + k, at, len, src);
                    const unsigned m = __ballot_sync(all, len.x > 0);
                    if (len.x > 0) put(live + row + listed + __popc(m & ((1u << lane) - 1u)), at, len, src);
                    listed += __popc(m);
                }
                if (lane == 0 && !shared_lists) count[l] = listed;
            }
        } else {
            // 32 rectangles of a layer per warp, a rectangle per lane
#pragma unroll 1
            for (int u = warp; u < layer_end * runs; u += nt >> 5) {
                const int l = u / runs, k = (u - l * runs) * 32 + lane;
                const size_t row = l * layer_stride + (size_t)s * max_regions;
                int2 at, len, src;
                fetch(l, k, at, len, src);
                if (k >= here) continue;
                put(table + row + first + k, at, len, src);
                if (!out || l < out_begin) continue;
                dc_region* o = out + (row - out_begin * layer_stride + first + k);
                if (out_aligned) put(o, at, len, src);
                else *o = dc_region{at.x, at.y, len.x, len.y, src.x, src.y};
            }
        }
    }
    if (shared_lists) {
        __syncthreads();
        if (tid == 0) {
            const int sharers = min((n + per_batch - 1) / per_batch, (int)gridDim.y);    // CTAs that have rectangles
            __threadfence();                               // behind the barrier: for what all warps have added
            last = atomicAdd(&places[n_layers * S + s], 1) == sharers - 1;
            __threadfence();
        }
        __syncthreads();
        if (!last) return;
        if (tid < layer_end) { count[tid] = __ldcg(&places[tid * S + s]); places[tid * S + s] = 0; }
        if (tid == 0) places[n_layers * S + s] = 0;
    }
    if (!FRAME && n_out && blockIdx.y == 0) for (int l = out_begin + tid; l < layer_end; l += nt) n_out[(l - out_begin) * S + s] = n_in[s];
    if (FRAME) {
        __syncthreads();
        for (int l = tid; l < n_layers; l += nt) {
            alive[l * S + s] = l < layer_end ? count[l] : 0;
            reuse_px[l * S + s] = 0;
            if (s == 0) dirty_count[l] = 0;
        }
    }
}

// ---- bulk copies (cp.async.bulk) for the reuse copy ----
#ifndef DC_COPY_WARPS
#define DC_COPY_WARPS 8
#endif
#ifndef DC_COPY_SEG
#define DC_COPY_SEG 256
#endif
constexpr int kCopyWarps = DC_COPY_WARPS;        // warps per CTA
constexpr int kSeg = DC_COPY_SEG;                // bytes one lane moves per round; a row span is cut into such segments
constexpr int kStageBytes = 32 * kSeg;           // staging of one warp: one segment per lane
constexpr size_t kCopySmem = (size_t)kCopyWarps * kStageBytes + 128 + kCopyWarps * sizeof(unsigned long long);
constexpr unsigned long long kCopyWaitNs = 2000000000ull;   // a warp gives up on its staging barrier after 2 s (far beyond any copy)

__device__ __forceinline__ uint32_t rs_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void rs_bar_init(void* bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(rs_smem(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void rs_expect(void* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(rs_smem(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool rs_try(void* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(rs_smem(bar)), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void rs_load(void* dst_smem, const void* src, uint32_t bytes, void* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(rs_smem(dst_smem)), "l"(src), "r"(bytes), "r"(rs_smem(bar)) : "memory");
}
__device__ __forceinline__ void rs_store(void* dst, const void* src_smem, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(rs_smem(src_smem)), "r"(bytes) : "memory");
}
__device__ __forceinline__ unsigned long long rs_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Bounded wait for a phase of the staging barrier; false when the limit passed.
__device__ __forceinline__ bool rs_wait(void* bar, uint32_t parity)
{
    if (rs_try(bar, parity)) return true;
    const unsigned long long t0 = rs_now();
    for (unsigned spin = 1;; ++spin) {
        if (rs_try(bar, parity)) return true;
        if ((spin & 255u) == 0 && rs_now() - t0 > kCopyWaitNs) return false;
    }
}
__device__ __forceinline__ void rs_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void rs_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void rs_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// What a warp needs for its bulk copies: its staging (32 segments), one mbarrier and its phase.
struct CopyLane { uint8_t* stage; unsigned long long* bar; uint32_t phase; bool dead; };

struct ClassifyArgs {
    const dc_region* regions; const int32_t* n_regions; int max_regions;
    const uint8_t* prev; uint8_t* out;           // maps as bytes
    int Ho, Wo, px_bytes;                        // px_bytes = cout * element size (multiple of 16)
    int tiles_x, tiles_y, S;
    int gpr, gpt, n_tiles;                       // gpr > 0: flat tiles of gpt (up to 16) groups of 8 pixels, gpr groups per image row; n_tiles: tiles in all
    uint32_t* masks; int32_t* dirty_list; int32_t* dirty_count; int32_t* reuse_px;
    const int32_t* alive;                        // per stream: rectangles alive at this layer, or NULL (unknown)
    unsigned long long* reused_total;
    int32_t* status;                             // device status word
    int parts;                                   // warps that share a tile's copies (each tests the rectangles, the first one records the outcome)
    // A caller's launch counts by itself, whatever ran before it (it may be a node of a graph that is launched many times): the
    // running counter holds finished tiles above dirty ones, the last tile moves the sum to dirty_count and leaves zero.  (A
    // ticket per CTA in an atomic of its own behind the count: 2 us longer.)  Else NULL: dirty_count was zeroed by the frame's
    // region propagation and counts directly.
    unsigned long long* running;
};

__device__ __forceinline__ void record_tile(const ClassifyArgs& a, int tile, bool dirty)
{
    if (!a.running) {
        if (dirty) a.dirty_list[atomicAdd(a.dirty_count, 1)] = tile;
        return;
    }
    const unsigned long long before = atomicAdd(a.running, (1ull << 32) | (dirty ? 1u : 0u));
    const int slot = (int)(uint32_t)before;
    if (dirty) a.dirty_list[slot] = tile;
    if ((int)(before >> 32) == a.n_tiles - 1) { *a.dirty_count = slot + (dirty ? 1 : 0); *a.running = 0; }
}

__device__ __forceinline__ void classify_tile(const ClassifyArgs& a, const int tile, const int part, const int lane, CopyLane& cl)
{
    const int per = a.tiles_x * a.tiles_y;
    const int s = tile / per, t = tile - s * per, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
    const int X0 = tx * DC_TILE_W, Y0 = ty * DC_TILE_H;
    const int X1 = min(X0 + DC_TILE_W, a.Wo), Y1 = min(Y0 + DC_TILE_H, a.Ho);
    const dc_region* regs = a.regions + (size_t)s * a.max_regions;
    // the first rectangles of a frame travel with their number; of a caller's list no more is read than that says
    dc_region first = empty_region();
    if (a.alive && lane < a.max_regions) first = regs[lane];
    // every rectangle of this stream has eroded away before this layer: nothing to test or copy
    const int n = (a.alive && a.alive[s] == 0) ? 0 : min(a.n_regions[s], a.max_regions);
    const size_t map_base = (size_t)s * a.Ho * a.Wo * a.px_bytes;
    uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;      // bit (row * DC_TILE_W + col) of the tile, row-major
    for (int base = 0; base < n; base += 32) {
        int i = base + lane;
        dc_region r = empty_region();
        int ix0 = 0, ix1 = 0, iy0 = 0, iy1 = 0;
        if (i < n) {
            r = a.alive && base == 0 ? first : regs[i];
            // Rectangles made by Step 5 and Table 2 lie inside the map on both sides.  One that does not (a caller's
            // own list) is not reused: neither side is ever addressed outside its map; the status word records it.
            const bool inside = r.x >= 0 && r.y >= 0 && r.sx >= 0 && r.sy >= 0 && r.w <= a.Wo && r.h <= a.Ho &&
                                r.x <= a.Wo - r.w && r.y <= a.Ho - r.h && r.sx <= a.Wo - r.w && r.sy <= a.Ho - r.h;
            if (r.w <= 0 || r.h <= 0) r = empty_region();
            else if (!inside) {
                if (t == 0 && a.status) atomicExch(a.status, (int)DC_ERR_ARG);
                r = empty_region();
            }
            ix0 = max(r.x, X0); ix1 = min(r.x + r.w, X1);
            iy0 = max(r.y, Y0); iy1 = min(r.y + r.h, Y1);
        }
        bool hit = ix1 > ix0 && iy1 > iy0;
        if (hit) {
            const uint32_t rowbits = ((1u << (ix1 - X0)) - 1u) & ~((1u << (ix0 - X0)) - 1u);   // DC_TILE_W-bit row pattern
            for (int y = iy0; y < iy1; ++y) {
                const int bit = DC_TILE_BIT(y - Y0, 0);
                const uint32_t v = rowbits << (bit & 31);
                switch (bit >> 5) { case 0: m0 |= v; break; case 1: m1 |= v; break; case 2: m2 |= v; break; default: m3 |= v; }
            }
        }
        // Section 5 "Reuse", step 1.  Inside the tile a rectangle is (iy1 - iy0) row spans, each contiguous in both maps
        // (all channels of ix1 - ix0 pixels).  Spans are cut into segments of kSeg bytes, and the segments of all the
        // rectangles that hit are numbered through: per round every lane moves one of them, a bulk copy into the warp's
        // staging, then a bulk copy out to the new map, so that a tile with several small rectangles costs one round
        // trip and not one per rectangle.  Addresses and sizes are multiples of 16 bytes (px_bytes is).
        unsigned hits = __ballot_sync(0xffffffffu, hit);
        if (hits == 0) continue;
        const int span_bytes = hit ? (ix1 - ix0) * a.px_bytes : 0;
        const int segs = (span_bytes + kSeg - 1) / kSeg, mine = hit ? (iy1 - iy0) * segs : 0;
        int begin = mine;                                               // inclusive sum over the lanes, then this lane's start
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, begin, o); if (lane >= o) begin += v; }
        const int items = __shfl_sync(0xffffffffu, begin, 31);
        begin -= mine;
        const int src_y = iy0 - r.y + r.sy, src_x = ix0 - r.x + r.sx;   // cached position of (ix0, iy0)
        for (int i0 = part * 32; i0 < items && !cl.dead; i0 += 32 * a.parts) {
            const int it = i0 + lane;
            const bool on = it < items;
            int owner = 0;                                              // the lane whose rectangle segment `it` belongs to
            for (unsigned h = hits; h; h &= h - 1) {
                const int k = __ffs(h) - 1;
                if (it >= __shfl_sync(0xffffffffu, begin, k)) owner = k;
            }
            const int o_first = __shfl_sync(0xffffffffu, begin, owner), o_segs = max(1, __shfl_sync(0xffffffffu, segs, owner));
            const int o_span = __shfl_sync(0xffffffffu, span_bytes, owner);
            const int o_x = __shfl_sync(0xffffffffu, ix0, owner), o_y = __shfl_sync(0xffffffffu, iy0, owner);
            const int o_sx = __shfl_sync(0xffffffffu, src_x, owner), o_sy = __shfl_sync(0xffffffffu, src_y, owner);
            const int loc = it - o_first, row = loc / o_segs, sg = loc - row * o_segs;
            const uint32_t bytes = on ? (uint32_t)min(kSeg, o_span - sg * kSeg) : 0u;
            const size_t seg_off = (size_t)sg * kSeg;
            const uint8_t* src = a.prev + map_base + ((size_t)(o_sy + row) * a.Wo + o_sx) * a.px_bytes + seg_off;
            uint8_t* dst = a.out + map_base + ((size_t)(o_y + row) * a.Wo + o_x) * a.px_bytes + seg_off;
            const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
            if (lane == 0) rs_expect(cl.bar, total);
            __syncwarp();
            if (on) rs_load(cl.stage + lane * kSeg, src, bytes, cl.bar);
            const bool landed = rs_wait(cl.bar, cl.phase);
            if (!__all_sync(0xffffffffu, landed)) {                     // never seen; leave rather than spin for ever
                if (lane == 0 && a.status) atomicExch(a.status, (int)DC_ERR_TIMEOUT);
                cl.dead = true;
                break;
            }
            cl.phase ^= 1u;
            if (on) rs_store(dst, cl.stage + lane * kSeg, bytes);
            rs_commit();
            rs_wait_read();                                             // staging may be overwritten by the next round
            __syncwarp();
        }
    }
    m0 = __reduce_or_sync(0xffffffffu, m0); m1 = __reduce_or_sync(0xffffffffu, m1);
    m2 = __reduce_or_sync(0xffffffffu, m2); m3 = __reduce_or_sync(0xffffffffu, m3);
    if (lane == 0 && part == 0) {
        uint32_t* mk = a.masks + (size_t)tile * 4;
        mk[0] = m0; mk[1] = m1; mk[2] = m2; mk[3] = m3;
        int covered = __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3);
        int in_tile = (X1 - X0) * (Y1 - Y0);
        if (covered) { atomicAdd(&a.reuse_px[s], covered); atomicAdd(a.reused_total, (unsigned long long)covered); }
        record_tile(a, tile, covered < in_tile);
    }
}


// The same for a layer with flat tiles: row i of the tile's bitmap is group tile * gpt + i, a group being 8 pixels of
// one image row, numbered (stream * Ho + y) * gpr + column group.  A tile may hold groups of several streams (small
// maps); each stream's rectangles are tested against that stream's groups only.
__device__ __forceinline__ void classify_tile_flat(const ClassifyArgs& a, const int tile, const int part, const int lane, CopyLane& cl)
{
    const int gps = a.Ho * a.gpr;                                  // groups per stream
    const int G0 = tile * a.gpt, G1 = min(G0 + a.gpt, a.S * gps);
    uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;
    int in_tile;
    {   // pixels of the tile that exist: a row's last group may be cut by the map's width
        const int g = G0 + lane, loc = g % gps, gx = loc % a.gpr;
        in_tile = __reduce_add_sync(0xffffffffu, g < G1 ? min(DC_TILE_W, a.Wo - gx * DC_TILE_W) : 0);
    }
    const int segs_max = (DC_TILE_W * a.px_bytes + kSeg - 1) / kSeg;   // segments of a whole group's pixels
    for (int s = G0 / gps; s * gps < G1; ++s) {
        const int g_lo = max(G0, s * gps), g_hi = min(G1, (s + 1) * gps);     // this stream's groups in the tile
        const int loc0 = g_lo - s * gps, y_first = loc0 / a.gpr, gx_first = loc0 - y_first * a.gpr;
        const dc_region* regs = a.regions + (size_t)s * a.max_regions;
        const int n = (a.alive && a.alive[s] == 0) ? 0 : min(a.n_regions[s], a.max_regions);
        const size_t map_base = (size_t)s * a.Ho * a.Wo * a.px_bytes;
        uint32_t s0 = 0, s1 = 0, s2 = 0, s3 = 0;                  // this stream's part of the bitmap
        for (int base = 0; base < n; base += 32) {
            const int i = base + lane;
            dc_region r = empty_region();
            uint32_t hit16 = 0;                                   // rows of the tile that the rectangle touches
            if (i < n) {
                r = regs[i];
                const bool inside = r.x >= 0 && r.y >= 0 && r.sx >= 0 && r.sy >= 0 && r.w <= a.Wo && r.h <= a.Ho &&
                                    r.x <= a.Wo - r.w && r.y <= a.Ho - r.h && r.sx <= a.Wo - r.w && r.sy <= a.Ho - r.h;
                if (r.w <= 0 || r.h <= 0) r = empty_region();
                else if (!inside) {                               // see classify_tile
                    if (loc0 == 0 && a.status) atomicExch(a.status, (int)DC_ERR_ARG);
                    r = empty_region();
                }
                if (r.w > 0) {
                    int y = y_first, gx = gx_first;
                    for (int g = g_lo; g < g_hi; ++g) {
                        const int x0 = gx * DC_TILE_W;
                        const int cx0 = max(r.x, x0), cx1 = min(r.x + r.w, min(x0 + DC_TILE_W, a.Wo));
                        if (y >= r.y && y < r.y + r.h && cx1 > cx0) {
                            const int row = g - G0;
                            const uint32_t v = (((1u << (cx1 - x0)) - 1u) & ~((1u << (cx0 - x0)) - 1u)) << ((row & 3) * DC_TILE_W);
                            switch (row >> 2) { case 0: s0 |= v; break; case 1: s1 |= v; break; case 2: s2 |= v; break; default: s3 |= v; }
                            hit16 |= 1u << row;
                        }
                        if (++gx == a.gpr) { gx = 0; ++y; }
                    }
                }
            }
            // the warp copies every touched row's span together (Section 5 "Reuse", step 1): per round one segment per lane
            unsigned hits = __ballot_sync(0xffffffffu, hit16 != 0);
            while (hits) {
                const int src_lane = __ffs(hits) - 1; hits &= hits - 1;
                const int rx = __shfl_sync(0xffffffffu, r.x, src_lane), ry = __shfl_sync(0xffffffffu, r.y, src_lane);
                const int rw = __shfl_sync(0xffffffffu, r.w, src_lane);
                const int rsx = __shfl_sync(0xffffffffu, r.sx, src_lane), rsy = __shfl_sync(0xffffffffu, r.sy, src_lane);
                const uint32_t h16 = __shfl_sync(0xffffffffu, hit16, src_lane);
                for (int i0 = part * 32; i0 < DC_TILE_H * segs_max && !cl.dead; i0 += 32 * a.parts) {
                    const int it = i0 + lane, row = it / segs_max, sg = it - row * segs_max;
                    uint32_t bytes = 0;
                    size_t src_off = 0, dst_off = 0;
                    if (row < DC_TILE_H && ((h16 >> row) & 1u)) {
                        const int loc = G0 + row - s * gps, y = loc / a.gpr, x0 = (loc - y * a.gpr) * DC_TILE_W;
                        const int cx0 = max(rx, x0), cx1 = min(rx + rw, min(x0 + DC_TILE_W, a.Wo));
                        const int span = (cx1 - cx0) * a.px_bytes - sg * kSeg;
                        if (span > 0) {
                            bytes = (uint32_t)min(kSeg, span);
                            src_off = ((size_t)(y - ry + rsy) * a.Wo + (cx0 - rx + rsx)) * a.px_bytes + (size_t)sg * kSeg;
                            dst_off = ((size_t)y * a.Wo + cx0) * a.px_bytes + (size_t)sg * kSeg;
                        }
                    }
                    const uint32_t total = __reduce_add_sync(0xffffffffu, bytes);
                    if (total == 0) continue;                     // the same in all lanes
                    if (lane == 0) rs_expect(cl.bar, total);
                    __syncwarp();
                    if (bytes) rs_load(cl.stage + lane * kSeg, a.prev + map_base + src_off, bytes, cl.bar);
                    const bool landed = rs_wait(cl.bar, cl.phase);
                    if (!__all_sync(0xffffffffu, landed)) {
                        if (lane == 0 && a.status) atomicExch(a.status, (int)DC_ERR_TIMEOUT);
                        cl.dead = true;
                        break;
                    }
                    cl.phase ^= 1u;
                    if (bytes) rs_store(a.out + map_base + dst_off, cl.stage + lane * kSeg, bytes);
                    rs_commit();
                    rs_wait_read();
                    __syncwarp();
                }
            }
        }
        s0 = __reduce_or_sync(0xffffffffu, s0); s1 = __reduce_or_sync(0xffffffffu, s1);
        s2 = __reduce_or_sync(0xffffffffu, s2); s3 = __reduce_or_sync(0xffffffffu, s3);
        const int covered_s = __popc(s0) + __popc(s1) + __popc(s2) + __popc(s3);
        if (lane == 0 && part == 0 && covered_s) { atomicAdd(&a.reuse_px[s], covered_s); atomicAdd(a.reused_total, (unsigned long long)covered_s); }
        m0 |= s0; m1 |= s1; m2 |= s2; m3 |= s3;
    }
    if (lane == 0 && part == 0) {
        uint32_t* mk = a.masks + (size_t)tile * 4;
        mk[0] = m0; mk[1] = m1; mk[2] = m2; mk[3] = m3;
        record_tile(a, tile, __popc(m0) + __popc(m1) + __popc(m2) + __popc(m3) < in_tile);
    }
}

// Staging and barrier of this warp, carved from the CTA's dynamic shared memory.
__device__ __forceinline__ CopyLane copy_lane_setup(uint8_t* smem_raw)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    CopyLane cl;
    cl.stage = base + (size_t)warp * kStageBytes;
    cl.bar = (unsigned long long*)(base + (size_t)kCopyWarps * kStageBytes) + warp;
    cl.phase = 0; cl.dead = false;
    if (lane == 0) rs_bar_init(cl.bar);
    __syncwarp();
    return cl;
}

__global__ void __launch_bounds__(kCopyWarps * 32) k_classify_copy(ClassifyArgs a)
{
    extern __shared__ uint8_t copy_smem[];
    CopyLane cl = copy_lane_setup(copy_smem);
    dc_pdl_wait();
    dc_pdl_release();
    const int w = blockIdx.x * kCopyWarps + (threadIdx.x >> 5), tile = w / a.parts, part = w - tile * a.parts;
    if (tile < a.n_tiles) {
        if (a.gpr > 0) classify_tile_flat(a, tile, part, threadIdx.x & 31, cl);
        else classify_tile(a, tile, part, threadIdx.x & 31, cl);
    }
    rs_wait_all();
}

// Every cached layer of a frame in one launch: the bitmaps, reuse copies and dirty lists of a layer depend only
// on the rectangles (known once propagation has run) and on the layer's own cached map, not on the layers before it.
// Warps are numbered through all layers' tiles; first_warp is the running sum.
struct ClassifyLayer {
    const dc_region* regions; uint8_t* map[2];
    int Ho, Wo, px_bytes, tiles_x, tiles_y, first_warp, gpr, gpt, parts;
    uint32_t* masks; int32_t* dirty_list; int32_t* dirty_count; int32_t* reuse_px;
    const int32_t* alive; unsigned long long* reused_total; int32_t* status;
};

__global__ void __launch_bounds__(kCopyWarps * 32) k_classify_copy_all(const ClassifyLayer* layers, int n_cached, int total_warps,
                                                                       int max_regions, int S, int cur)
{
    extern __shared__ uint8_t copy_smem[];
    CopyLane cl = copy_lane_setup(copy_smem);
    // Both match sets' tables were complete when the cache was created (dc_cache_create waits for them): a warp finds its layer and tile while the kernel before still runs (half a dozen
    // loads one behind another; a pass in us before and so: small CNN, one
    // stream, 86.4 and 85.8; every layer kind, 16 streams, 162.2 and 160.6).
    const int w = blockIdx.x * kCopyWarps + (threadIdx.x >> 5);
    int lo = 0, hi = n_cached - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (__ldg(&layers[mid].first_warp) <= w) lo = mid; else hi = mid - 1;
    }
    const ClassifyLayer& L = layers[lo];
    ClassifyArgs a;
    a.regions = L.regions; a.n_regions = L.alive; a.max_regions = max_regions;     // the rectangles left at this layer
    const uint8_t* const m0 = L.map[0]; const uint8_t* const m1 = L.map[1];
    a.prev = cur ? m1 : m0; a.out = (uint8_t*)(cur ? m0 : m1);
    a.Ho = L.Ho; a.Wo = L.Wo; a.px_bytes = L.px_bytes; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y; a.S = S;
    a.gpr = L.gpr; a.gpt = L.gpt; a.n_tiles = 0;
    a.masks = L.masks; a.dirty_list = L.dirty_list; a.dirty_count = L.dirty_count; a.reuse_px = L.reuse_px;
    a.alive = L.alive; a.reused_total = L.reused_total; a.status = L.status;
    a.parts = L.parts; a.running = nullptr;
    const int u = w - L.first_warp, tile = u / a.parts, part = u - tile * a.parts;
    dc_pdl_wait();
    dc_pdl_release();
    if (w >= total_warps) return;                       // no copy was issued by this warp
    if (a.gpr > 0) classify_tile_flat(a, tile, part, threadIdx.x & 31, cl);
    else classify_tile(a, tile, part, threadIdx.x & 31, cl);
    rs_wait_all();
}

}  // namespace

// Warps per tile of a layer: one where there are tiles enough to fill the machine (24 warps per SM, twice over); otherwise
// the copies of a tile, up to 128 pixels of px_bytes in rounds of 32 segments, are dealt to as many as have a round to do.
static int copy_parts(const dc_cache* c, long long tiles_in_launch, int px_bytes)
{
    const int rounds = dc_div_up(DC_TILE_H * dc_div_up(DC_TILE_W * px_bytes, kSeg), 32);
    long long room = (long long)c->num_sms * 48 / (tiles_in_launch > 0 ? tiles_in_launch : 1);
    if (room > rounds) room = rounds;
    return room < 1 ? 1 : room > 8 ? 8 : (int)room;
}

// Builds the device table for k_classify_copy_all over the rectangles and counters of a match set (once, after every map is allocated).
int dc_build_classify_table(dc_cache* c, dc_match_set& m)
{
    const int n = c->n_layers;
    ClassifyLayer* h = (ClassifyLayer*)malloc(sizeof(ClassifyLayer) * (n > 0 ? n : 1));
    if (!h) return DC_ERR_ALLOC;
    int k = 0, warps = 0;
    long long tiles = 0;
    for (int i = 0; i < n; ++i) if (dc_layer_cached(c, i)) tiles += dc_layer_tiles(c, c->L[i]);
    for (int i = 0; i < n; ++i) {
        if (!dc_layer_cached(c, i)) continue;
        dc_layer_rt& L = c->L[i];
        ClassifyLayer& e = h[k++];
        e.regions = m.live + (size_t)i * c->S * c->max_regions;
        e.map[0] = (uint8_t*)L.map[0]; e.map[1] = (uint8_t*)L.map[1];
        e.Ho = L.d.out_h; e.Wo = L.d.out_w; e.px_bytes = L.d.cout * c->elt;
        e.tiles_x = L.tiles_x; e.tiles_y = L.tiles_y; e.first_warp = warps;
        e.gpr = L.flat ? L.gpr : 0; e.gpt = L.gpt;
        e.masks = L.masks; e.dirty_list = L.dirty_list; e.dirty_count = m.dirty_count + i;
        e.reuse_px = m.reuse_px + (size_t)i * c->S; e.alive = m.alive + (size_t)i * c->S;
        e.reused_total = c->reused_total + i;
        e.status = c->status;
        e.parts = copy_parts(c, tiles, e.px_bytes);
        warps += dc_layer_tiles(c, L) * e.parts;
    }
    c->n_cached = k; c->classify_warps = warps;
    int rc = DC_OK;
    if (k > 0) {
        if (cudaMalloc(&m.classify_table, sizeof(ClassifyLayer) * k) != cudaSuccess) { cudaGetLastError(); rc = DC_ERR_ALLOC; }
        else if (cudaMemcpyAsync(m.classify_table, h, sizeof(ClassifyLayer) * k, cudaMemcpyHostToDevice, c->stream) != cudaSuccess) rc = DC_ERR_CUDA;
        else c->bytes += sizeof(ClassifyLayer) * k;
    }
    free(h);
    return rc;
}

// All cached layers at once; `cur` is the index of the map that holds the cached values (the same for every layer:
// they all flip once per frame).  Region propagation has zeroed the dirty counts and the reuse counters.
int dc_launch_classify_all(dc_cache* c, int cur)
{
    if (c->n_cached <= 0) return DC_OK;
    {
        dc_prof_scope ps(c, DC_ST_CLASSIFY_COPY);
        static dc_once_per_device attr_set;
        if (attr_set.first(c->device))
            DC_CUDA(cudaFuncSetAttribute(k_classify_copy_all, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCopySmem));
        DC_CUDA(dc_launch_pdl(k_classify_copy_all, dim3((unsigned)dc_div_up(c->classify_warps, kCopyWarps)), kCopyWarps * 32, kCopySmem, c->stream,
                              (const ClassifyLayer*)c->classify_table, c->n_cached, c->classify_warps, c->max_regions, c->S, cur));
    }
    c->launches += 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

// The layer table as k_propagate reads it.
int dc_build_propagate_table(dc_cache* c, const dc_layer_desc* layers)
{
    const int n = c->n_layers;
    PropLayer t[DC_MAX_LAYERS];
    int last_use[DC_MAX_LAYERS], frame_use = -1;           // last layer that reads l's rectangle other than as "the layer before", or the frame's
    for (int l = 0; l < n; ++l) last_use[l] = -1;
    for (int l = 0; l < n; ++l) {
        const dc_layer_desc& d = layers[l];
        const bool two = d.kind == DC_ADD || d.kind == DC_CONCAT;
        if (d.in0 < 0 || (two && d.in1 < 0)) frame_use = l;
        if (d.in0 >= 0 && d.in0 != l - 1) last_use[d.in0] = l;
        if (two && d.in1 >= 0 && d.in1 != l - 1) last_use[d.in1] = l;
    }
    for (int l = 0; l < n; ++l) {
        const dc_layer_desc& d = layers[l];
        const int ih = d.in0 < 0 ? c->cfg.height : layers[d.in0].out_h, iw = d.in0 < 0 ? c->cfg.width : layers[d.in0].out_w;
        PropLayer& e = t[l];
        e = PropLayer();
        e.links = make_int4(d.in0 < 0 ? -1 : d.in0, d.in1 < 0 ? -1 : d.in1, d.kind, last_use[l] > frame_use ? last_use[l] : frame_use);
        e.rule[0] = d.kind == DC_RESIZE_AREA ? make_int4(iw, d.out_w, 0, 0) : make_int4(d.kw, d.sw, d.pw, 0);
        e.rule[1] = d.kind == DC_RESIZE_AREA ? make_int4(ih, d.out_h, 0, 0) : make_int4(d.kh, d.sh, d.ph, 0);
        auto window = [&](int kh, int kw, int sh, int sw, int ph, int pw) {
            if ((sh & (sh - 1)) != 0 || (sw & (sw - 1)) != 0) return;
            const int simple = l == 0 || d.in0 == l - 1;       // layer 0 reads the frame, which is what the walk starts from
            e.links.z = kWindow;
            e.axis[0] = make_int4(pw + sw - 1, pw - kw, 0, simple);
            e.axis[1] = make_int4(ph + sh - 1, ph - kh, 0, simple);
            while ((1 << e.axis[0].z) < sw) ++e.axis[0].z;
            while ((1 << e.axis[1].z) < sh) ++e.axis[1].z;
        };
        if (d.kind == DC_CONV || d.kind == DC_MAXPOOL) window(d.kh, d.kw, d.sh, d.sw, d.ph, d.pw);
        else if (d.kind == DC_LRN) window(2 * d.ph + 1, 2 * d.ph + 1, 1, 1, d.ph, d.ph);
        else if (d.kind == DC_RELU) window(1, 1, 1, 1, 0, 0);
    }
    if (cudaMalloc(&c->prop_table, sizeof(PropLayer) * n) != cudaSuccess) { cudaGetLastError(); return DC_ERR_ALLOC; }
    c->bytes += sizeof(PropLayer) * n;
    DC_CUDA(cudaMemcpy(c->prop_table, t, sizeof(PropLayer) * n, cudaMemcpyHostToDevice));
    return DC_OK;
}

// for_frame: the rectangles of the frame being inferred (counts what is alive, zeroes the reuse step's counters);
// otherwise a caller's, returned in out / n_out for layers out_begin .. layer_end - 1.
int dc_launch_propagate(dc_cache* c, const dc_region* in, const int32_t* n_in, int layer_end, bool for_frame, dc_region* table, dc_region* out, int out_begin, int32_t* n_out)
{
    dc_prof_scope ps(c, DC_ST_PROPAGATE);
    // As many walkers as the rectangles need and shared memory has room for, and at least eight warps for the writing.  A caller's lists, whose
    // every slot is written, go to CTAs of 32 rectangles, or of 64 where those are more than the SMs.  us with 1024 walkers, 256 and 128: 12 layers of
    // 320 slots, 1 stream 8.8, 3.8, 3.6, 64 streams 10.0, 5.7, 6.3; 71 layers of 784 slots, 1 stream 8.2, 6.7, 4.9, 8 streams 8.3, 7.3, 10.4.
    const int room = (int)(kWalkBytes / (8 * (size_t)layer_end)) / 32 * 32, most = room > 1024 ? 1024 : room;
    const int lists = c->S * dc_div_up(c->max_regions, 32) <= c->num_sms ? 128 : 256;
    const int cap = for_frame || lists > most ? most : lists;
    const int walkers = c->max_regions >= cap / kLanes ? cap : dc_div_up(c->max_regions * kLanes, 32) * 32;
    const int threads = walkers < 256 ? 256 : walkers;
    const size_t smem = 8 * (size_t)layer_end * walkers;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) {
        DC_CUDA(cudaFuncSetAttribute(k_propagate<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWalkBytes));
        DC_CUDA(cudaFuncSetAttribute(k_propagate<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWalkBytes));
        DC_CUDA(cudaFuncSetAttribute(k_propagate<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWalkBytes));
    }
    // A frame whose slots are more than two batches' gets two or four CTAs per stream, as long as the SMs take them; those without a rectangle return at
    // once.  us with a thread per rectangle and no table in shared memory, with one CTA, and so: 19 layers, two full-HD streams, 8-pixel blocks, 9.5,
    // 14.3, 10.5, with their blocks' own vectors 28.5, 50.5, 21.7; 71 layers, one stream of 224 x 224, likewise 22.3, 17.0, 14.5.  With 32
    // full-HD streams (launch to end, 19 layers), where hardly more rectangles than a batch turn up, 14.8, 16.6, 16.9, with own vectors 25.1, 39.3, 22.3.
    const int batches = dc_div_up(c->max_regions, walkers / kLanes), side = c->num_sms / c->S;
    const int ctas = !for_frame ? batches : side < 2 || batches < 3 ? 1 : side < 4 || batches < 4 ? 2 : 4;
    const dim3 grid((unsigned)c->S, (unsigned)ctas);
    DC_CUDA(dc_launch_pdl(!for_frame ? k_propagate<false, false> : ctas > 1 ? k_propagate<true, true> : k_propagate<true, false>, grid, threads, smem, c->stream, (const PropLayer*)c->prop_table, layer_end, c->n_layers, c->S, c->max_regions, walkers, in, n_in,
                          table, c->live, c->alive, c->reuse_px, c->dirty_count, c->places, out, out_begin, n_out));
    c->launches += 1;
    return DC_OK;
}

// count, px: where the dirty tiles and the reused pixels per stream are counted.  running: a counter that is zero between
// launches, or NULL: count is zero when the kernel starts.
int dc_launch_classify_copy(dc_cache* c, int layer, const dc_region* regions, const int32_t* n_regions,
                            const void* prev_out, void* out, int32_t* count, int32_t* px, unsigned long long* running)
{
    dc_layer_rt& L = c->L[layer];
    ClassifyArgs a;
    a.regions = regions; a.n_regions = n_regions; a.max_regions = c->max_regions;
    a.prev = (const uint8_t*)prev_out; a.out = (uint8_t*)out;
    a.Ho = L.d.out_h; a.Wo = L.d.out_w; a.px_bytes = L.d.cout * c->elt;
    a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y; a.S = c->S;
    a.gpr = L.flat ? L.gpr : 0; a.gpt = L.gpt; a.n_tiles = dc_layer_tiles(c, L);
    a.masks = L.masks; a.dirty_list = L.dirty_list; a.dirty_count = count;
    a.reuse_px = px;
    a.running = running; a.parts = copy_parts(c, dc_layer_tiles(c, L), a.px_bytes);
    a.reused_total = c->reused_total + layer;
    a.status = c->status;
    a.alive = running ? nullptr : c->alive + (size_t)layer * c->S;      // counted for the frame's rectangles alone, not for a caller's in the same table
    const int warps = dc_layer_tiles(c, L) * a.parts;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device))
        DC_CUDA(cudaFuncSetAttribute(k_classify_copy, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCopySmem));
    { dc_prof_scope ps(c, DC_ST_CLASSIFY_COPY); DC_CUDA(dc_launch_pdl(k_classify_copy, dim3((unsigned)dc_div_up(warps, kCopyWarps)), kCopyWarps * 32, kCopySmem, c->stream, a)); }
    c->launches += 1;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}
