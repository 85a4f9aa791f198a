// Region propagation (Section 5, Table 2) and the reuse step of the cache-aware convolution
// (Section 5, "Reuse": copy cached regions, build the bitmap, list what is left to compute).
//
//   k_propagate      one thread per (stream, rectangle slot) walks the layer table in order and
//                    writes the rectangle's image after every layer; a vanished rectangle is all zeros.
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

// A layer as propagation sees it.  from0 / from1: where the input's rectangle is: kFrame, kPrevious (the layer before, still in
// registers), kTable (the table in global memory), or one of the kSlots places of the thread in shared memory; keep: the
// place that this layer's own rectangle takes, or -1.  drop: places whose rectangles no later layer needs (bit mask); closed: no later
// layer reads the frame's rectangle or the table.
// window: the rule is that of a sliding window whose strides are powers of two (convolutions, pooling; LRN is one at stride 1, ReLU one of
// a single pixel): on either axis first = (x + c1) >> sh, last = (x + w + c2) >> sh.
constexpr int kSlots = 6, kFrame = -1, kPrevious = -2, kTable = -3;
struct __align__(16) PropLayer {
    int window, c1x, c2x, shx, c1y, c2y, shy, from0;
    int from1, two, in0, in1, keep, drop, closed, kind;
    int kh, kw, sh, sw, ph, pw, in_h, in_w, out_h, out_w, pad0, pad1;
};

__device__ __forceinline__ dc_region apply_window(const PropLayer& L, dc_region a)
{
    const int dx = (a.x + L.c1x) >> L.shx, dw = ((a.x + a.w + L.c2x) >> L.shx) - dx + 1;
    const int dy = (a.y + L.c1y) >> L.shy, dh = ((a.y + a.h + L.c2y) >> L.shy) - dy + 1;
    // the cached side on its own; smaller size wins
    const int qx = (a.sx + L.c1x) >> L.shx, qw = ((a.sx + a.w + L.c2x) >> L.shx) - qx + 1;
    const int qy = (a.sy + L.c1y) >> L.shy, qh = ((a.sy + a.h + L.c2y) >> L.shy) - qy + 1;
    const int w = min(dw, qw), h = min(dh, qh);
    if (a.w <= 0 || a.h <= 0 || w <= 0 || h <= 0) return empty_region();
    dc_region o = {dx, dy, w, h, qx, qy};
    return o;
}

__device__ dc_region apply_layer(const PropLayer& L, dc_region a, dc_region b)
{
    if (a.w <= 0 || a.h <= 0) return empty_region();
    switch (L.kind) {
    case DC_CONV: case DC_MAXPOOL: case DC_RESIZE_AREA: {
        // D_t on the current rectangle and, independently, on the cached one; smaller size wins
        int dx, dw, dy, dh, qx, qw, qy, qh;
        if (L.kind == DC_RESIZE_AREA) {
            resize_axis(a.x, a.w, L.in_w, L.out_w, dx, dw);  resize_axis(a.y, a.h, L.in_h, L.out_h, dy, dh);
            resize_axis(a.sx, a.w, L.in_w, L.out_w, qx, qw); resize_axis(a.sy, a.h, L.in_h, L.out_h, qy, qh);
        } else {
            erode_axis(a.x, a.w, L.kw, L.sw, L.pw, dx, dw);  erode_axis(a.y, a.h, L.kh, L.sh, L.ph, dy, dh);
            erode_axis(a.sx, a.w, L.kw, L.sw, L.pw, qx, qw); erode_axis(a.sy, a.h, L.kh, L.sh, L.ph, qy, qh);
        }
        int w = min(dw, qw), h = min(dh, qh);
        if (w <= 0 || h <= 0) return empty_region();
        dc_region o = {dx, dy, w, h, qx, qy};
        return o;
    }
    case DC_ADD: case DC_CONCAT: {
        // the overlapped region; both inputs must agree on the displacement
        if (b.w <= 0 || b.h <= 0) return empty_region();
        if (a.sx - a.x != b.sx - b.x || a.sy - a.y != b.sy - b.y) return empty_region();
        int x0 = max(a.x, b.x), y0 = max(a.y, b.y);
        int x1 = min(a.x + a.w, b.x + b.w), y1 = min(a.y + a.h, b.y + b.h);
        if (x1 <= x0 || y1 <= y0) return empty_region();
        dc_region o = {x0, y0, x1 - x0, y1 - y0, x0 + (a.sx - a.x), y0 + (a.sy - a.y)};
        return o;
    }
    case DC_FC:
        return empty_region();
    default:
        return a;
    }
}

// The tables are 8-byte aligned: three stores, not six.
__device__ __forceinline__ void store_region(dc_region* t, const dc_region& o)
{
    uint2* p = (uint2*)t;
    p[0] = make_uint2(o.x, o.y); p[1] = make_uint2(o.w, o.h); p[2] = make_uint2(o.sx, o.sy);
}

// One CTA per stream (more for a caller's lists, which count nothing), a thread one rectangle at a time.  Rectangles that a
// later layer than the next one needs (residual branches) wait in shared memory, and so does the layer table: the walk is
// a chain of a few dozen arithmetic steps per layer.  A warp whose rectangles have all vanished, those kept for later layers
// too, writes the zeros of the layers that are left without walking them.
// us for ResNet-50's 71 layers: table in global memory 48, an atomic per rectangle and layer 27, so 24; VGG, 8 full-HD
// frames: 12.5 with the atomics, 7.7 so.
// alive, live: how many rectangles are left at each layer and stream, and these alone, in any order (they are disjoint): most of a
// frame's erode within a few layers, and the reuse step tests every tile against all it is given.  A warp asks for its places in a
// layer's list with one atomic and fills them while the next layer is worked out.
// out, n_out: a caller's copies of layers out_begin .. layer_end - 1 and of the counts.  alive (or NULL): the lists are wanted, and the
// counters of the reuse step are zeroed.
__global__ void __launch_bounds__(1024) k_propagate(const PropLayer* layers, int layer_end, int n_layers, int S, int max_regions,
                                                   const dc_region* in, const int32_t* n_in, dc_region* table, dc_region* live, int32_t* alive, int32_t* reuse_px,
                                                   int32_t* dirty_count, dc_region* out, int out_begin, int32_t* n_out)
{
    __shared__ PropLayer sl[DC_MAX_LAYERS];
    extern __shared__ int32_t keep[];                      // [places in use][6][threads]
    __shared__ int32_t count[DC_MAX_LAYERS];
    const int s = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    for (int i = tid; i < layer_end * (int)(sizeof(PropLayer) / 16); i += nt) ((int4*)sl)[i] = __ldg((const int4*)layers + i);
    if (tid < DC_MAX_LAYERS) count[tid] = 0;
    dc_pdl_wait();
    dc_pdl_release();
    __syncthreads();
    const size_t layer_stride = (size_t)S * max_regions;
    const int n = min(n_in[s], max_regions);              // a caller's count beyond the table is cut, never written
    // a caller's list has zeros behind its rectangles
    const int rows = out ? max_regions : n;
    for (int first = blockIdx.y * nt; first < rows; first += gridDim.y * nt) {
        const int i = first + tid;
        const size_t slot = (size_t)s * max_regions + i;
        const bool on = i < n, there = i < rows;
        const dc_region r0 = on ? in[slot] : empty_region();
        dc_region prev = r0;
        auto fetch = [&](int from, int layer) -> dc_region {
            if (from == kFrame) return r0;
            if (from == kPrevious) return prev;
            if (from == kTable) return on ? table[layer * layer_stride + slot] : empty_region();
            const int32_t* k = keep + from * 6 * nt + tid;
            dc_region r = {k[0], k[nt], k[2 * nt], k[3 * nt], k[4 * nt], k[5 * nt]};
            return r;
        };
        uint32_t kept = 0;                                             // places that hold a living rectangle of this thread
        unsigned noted = 0;                                            // the warp's living rectangles of the layer before (prev), and their
        int place = 0;                                                 // first place in that layer's list (lane 0)
        auto list_prev = [&](int layer) {
            const int at = __shfl_sync(0xffffffffu, place, 0) + __popc(noted & ((1u << lane) - 1u));
            if ((noted >> lane) & 1u) store_region(live + layer * layer_stride + (size_t)s * max_regions + at, prev);
        };
        int l = 0;
        for (bool dead = i - lane >= rows; l < layer_end && !dead; ++l) {
            const PropLayer& L = sl[l];
            const dc_region a = fetch(L.from0, L.in0);
            dc_region o;
            if (L.window) o = apply_window(L, a);
            else o = apply_layer(L, a, L.two ? fetch(L.from1, L.in1) : a);
            kept &= ~(uint32_t)L.drop;
            if (L.keep >= 0) {
                int32_t* k = keep + L.keep * 6 * nt + tid;
                k[0] = o.x; k[nt] = o.y; k[2 * nt] = o.w; k[3 * nt] = o.h; k[4 * nt] = o.sx; k[5 * nt] = o.sy;
                kept = o.w > 0 ? kept | (1u << L.keep) : kept & ~(1u << L.keep);
            }
            if (there) {
                store_region(table + l * layer_stride + slot, o);
                if (out && l >= out_begin) out[(l - out_begin) * layer_stride + slot] = o;
            }
            if (noted) list_prev(l - 1);
            const unsigned living = __ballot_sync(0xffffffffu, o.w > 0);
            noted = alive ? living : 0u;
            if (noted && lane == 0) place = atomicAdd(&count[l], __popc(noted));
            dead = !living && L.closed && !__any_sync(0xffffffffu, kept != 0);
            prev = o;
        }
        if (noted) list_prev(l - 1);
        // the zeros: a warp's rectangles are one run of memory
        const int run = 3 * min(32, rows - (i - lane));
        for (; l < layer_end; ++l) {
            uint2* t = (uint2*)(table + l * layer_stride + slot - lane);
            for (int k = lane; k < run; k += 32) t[k] = make_uint2(0, 0);
            if (out && l >= out_begin && there) out[(l - out_begin) * layer_stride + slot] = empty_region();
        }
    }
    if (n_out && blockIdx.y == 0) for (int l = out_begin + tid; l < layer_end; l += nt) n_out[(l - out_begin) * S + s] = n_in[s];
    if (alive) {
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
    // every rectangle of this stream has eroded away before this layer: nothing to test or copy
    const int n = (a.alive && a.alive[s] == 0) ? 0 : min(a.n_regions[s], a.max_regions);
    const size_t map_base = (size_t)s * a.Ho * a.Wo * a.px_bytes;
    uint32_t m0 = 0, m1 = 0, m2 = 0, m3 = 0;      // bit (row * DC_TILE_W + col) of the tile, row-major
    for (int base = 0; base < n; base += 32) {
        int i = base + lane;
        dc_region r = empty_region();
        int ix0 = 0, ix1 = 0, iy0 = 0, iy1 = 0;
        if (i < n) {
            r = regs[i];
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
        int first = mine;                                               // inclusive sum over the lanes, then this lane's start
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, first, o); if (lane >= o) first += v; }
        const int items = __shfl_sync(0xffffffffu, first, 31);
        first -= mine;
        const int src_y = iy0 - r.y + r.sy, src_x = ix0 - r.x + r.sx;   // cached position of (ix0, iy0)
        for (int i0 = part * 32; i0 < items && !cl.dead; i0 += 32 * a.parts) {
            const int it = i0 + lane;
            const bool on = it < items;
            int owner = 0;                                              // the lane whose rectangle segment `it` belongs to
            for (unsigned h = hits; h; h &= h - 1) {
                const int k = __ffs(h) - 1;
                if (it >= __shfl_sync(0xffffffffu, first, k)) owner = k;
            }
            const int o_first = __shfl_sync(0xffffffffu, first, owner), o_segs = max(1, __shfl_sync(0xffffffffu, segs, owner));
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
    dc_pdl_wait();
    dc_pdl_release();
    const int w = blockIdx.x * kCopyWarps + (threadIdx.x >> 5);
    if (w >= total_warps) return;                       // no copy was issued by this warp
    int lo = 0, hi = n_cached - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (layers[mid].first_warp <= w) lo = mid; else hi = mid - 1;
    }
    const ClassifyLayer& L = layers[lo];
    ClassifyArgs a;
    a.regions = L.regions; a.n_regions = L.alive; a.max_regions = max_regions;     // the rectangles left at this layer
    a.prev = L.map[cur]; a.out = L.map[cur ^ 1];
    a.Ho = L.Ho; a.Wo = L.Wo; a.px_bytes = L.px_bytes; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y; a.S = S;
    a.gpr = L.gpr; a.gpt = L.gpt; a.n_tiles = 0;
    a.masks = L.masks; a.dirty_list = L.dirty_list; a.dirty_count = L.dirty_count; a.reuse_px = L.reuse_px;
    a.alive = L.alive; a.reused_total = L.reused_total; a.status = L.status;
    a.parts = L.parts; a.running = nullptr;
    const int u = w - L.first_warp, tile = u / a.parts, part = u - tile * a.parts;
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

// Builds the device table for k_classify_copy_all (once, after every map is allocated).
int dc_build_classify_table(dc_cache* c)
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
        e.regions = c->live + (size_t)i * c->S * c->max_regions;
        e.map[0] = (uint8_t*)L.map[0]; e.map[1] = (uint8_t*)L.map[1];
        e.Ho = L.d.out_h; e.Wo = L.d.out_w; e.px_bytes = L.d.cout * c->elt;
        e.tiles_x = L.tiles_x; e.tiles_y = L.tiles_y; e.first_warp = warps;
        e.gpr = L.flat ? L.gpr : 0; e.gpt = L.gpt;
        e.masks = L.masks; e.dirty_list = L.dirty_list; e.dirty_count = c->dirty_count + i;
        e.reuse_px = c->reuse_px + (size_t)i * c->S; e.alive = c->alive + (size_t)i * c->S;
        e.reused_total = c->reused_total + i;
        e.status = c->status;
        e.parts = copy_parts(c, tiles, e.px_bytes);
        warps += dc_layer_tiles(c, L) * e.parts;
    }
    c->n_cached = k; c->classify_warps = warps;
    int rc = DC_OK;
    if (k > 0) {
        if (cudaMalloc(&c->classify_table, sizeof(ClassifyLayer) * k) != cudaSuccess) { cudaGetLastError(); rc = DC_ERR_ALLOC; }
        else if (cudaMemcpy(c->classify_table, h, sizeof(ClassifyLayer) * k, cudaMemcpyHostToDevice) != cudaSuccess) rc = DC_ERR_CUDA;
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
    int last_use[DC_MAX_LAYERS];                           // last layer that needs l's rectangle other than as "the layer before"
    for (int l = 0; l < n; ++l) last_use[l] = -1;
    for (int l = 0; l < n; ++l) {
        const dc_layer_desc& d = layers[l];
        if (d.in0 >= 0 && d.in0 != l - 1) last_use[d.in0] = l;
        if ((d.kind == DC_ADD || d.kind == DC_CONCAT) && d.in1 >= 0 && d.in1 != l - 1) last_use[d.in1] = l;
    }
    int owner[kSlots];
    for (int k = 0; k < kSlots; ++k) owner[k] = -1;
    auto from = [&](int l, int in) {
        if (in < 0) return kFrame;
        if (in == l - 1) return kPrevious;
        for (int k = 0; k < kSlots; ++k) if (owner[k] == in) return k;
        return kTable;
    };
    for (int l = 0; l < n; ++l) {
        const dc_layer_desc& d = layers[l];
        const int ih = d.in0 < 0 ? c->cfg.height : layers[d.in0].out_h, iw = d.in0 < 0 ? c->cfg.width : layers[d.in0].out_w;
        PropLayer& e = t[l];
        e = PropLayer();
        e.kind = d.kind; e.kh = d.kh; e.kw = d.kw; e.sh = d.sh; e.sw = d.sw; e.ph = d.ph; e.pw = d.pw;
        e.in_h = ih; e.in_w = iw; e.out_h = d.out_h; e.out_w = d.out_w; e.in0 = d.in0; e.in1 = d.in1;
        e.from0 = from(l, d.in0); e.from1 = from(l, d.in1); e.keep = -1;
        e.two = d.kind == DC_ADD || d.kind == DC_CONCAT;
        auto window = [&](int kh, int kw, int sh, int sw, int ph, int pw) {
            if ((sh & (sh - 1)) != 0 || (sw & (sw - 1)) != 0) return;
            e.window = 1;
            e.c1x = pw + sw - 1; e.c2x = pw - kw; e.c1y = ph + sh - 1; e.c2y = ph - kh;
            while ((1 << e.shx) < sw) ++e.shx;
            while ((1 << e.shy) < sh) ++e.shy;
        };
        if (d.kind == DC_CONV || d.kind == DC_MAXPOOL) window(d.kh, d.kw, d.sh, d.sw, d.ph, d.pw);
        else if (d.kind == DC_LRN) window(2 * d.ph + 1, 2 * d.ph + 1, 1, 1, d.ph, d.ph);
        else if (d.kind == DC_RELU) window(1, 1, 1, 1, 0, 0);
        for (int k = 0; k < kSlots; ++k) if (owner[k] >= 0 && last_use[owner[k]] <= l) { owner[k] = -1; t[l].drop |= 1 << k; }
        if (last_use[l] > l)
            for (int k = 0; k < kSlots; ++k) if (owner[k] < 0) { owner[k] = l; t[l].keep = k; if (k >= c->prop_slots) c->prop_slots = k + 1; break; }
    }
    for (int l = n - 1, open = 0; l >= 0; --l) {
        t[l].closed = !open;
        auto outside = [](int from) { return from == kFrame || from == kTable; };
        open = open || outside(t[l].from0) || (t[l].two && outside(t[l].from1));
    }
    if (cudaMalloc(&c->prop_table, sizeof(PropLayer) * n) != cudaSuccess) { cudaGetLastError(); return DC_ERR_ALLOC; }
    c->bytes += sizeof(PropLayer) * n;
    DC_CUDA(cudaMemcpy(c->prop_table, t, sizeof(PropLayer) * n, cudaMemcpyHostToDevice));
    return DC_OK;
}

// for_frame: the rectangles of the frame being inferred (counts what is alive, zeroes the reuse step's counters);
// otherwise a caller's, returned in out / n_out for layers out_begin .. layer_end - 1.
int dc_launch_propagate(dc_cache* c, const dc_region* in, const int32_t* n_in, int layer_end, bool for_frame, dc_region* out, int out_begin, int32_t* n_out)
{
    dc_prof_scope ps(c, DC_ST_PROPAGATE);
    // a thread per rectangle where the frame can have many
    const int threads = c->max_regions > 512 ? 1024 : 256;
    const size_t smem = (size_t)c->prop_slots * 6 * threads * sizeof(int32_t);
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) DC_CUDA(cudaFuncSetAttribute(k_propagate, cudaFuncAttributeMaxDynamicSharedMemorySize, kSlots * 6 * 1024 * (int)sizeof(int32_t)));
    const dim3 grid((unsigned)c->S, for_frame ? 1u : (unsigned)dc_div_up(c->max_regions, threads));
    DC_CUDA(dc_launch_pdl(k_propagate, grid, threads, smem, c->stream, (const PropLayer*)c->prop_table, layer_end, c->n_layers, c->S, c->max_regions, in, n_in,
                          c->table, c->live, for_frame ? c->alive : nullptr, c->reuse_px, c->dirty_count, out, out_begin, n_out));
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
