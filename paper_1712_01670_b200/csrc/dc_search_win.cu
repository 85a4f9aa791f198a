// Step 2 (Section 4) for any block size, search unit and frame layout: the kernels behind every search that the
// 16-pixel kernels of dc_match.cu do not take - other block sizes, blocks clipped by the frame's edge - and behind
// dc_search_blocks_noalloc.
//
// One CTA per tile of TX x TY blocks.  The part of the previous frame that any candidate of the tile can touch (the tile
// and R pixels around it) is staged once in shared memory, one 32-bit word per pixel (R, G, B, 0), so a candidate starts
// at a word whatever its displacement and whatever the alignment of the caller's rows.  Walks with a range beyond
// kWalkReach may stage that much and fetch the rare candidate outside from global memory.
//   k_win_walk  diamond and three step search: one warp per block, lane l owns pixels l, l + 32, ... of the block.  The
//               window's row pitch is congruent to the block edge modulo 32, so the lanes of a load fall in 32
//               different banks.  The points of a round are scored as straight-line code, their loads all in flight.
//   k_win_all   exhaustive search: a lane owns one horizontal displacement and E_ROWS vertical ones; walking down a
//               column of the block it loads one window word and one block word per row for E_ROWS differences.
// Candidates are ordered by (SSE, |dx| + |dy|, dy, dx).  Integer arithmetic only.
//
// What bounds them: with few blocks the chain of rounds of one walk (a round is one trip to shared memory and back),
// otherwise instruction issue.
#include "dc_common.cuh"
#include "dc_search_win.cuh"
#include "dc_walk.cuh"

namespace {

constexpr int E_ROWS = 8;                 // vertical displacements a lane scores together
constexpr int kMaxWarps = 16;
// Pixels around the tile that walks over a longer range stage at least.  A walk visits a few dozen candidates near its start;
// staging 64 pixels on every side of a few small blocks cost more than all of them (see dc_launch_search_win).
constexpr int kWalkReach = 32;

// Pixel at byte address p of a buffer [lo, hi): whole aligned words where they lie inside the buffer, bytes at its ends.
__device__ __forceinline__ uint32_t load_pixel(const uint8_t* p, const uint8_t* lo, const uint8_t* hi)
{
    const uint32_t* q = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
    const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u;
    if ((const uint8_t*)q >= lo && (const uint8_t*)(q + 2) <= hi) {
        const uint32_t a = dc_ld(q), b = sh > 8 ? dc_ld(q + 1) : 0u;
        return __funnelshift_r(a, b, sh) & 0x00ffffffu;
    }
    return (uint32_t)dc_ld(p) | ((uint32_t)dc_ld(p + 1) << 8) | ((uint32_t)dc_ld(p + 2) << 16);
}

struct Tile { int s, bx0, by0, nbx, nby; };       // stream, first block, blocks of the tile that exist

__device__ __forceinline__ Tile tile_of(const dc_win_args& a)
{
    Tile t;
    t.s = blockIdx.z;
    t.bx0 = blockIdx.x * a.TX; t.by0 = blockIdx.y * a.TY;
    t.nbx = min(a.TX, a.Gx - t.bx0); t.nby = min(a.TY, a.Gy - t.by0);
    return t;
}
__device__ __forceinline__ bool searched(const dc_win_args& a, int bx, int by)
{
    return a.skip_k <= 1 || (bx % a.skip_k == 0 && by % a.skip_k == 0);
}
// blocks this launch is about: all, or those that the frame's edge clips
__device__ __forceinline__ bool mine(const dc_win_args& a, int bx, int by)
{
    return a.only_clipped == 0 || a.W - bx * a.B < a.B || a.H - by * a.B < a.B;
}

__device__ __forceinline__ bool any_mine(const dc_win_args& a, const Tile& t)
{
    const bool right = t.bx0 + t.nbx == a.Gx && a.W % a.B != 0, bottom = t.by0 + t.nby == a.Gy && a.H % a.B != 0;
    return a.only_clipped == 0 || right || bottom;
}

// The window, rows warp by warp, a lane four pixels: the 12 bytes come as four aligned words, whatever the row's alignment, also where some of
// them lie beside the frame (what does is never part of a valid candidate).  Only lanes whose words may leave the buffer, at its two
// ends, go pixel by pixel.
__device__ __forceinline__ void stage_window(const dc_win_args& a, const Tile& t, uint32_t* win)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int x0 = t.bx0 * a.B - a.Rw, y0 = t.by0 * a.B - a.Rw, margin = a.margin, cols = a.win_cols - margin;
    const uint8_t* prev = a.prev + (size_t)t.s * a.prev_stream;
    const int y_lo = max(y0 + margin, 0), y_hi = min(y0 + a.win_rows - margin, a.H) - 1;
    // a narrow window: several rows per warp
    const int lpr = cols - margin > 64 ? 32 : cols - margin > 32 ? 16 : 8, rpw = 32 / lpr, l = lane & (lpr - 1);
    const int first_row = y_lo + warp * rpw + lane / lpr, row_step = warps * rpw;
    const uint32_t m = 0x00ffffffu;
    for (int c = margin + 4 * l; c < cols; c += 4 * lpr) {             // once, but for windows wider than 128 pixels
        const int x = x0 + c;
        if (x + 4 <= 0 || x >= a.W) continue;
        uint32_t* dst = win + (first_row - y0) * a.win_pitch + c;
        const uint8_t* p = prev + (ptrdiff_t)first_row * (ptrdiff_t)a.prev_pitch + (ptrdiff_t)x * 3;
        if ((const uint8_t*)((uintptr_t)p & ~(uintptr_t)3) >= a.prev && prev + (ptrdiff_t)y_hi * (ptrdiff_t)a.prev_pitch + (ptrdiff_t)x * 3 + 16 <= a.prev_end) {
#pragma unroll 3
            for (int y = first_row; y <= y_hi; y += row_step, p += row_step * a.prev_pitch, dst += row_step * a.win_pitch) {
                const uint32_t* q = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
                const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u;
                const uint32_t w0 = dc_ld(q), w1 = dc_ld(q + 1), w2 = dc_ld(q + 2), w3 = dc_ld(q + 3);
                const uint32_t b0 = __funnelshift_r(w0, w1, sh), b1 = __funnelshift_r(w1, w2, sh), b2 = __funnelshift_r(w2, w3, sh);
                dst[0] = b0 & m; dst[1] = __funnelshift_r(b0, b1, 24) & m; dst[2] = __funnelshift_r(b1, b2, 16) & m; dst[3] = b2 >> 8;
            }
        } else {
            for (int y = first_row; y <= y_hi; y += row_step, p += row_step * a.prev_pitch, dst += row_step * a.win_pitch)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x + k >= 0 && x + k < a.W) dst[k] = load_pixel(p + 3 * k, a.prev, a.prev_end);
        }
    }
}

// Step 3's set S: per CTA in shared memory, then three atomics
__device__ __forceinline__ void publish(const dc_win_args& a, const Tile& t, int bx, int by, int dx, int dy, uint32_t sse, int32_t* sums)
{
    const size_t g = (size_t)t.s * a.Gx * a.Gy + (size_t)by * a.Gx + bx;
    a.mv[2 * g] = (int16_t)dx; a.mv[2 * g + 1] = (int16_t)dy; a.sse[g] = sse;
    const int e = (a.H - by * a.B < a.B ? 2 : 0) + (a.W - bx * a.B < a.B ? 1 : 0);
    if (sse <= a.limit[e]) { atomicAdd(&sums[0], dx); atomicAdd(&sums[1], dy); atomicAdd(&sums[2], 1); }
}
__device__ __forceinline__ void mark_skipped(const dc_win_args& a, const Tile& t, int bx, int by)
{
    const size_t g = (size_t)t.s * a.Gx * a.Gy + (size_t)by * a.Gx + bx;
    a.mv[2 * g] = 0; a.mv[2 * g + 1] = 0; a.sse[g] = 0xffffffffu;
}
// Called once by every warp when its blocks are done: the CTA's last warp adds the sums, nobody waits for a longer walk.
__device__ __forceinline__ void flush_sums(const dc_win_args& a, const Tile& t, int32_t* sums)
{
    __syncwarp();
    if ((threadIdx.x & 31) != 0) return;
    __threadfence_block();
    if (atomicAdd(&sums[3], 1) != (int)(blockDim.x >> 5) - 1) return;
    __threadfence_block();
    const int n = atomicAdd(&sums[2], 0);
    if (n == 0) return;
    atomicAdd(&a.acc[4 * t.s + 0], atomicAdd(&sums[0], 0));
    atomicAdd(&a.acc[4 * t.s + 1], atomicAdd(&sums[1], 0));
    atomicAdd(&a.acc[4 * t.s + 2], n);
}

// ---- walks -----------------------------------------------------------------------------------------------------------
// FAR: the window holds fewer than R pixels around the tile.  BT, PT: block edge and window pitch where they are known at compile time
// (walk_pitch), else 0.  EDGE: no room for points beyond the range; rounds that the range or the frame cuts have a path of their own.
template <int ITERS, bool FAR, int BT, int PT, bool EDGE>
struct Walk {
    uint32_t base;                  // shared-memory byte address of displacement (0, 0)
    int pitch4_;                    // window row in bytes
    Within valid;                   // displacements that keep the block inside the frame and the range
    const dc_win_args* args;        // FAR: where candidates outside the window come from:
    const uint8_t* home;            // the block's position in the previous frame
    uint32_t cw[ITERS], off[ITERS]; // this lane's pixels and their byte offsets in the window
    uint32_t on;                    // which of them exist
    bool whole;                     // the block is not clipped: the first FULL exist in every lane
    static constexpr int FULL = ITERS <= 8 ? ITERS - 1 : ITERS / 2;
    int at; uint32_t bs;            // best point so far and its SSE

    __device__ __forceinline__ int pitch4() const { return PT ? PT * 4 : pitch4_; }
    __device__ __forceinline__ bool staged(int dx, int dy, int reach) const
    {
        return !FAR || (abs(dx) + reach <= kWalkReach && abs(dy) + reach <= kWalkReach);
    }
    // A candidate outside the window, from global memory: eight of the lane's pixels in flight.
    __device__ uint32_t far(int dx, int dy) const
    {
        const uint8_t* p0 = home + (ptrdiff_t)dy * (ptrdiff_t)args->prev_pitch + dx * 3;
        const int B = args->B, inv = (65536 + B - 1) / B;                        // p / B for p < 1024: p * inv >> 16
        // two aligned words around any pixel of the block lie inside the buffer (the same in all lanes)
        const bool words = p0 - 3 >= args->prev && p0 + (size_t)(B - 1) * args->prev_pitch + (size_t)B * 3 + 8 <= args->prev_end;
        uint32_t acc = 0;
#pragma unroll
        for (int i0 = 0; i0 < ITERS; i0 += 8) {
            if (i0 * 32 >= B * B) break;
            uint32_t px[8];
            if (words) {
                uint32_t lo[8], hi[8], sh[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i0 + j, q = i * 32 + (int)(threadIdx.x & 31), r = q * inv >> 16, c = q - r * B;
                    const bool there = i < ITERS && ((on >> (i & 31)) & 1u);     // else the block's first pixel, masked
                    const uint8_t* p = there ? p0 + (size_t)r * args->prev_pitch + c * 3 : p0;
                    const uint32_t* w = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
                    sh[j] = ((uint32_t)(uintptr_t)p & 3u) * 8u;
                    lo[j] = dc_ld(w); hi[j] = dc_ld(w + 1);
                }
#pragma unroll
                for (int j = 0; j < 8; ++j) px[j] = __funnelshift_r(lo[j], hi[j], sh[j]) & 0x00ffffffu;
            } else {
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int i = i0 + j, q = i * 32 + (int)(threadIdx.x & 31), r = q * inv >> 16, c = q - r * B;
                    px[j] = i < ITERS && ((on >> (i & 31)) & 1u) ? load_pixel(p0 + (size_t)r * args->prev_pitch + c * 3, args->prev, args->prev_end) : 0u;
                }
            }
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                if (i0 + j >= ITERS) break;
                const uint32_t d = ((on >> (i0 + j)) & 1u) ? __vabsdiffu4(cw[i0 + j], px[j]) : 0u;
                acc = __dp4a(d, d, acc);
            }
        }
        return __reduce_add_sync(0xffffffffu, acc);
    }
    __device__ __forceinline__ uint32_t score(int dx, int dy) const
    {
        if constexpr (FAR) { if (!staged(dx, dy, 0)) return far(dx, dy); }
        const uint32_t p = base + (uint32_t)(dy * pitch4() + dx * 4);
        uint32_t acc = 0;
#pragma unroll
        for (int i = 0; i < ITERS; ++i) {
            const uint32_t d = ((on >> i) & 1u) ? __vabsdiffu4(cw[i], lds_at<0>(p + off[i])) : 0u;
            acc = __dp4a(d, d, acc);
        }
        return __reduce_add_sync(0xffffffffu, acc);
    }
    // The points of `set` one by one, for blocks that the frame's edge cuts and centres near the end of the window.  d: the lanes' points.
    __device__ __forceinline__ void slow_set(unsigned set, int d, int lane, uint32_t& mine) const
    {
#pragma unroll 1
        while (set) {
            const int i = __ffs(set) - 1, p = __shfl_sync(0xffffffffu, d, i);
            set &= set - 1;
            const uint32_t s = score(disp_x(p), disp_y(p));
            mine = lane == i ? s : mine;
        }
    }
    // The points of SET around the centre at pc, all staged, as straight-line code; lane i keeps the score of point i.
    template <uint32_t SET>
    __device__ __forceinline__ void fast_set(uint32_t pc, int lane, uint32_t& mine) const
    {
        uint32_t s[13];
#pragma unroll
        for (int k = 0; k < 13; ++k) s[k] = 0;
#pragma unroll
        for (int i = 0; i < ITERS; ++i) add_point<SET, 0>(i, pc + off[i], s);
        keep<SET, 0>(s, lane, mine);
    }
    template <uint32_t SET, int I>
    __device__ __forceinline__ void add_point(int i, uint32_t p, uint32_t (&s)[13]) const
    {
        if constexpr (I < 13) {
            if constexpr (((SET >> I) & 1u) != 0) {
                const uint32_t v = PT ? lds_at<(point_y(I) * PT + point_x(I)) * 4>(p) : lds_at<point_x(I) * 4>(p + (uint32_t)(point_y(I) * pitch4_));
                uint32_t d = __vabsdiffu4(cw[i], v);
                if (i >= FULL) d &= 0u - ((on >> i) & 1u);
                s[I] = __dp4a(d, d, s[I]);
            }
            add_point<SET, I + 1>(i, p, s);
        }
    }
    template <uint32_t SET, int I>
    __device__ __forceinline__ void keep(const uint32_t (&s)[13], int lane, uint32_t& mine) const
    {
        if constexpr (I < 13) {
            if constexpr (((SET >> I) & 1u) != 0) {
                const uint32_t v = __reduce_add_sync(0xffffffffu, s[I]);
                mine = lane == I ? v : mine;
            }
            keep<SET, I + 1>(s, lane, mine);
        }
    }
    // large diamond until its centre wins, then one small diamond.  A point's score stands in its lane, which drops it where it is no valid
    // candidate (a centre's points are staged, whatever the range); the best lane names the next centre.
    __device__ __forceinline__ void diamond(int R, int32_t* status)
    {
        const unsigned all = 0xffffffffu;
        const int lane = threadIdx.x & 31, point = lane_point(lane);
        at = disp(0, 0); bs = 0xffffffffu;
        int kind = KIND_FIRST;
#pragma unroll 1
        for (int moves_left = (2 * R + 1) * (2 * R + 1);; --moves_left) {     // every move strictly lowers the key: never used up
            const int cx = disp_x(at), cy = disp_y(at), d = at + point;
            const bool ok = lane < 13 && within(d, valid);
            uint32_t mine = 0xffffffffu;
            if (whole && staged(cx, cy, 2) && (!EDGE || (within(at - pair(2, 2), valid) && within(at + pair(2, 2), valid)))) {
                const uint32_t pc = base + (uint32_t)(cy * pitch4() + cx * 4);
                switch (kind) {
                case 0: fast_set<kind_mask(0)>(pc, lane, mine); break;
                case 1: fast_set<kind_mask(1)>(pc, lane, mine); break;
                case 2: fast_set<kind_mask(2)>(pc, lane, mine); break;
                case 3: fast_set<kind_mask(3)>(pc, lane, mine); break;
                case 4: fast_set<kind_mask(4)>(pc, lane, mine); break;
                case 5: fast_set<kind_mask(5)>(pc, lane, mine); break;
                case 6: fast_set<kind_mask(6)>(pc, lane, mine); break;
                case 7: fast_set<kind_mask(7)>(pc, lane, mine); break;
                case KIND_FIRST: fast_set<kind_mask(KIND_FIRST)>(pc, lane, mine); break;
                default: fast_set<kind_mask(KIND_SMALL)>(pc, lane, mine); break;
                }
            } else {
                slow_set(c_kind_mask[kind] & __ballot_sync(all, ok), d, lane, mine);
            }
            if (lane == 8 && kind != KIND_FIRST) mine = bs;               // the centre
            if (!ok) mine = 0xffffffffu;
            const int g = best_lane(mine, d, bs);
            at = __shfl_sync(all, d, g);
            if (kind == KIND_SMALL) return;
            if (g == 8) { kind = KIND_SMALL; continue; }
            if (moves_left <= 0) { if (lane == 0 && status) atomicExch(status, (int)DC_ERR_TIMEOUT); return; }
            kind = g;
        }
    }
    // nine-point passes with step S0, S0/2, ..., 1; S0 = largest power of two with 2 S0 - 1 <= R.  Lane g < 9 holds point g of the grid
    // (4: its centre, the best so far).
    __device__ __forceinline__ void three_step(int R)
    {
        const unsigned all = 0xffffffffu;
        const int lane = threadIdx.x & 31, point = pair(lane % 3 - 1, lane / 3 - 1);
        at = disp(0, 0); bs = score(0, 0);
        int step = R < 1 ? 0 : 1;
        while (step > 0 && 4 * step - 1 <= R) step *= 2;
#pragma unroll 1
        for (; step >= 1; step >>= 1) {
            const int cx = disp_x(at), cy = disp_y(at), d = at + step * point;
            const bool ok = lane < 9 && within(d, valid);
            uint32_t mine = 0xffffffffu;
            if (whole && staged(cx, cy, step)) {
                const uint32_t pc = base + (uint32_t)(cy * pitch4() + cx * 4);
                uint32_t s[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) s[k] = 0;
#pragma unroll
                for (int i = 0; i < ITERS; ++i)
#pragma unroll
                    for (int k = 0; k < 9; ++k)
                        if (k != 4) {
                            uint32_t e = __vabsdiffu4(cw[i], lds_at<0>(pc + off[i] + (uint32_t)((k / 3 - 1) * step * pitch4() + (k % 3 - 1) * step * 4)));
                            if (i >= FULL) e &= 0u - ((on >> i) & 1u);
                            s[k] = __dp4a(e, e, s[k]);
                        }
#pragma unroll
                for (int k = 0; k < 9; ++k)
                    if (k != 4) { const uint32_t v = __reduce_add_sync(all, s[k]); mine = lane == k ? v : mine; }
            } else {
                slow_set(0x1efu & __ballot_sync(all, ok), d, lane, mine);
            }
            if (lane == 4) mine = bs;
            if (!ok) mine = 0xffffffffu;
            const int g = best_lane(mine, d, bs);
            at = __shfl_sync(all, d, g);
        }
    }
};

// Window pitch of the instances that know their block edge: room for eight blocks and a range of 16 around them, congruent to B modulo 32.
__host__ __device__ constexpr int walk_pitch(int B) { return 8 * B + 36 + ((B - (8 * B + 36)) % 32 + 32) % 32; }

// Three CTAs per SM where the lane's pixels leave the registers for it (10-pixel blocks, 720p, 4 streams: 78 us, 90 with two; 16-pixel blocks
// with three: twice as slow).  AHEAD: two, with 64 registers a thread for the loads of a round; up to two tiles per SM it is the faster one
// (16 streams of 160 x 128, 10 pixels: 16.3 and 10.8 us).
// What it spends its instructions on (720p, 4 streams, 10 pixels, 1430 per block before): the candidates a third, so addresses known at compile
// time, window rows by addition and whole blocks without a test per pixel: 80 us with run-time addresses and a path of their own for cut
// rounds, 65 without these two, 57 so.
template <int ITERS, bool FAR, int BT, bool AHEAD, bool EDGE = false>
__global__ void __launch_bounds__(kMaxWarps * 32, ITERS <= 4 && !FAR && !AHEAD ? 3 : ITERS <= 8 ? 2 : 1) k_win_walk(const __grid_constant__ dc_win_args a)
{
    extern __shared__ __align__(16) uint32_t win[];
    __shared__ int32_t sums[4];
    constexpr int PT = BT ? walk_pitch(BT) : 0;
    const int B = BT ? BT : a.B;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    dc_pdl_wait();
    dc_pdl_release();
    const Tile t = tile_of(a);
    if (!any_mine(a, t)) return;
    const int ly = warp * a.inv_TX >> 16, lx = warp - ly * a.TX, bx = t.bx0 + lx, by = t.by0 + ly;
    const bool block = ly < a.TY && lx < t.nbx && ly < t.nby && mine(a, bx, by), walk = block && searched(a, bx, by);
    Walk<ITERS, FAR, BT, PT, EDGE> w;
    const int x0 = bx * B, y0 = by * B, bw = min(B, a.W - x0), bh = min(B, a.H - y0);
    w.on = 0;
    w.whole = walk && bw == B && bh == B;
    const uint8_t* home = a.cur + (size_t)t.s * a.cur_stream + (size_t)y0 * a.cur_pitch + (size_t)x0 * 3;
    // two aligned words around any pixel of the block lie inside the buffer (the same in all lanes)
    const bool words = home - 3 >= a.cur && home + (size_t)(B - 1) * a.cur_pitch + (size_t)B * 3 + 8 <= a.cur_end;
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {                                 // issued first: in flight while the window is staged
        const int p = i * 32 + lane, r = p / B, c = p - r * B;
        const bool exists = p < B * B;
        w.off[i] = exists ? (uint32_t)(r * (PT ? PT : a.win_pitch) + c) * 4u : 0u;     // a lane without a last pixel reads the block's first one, masked
        w.cw[i] = 0;
        if (w.whole && words) {
            const uint8_t* q = home + (exists ? (size_t)r * a.cur_pitch + c * 3 : 0);
            const uint32_t* v = (const uint32_t*)((uintptr_t)q & ~(uintptr_t)3);
            w.cw[i] = __funnelshift_r(dc_ld(v), dc_ld(v + 1), ((uint32_t)(uintptr_t)q & 3u) * 8u) & 0x00ffffffu;
            if (exists) w.on |= 1u << i;
        } else if (walk && r < bh && c < bw) {
            w.on |= 1u << i;
            w.cw[i] = load_pixel(home + (size_t)r * a.cur_pitch + c * 3, a.cur, a.cur_end);
        }
    }
    if (threadIdx.x < 4) sums[threadIdx.x] = 0;
    stage_window(a, t, win);
    __syncthreads();
    if (walk) {
        w.base = (uint32_t)__cvta_generic_to_shared(win) + (uint32_t)((ly * B + a.Rw) * (PT ? PT : a.win_pitch) + lx * B + a.Rw) * 4u;
        if (FAR) { w.args = &a; w.home = a.prev + (size_t)t.s * a.prev_stream + (size_t)y0 * a.prev_pitch + (size_t)x0 * 3; }
        w.pitch4_ = a.win_pitch * 4;
        w.valid = Within{disp(max(-a.R, -x0), max(-a.R, -y0)), disp(min(a.R, a.W - bw - x0), min(a.R, a.H - bh - y0))};
        if (a.search == DC_SEARCH_THREE_STEP) w.three_step(a.R); else w.diamond(a.R, a.status);
        if (lane == 0) publish(a, t, bx, by, disp_x(w.at), disp_y(w.at), w.bs, sums);
    } else if (block && lane == 0) {
        mark_skipped(a, t, bx, by);
    }
    flush_sums(a, t, sums);
}

// ---- every displacement ------------------------------------------------------------------------------------------------
// A block's candidates are (2R + 1) columns dx times ceil((2R + 1) / E_ROWS) groups of rows dy; the items are dealt to
// lanes, 32 at a time to a warp, so that a block of a small range still fills warps and a small frame fills the CTA.
__global__ void __launch_bounds__(kMaxWarps * 32) k_win_all(const dc_win_args a)
{
    extern __shared__ __align__(16) uint32_t win[];
    __shared__ int32_t sums[4];
    __shared__ unsigned long long best[kMaxWarps];                    // per block of the tile
    uint32_t* cur = win + a.win_rows * a.win_pitch;                   // [TX * TY][B * B]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    dc_pdl_wait();
    dc_pdl_release();
    const Tile t = tile_of(a);
    if (!any_mine(a, t)) return;
    const int nblk = a.TX * a.TY, BB = a.B * a.B;
    for (int i = threadIdx.x; i < nblk * BB; i += blockDim.x) {
        const int k = i / BB, p = i - k * BB, r = p / a.B, c = p - r * a.B;
        const int bx = t.bx0 + k % a.TX, by = t.by0 + k / a.TX, x = bx * a.B + c, y = by * a.B + r;
        cur[i] = x < a.W && y < a.H ? load_pixel(a.cur + (size_t)t.s * a.cur_stream + (size_t)y * a.cur_pitch + (size_t)x * 3, a.cur, a.cur_end) : 0u;
    }
    if (threadIdx.x < kMaxWarps) best[threadIdx.x] = ~0ull;
    if (threadIdx.x < 4) sums[threadIdx.x] = 0;
    stage_window(a, t, win);
    __syncthreads();
    const int n_d = 2 * a.R + 1, chunks = (n_d + E_ROWS - 1) / E_ROWS, items = n_d * chunks, groups = (items + 31) >> 5;
    for (int u = warp; u < nblk * groups; u += warps) {
        const int k = u / groups, lx = k % a.TX, ly = k / a.TX, bx = t.bx0 + lx, by = t.by0 + ly;
        if (lx >= t.nbx || ly >= t.nby || !mine(a, bx, by) || !searched(a, bx, by)) continue;
        const int x0 = bx * a.B, y0 = by * a.B, bw = min(a.B, a.W - x0), bh = min(a.B, a.H - y0);
        const int item = min((u - k * groups) * 32 + lane, items - 1);    // surplus lanes repeat the last item
        const int chunk = item / n_d, dxi = item - chunk * n_d;
        uint32_t acc[E_ROWS];
#pragma unroll
        for (int d = 0; d < E_ROWS; ++d) acc[d] = 0;
        const uint32_t* col = win + (ly * a.B + chunk * E_ROWS) * a.win_pitch + lx * a.B + dxi;     // dy = -R + chunk * E_ROWS, block row 0
        const uint32_t* cc = cur + k * BB;
#pragma unroll 1
        for (int x = 0; x < bw; ++x) {
            uint32_t w[E_ROWS];                                       // rows y .. y + E_ROWS - 1 of the column, as a ring
#pragma unroll
            for (int d = 0; d < E_ROWS - 1; ++d) w[d] = col[d * a.win_pitch + x];
            const uint32_t* next = col + (E_ROWS - 1) * a.win_pitch + x;
            const uint32_t* pc = cc + x;
#pragma unroll 1
            for (int yb = 0; yb < bh; yb += E_ROWS) {
                if (yb + E_ROWS <= bh) {                              // all rows of the group at once: their loads travel together
                    uint32_t v[E_ROWS], p[E_ROWS];
#pragma unroll
                    for (int j = 0; j < E_ROWS; ++j) { v[j] = next[j * a.win_pitch]; p[j] = pc[j * a.B]; }
#pragma unroll
                    for (int j = 0; j < E_ROWS; ++j) {
                        w[(j + E_ROWS - 1) % E_ROWS] = v[j];
#pragma unroll
                        for (int d = 0; d < E_ROWS; ++d) { const uint32_t e = __vabsdiffu4(p[j], w[(j + d) % E_ROWS]); acc[d] = __dp4a(e, e, acc[d]); }
                    }
                    next += E_ROWS * a.win_pitch; pc += E_ROWS * a.B;
                    continue;
                }
#pragma unroll
                for (int j = 0; j < E_ROWS - 1; ++j) {                // the remaining rows, fewer than E_ROWS
                    if (yb + j >= bh) break;                          // the same in all lanes
                    w[(j + E_ROWS - 1) % E_ROWS] = *next;
                    const uint32_t p = *pc;
                    next += a.win_pitch; pc += a.B;
#pragma unroll
                    for (int d = 0; d < E_ROWS; ++d) { const uint32_t e = __vabsdiffu4(p, w[(j + d) % E_ROWS]); acc[d] = __dp4a(e, e, acc[d]); }
                }
            }
        }
        const int dx = dxi - a.R, dy0 = chunk * E_ROWS - a.R;
        const bool x_ok = x0 + dx >= 0 && x0 + dx + bw <= a.W;
        unsigned long long key = ~0ull;
#pragma unroll
        for (int d = 0; d < E_ROWS; ++d) {
            const int dy = dy0 + d;
            if (x_ok && dy <= a.R && y0 + dy >= 0 && y0 + dy + bh <= a.H) {
                const unsigned long long v = ((unsigned long long)acc[d] << 32) | tie_key(dx, dy);
                key = v < key ? v : key;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o);
            key = other < key ? other : key;
        }
        if (lane == 0) atomicMin(&best[k], key);
    }
    __syncthreads();
    if (threadIdx.x < nblk) {
        const int lx = threadIdx.x % a.TX, ly = threadIdx.x / a.TX, bx = t.bx0 + lx, by = t.by0 + ly;
        if (lx < t.nbx && ly < t.nby && mine(a, bx, by)) {
            const unsigned long long k = best[threadIdx.x];           // the zero vector is always a candidate
            if (searched(a, bx, by)) publish(a, t, bx, by, (int)(k & 0xff) - 128, (int)((k >> 8) & 0xff) - 128, (uint32_t)(k >> 32), sums);
            else mark_skipped(a, t, bx, by);
        }
    }
    flush_sums(a, t, sums);
}

template <typename K>
int launch(K kernel, const dc_win_args& a, int threads, size_t smem, int device, dc_once_per_device& attr_set, cudaStream_t stream)
{
    if (attr_set.first(device)) DC_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024));
    DC_CUDA(dc_launch_pdl(kernel, dim3((unsigned)a.tiles_x, (unsigned)a.tiles_y, (unsigned)a.S), threads, smem, stream, a));
    return DC_OK;
}

}  // namespace

int dc_launch_search_win(dc_win_args a, int num_sms, int device, cudaStream_t stream)
{
    const bool all = a.search == DC_SEARCH_EXHAUSTIVE;
    const int iters = dc_div_up(a.B * a.B, 32);                       // pixels a lane owns
    size_t smem = 0;
    bool known = false;                                               // the instance that knows block edge and pitch
    auto shape = [&](int TX, int TY) {
        a.TX = TX; a.TY = TY; a.inv_TX = (65536 + TX - 1) / TX;
        a.tiles_x = dc_div_up(a.Gx, TX); a.tiles_y = dc_div_up(a.Gy, TY);
        a.win_cols = ((TX * a.B + 2 * (a.Rw - a.margin) + 3) & ~3) + 2 * a.margin;   // staged in groups of four
        a.win_rows = TY * a.B + 2 * a.Rw + (all ? E_ROWS - 1 : 0);    // rows only touched by displacements beyond R (scored, never compared)
        a.win_pitch = known ? walk_pitch(a.B) : a.win_cols + ((a.B - a.win_cols) % 32 + 32) % 32;   // = B modulo 32
        smem = (size_t)a.win_rows * a.win_pitch * 4 + (all ? (size_t)TX * TY * a.B * a.B * 4 : 0);
    };
    // Wide tiles stage fewer window pixels per block; they shrink while the window is too large for three CTAs per SM, and
    // while the frames have fewer tiles than the machine has SMs (down to two blocks, one for the exhaustive search).
    int TX = 0, TY = 0;
    auto fit = [&](int Rw) {                                          // returns the window pixels staged per block
        a.Rw = Rw; a.margin = 0;
        TX = a.Gx < 8 ? a.Gx : 8; TY = TX < 4 ? 4 : 2;
        if (TY > a.Gy) TY = a.Gy;
        shape(TX, TY);
        while (TX * TY > 1 && (smem > 200 * 1024 || (TX * TY > 2 && smem > 72 * 1024) ||
                               ((long long)a.tiles_x * a.tiles_y * a.S < num_sms && TX * TY > (all ? 1 : 2)))) {
            if (TY > 1 && (TY > TX || smem <= 72 * 1024)) TY = (TY + 1) / 2; else if (TX > 1) TX = (TX + 1) / 2; else TY = (TY + 1) / 2;
            shape(TX, TY);
        }
        return a.win_rows * a.win_cols / (TX * TY);
    };
    // Walks over a long range: a window of kWalkReach where that stages less than a fifth per block.  (Match calls with the whole
    // window and with the capped one, range 64, diamond: 1080p, 16 streams, 8-pixel blocks, 13 times the pixels: 13456 and 1610 us;
    // 20 pixels, 6.6 times: 4145 and 2184; 227 x 227, 24 pixels, 2.7 times: 72 and 125.  Range 40, 1.4 to 1.8 times: 513 and 571.)
    const int whole = fit(a.R);
    bool far = !all && a.R > kWalkReach;
    if (far && whole <= 5 * fit(kWalkReach)) { far = false; fit(a.R); }
    // exhaustive: as many warps as there are groups of 32 items, up to 16
    const int n_d = 2 * a.R + 1, groups = (n_d * dc_div_up(n_d, E_ROWS) + 31) / 32;
    int warps = TX * TY < 8 ? 8 : TX * TY;                            // walks: a warp per block; spare ones help to stage the window
    if (all) { const long long units = (long long)TX * TY * groups; warps = units < 4 ? 4 : units > kMaxWarps ? kMaxWarps : (int)units; }
    const bool few = (long long)a.tiles_x * a.tiles_y * a.S <= 2 * num_sms;
    // The points around a centre at the end of the range lie up to two pixels beyond it: room for them (not staged), and the pitch of an instance
    // that knows it, where the tile keeps its CTAs per SM.  (1080p, 4 streams, diamond, 16 pixels, range 48: 577 us with tiles shrunk to make that
    // room, 282 with a known pitch whatever it costs, 262 so.)  Large blocks of a short range have no use for it: so many of a round's points
    // are no candidates that a path of their own is cheaper (32 pixels, range 8: 239 and 209 us, range 16 335 and 318; 24 pixels, range 24, 278 and
    // 284; four streams of 640 x 360, two tiles per SM, 32 pixels, range 16, 27.9 and 28.8).
    bool edge = false;
    if (a.search == DC_SEARCH_DIAMOND && !far) {
        const int threads = iters > 8 ? 512 : iters <= 4 && !few ? 1536 : 1024;   // an SM's, by the registers of the instance (launch bounds of k_win_walk)
        auto ctas = [&] { const int by_smem = (int)(228 * 1024 / (smem + 1024 + 64)), by_regs = threads / (warps * 32); return by_smem < by_regs ? by_smem : by_regs; };
        const int most = few && ctas() > 2 ? 2 : ctas();
        a.Rw += 2; a.margin = 2;
        known = a.B <= 16 && ((TX * a.B + 2 * a.R + 3) & ~3) + 4 <= walk_pitch(a.B);
        shape(TX, TY);
        if (known && ctas() < most) { known = false; shape(TX, TY); }
        edge = ctas() < most || (iters > 8 && a.R <= (iters <= 16 ? 6 : few ? 8 : 16));
        if (edge) { a.Rw -= 2; a.margin = 0; shape(TX, TY); }
    }
    if (all) { static dc_once_per_device set; return launch(k_win_all, a, warps * 32, smem, device, set, stream); }
    // one instance per block edge up to 16, for ranges whose window fits its pitch (three step search: addresses with run-time steps gain
    // nothing from it), and one per number of pixels a lane owns
#define DC_WALK_(n, ...) { static dc_once_per_device set; return launch(k_win_walk<n, __VA_ARGS__>, a, warps * 32, smem, device, set, stream); }
    if (known) switch (a.B) {
#define DC_WALK(b) case b: if (few) DC_WALK_((b * b + 31) / 32, false, b, true) DC_WALK_((b * b + 31) / 32, false, b, false)
        DC_WALK(4) DC_WALK(5) DC_WALK(6) DC_WALK(7) DC_WALK(8) DC_WALK(9) DC_WALK(10) DC_WALK(11)
#undef DC_WALK
#define DC_WALK(b) case b: DC_WALK_((b * b + 31) / 32, false, b, false)
        DC_WALK(12) DC_WALK(13) DC_WALK(14) DC_WALK(15) DC_WALK(16)
#undef DC_WALK
    }
#define DC_WALK(n) { if (far) DC_WALK_(n, true, 0, false) if (edge) DC_WALK_(n, false, 0, false, true) DC_WALK_(n, false, 0, false) }
    switch (iters) {
    case 1: DC_WALK(1)
    case 2: DC_WALK(2)
    case 3: DC_WALK(3)
    case 4: DC_WALK(4)
    case 5: DC_WALK(5)
    case 6: DC_WALK(6)
    case 7: DC_WALK(7)
    case 8: DC_WALK(8)
    default: if (iters <= 16) DC_WALK(16) DC_WALK(32)
    }
#undef DC_WALK
#undef DC_WALK_
}
