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
// otherwise instruction issue.  The kernels before kept one warp per block too, but fetched every candidate from global
// memory, two loads and a funnel shift per four bytes (byte by byte without a cache).
#include "dc_common.cuh"
#include "dc_search_win.cuh"

namespace {

constexpr int E_ROWS = 8;                 // vertical displacements a lane scores together
constexpr int kMaxWarps = 16;
// Pixels around the tile that walks over a longer range stage at least.  A walk visits a few dozen candidates near its start;
// staging 64 pixels on every side of a few small blocks cost more than all of them (see dc_launch_search_win).
constexpr int kWalkReach = 32;

__device__ __forceinline__ uint32_t tie_of(int dx, int dy)
{
    return ((uint32_t)(abs(dx) + abs(dy)) << 16) | ((uint32_t)(dy + 128) << 8) | (uint32_t)(dx + 128);
}

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
    const int tx = blockIdx.x % a.tiles_x, u = blockIdx.x / a.tiles_x;
    t.s = u / a.tiles_y;
    t.bx0 = tx * a.TX; t.by0 = (u - t.s * a.tiles_y) * a.TY;
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

// The window, rows warp by warp, a lane four pixels: the 12 bytes come as four aligned words, whatever the row's
// alignment.  Groups that cross the frame's left or right edge, and the few at the ends of the buffer, go pixel by pixel.
// What lies outside the frame is never part of a valid candidate.
__device__ __forceinline__ void stage_window(const dc_win_args& a, const Tile& t, uint32_t* win)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    const int x0 = t.bx0 * a.B - a.Rw, y0 = t.by0 * a.B - a.Rw;
    const uint8_t* prev = a.prev + (size_t)t.s * a.prev_stream;
    const int y_lo = max(y0, 0), y_hi = min(y0 + a.win_rows, a.H) - 1;
    const uint8_t* first = prev + (size_t)y_lo * a.prev_pitch + (size_t)max(x0, 0) * 3;
    const uint8_t* last = prev + (size_t)y_hi * a.prev_pitch + (size_t)min(x0 + a.win_cols, a.W) * 3;
    const bool words = (const uint8_t*)((uintptr_t)first & ~(uintptr_t)3) >= a.prev && last + 8 <= a.prev_end;
    // a narrow window: several rows per warp
    const int lpr = a.win_cols > 64 ? 32 : a.win_cols > 32 ? 16 : 8, rpw = 32 / lpr, l = lane % lpr;
#pragma unroll 2
    for (int y = y_lo + warp * rpw + lane / lpr; y <= y_hi; y += warps * rpw) {
        const uint8_t* row = prev + (size_t)y * a.prev_pitch;
        uint32_t* dst = win + (y - y0) * a.win_pitch;
        for (int c = 4 * l; c < a.win_cols; c += 4 * lpr) {
            const int x = x0 + c;
            if (words && x >= 0 && x + 4 <= a.W) {
                const uint8_t* p = row + (size_t)x * 3;
                const uint32_t* q = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
                const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u, m = 0x00ffffffu;
                const uint32_t w0 = dc_ld(q), w1 = dc_ld(q + 1), w2 = dc_ld(q + 2), w3 = sh ? dc_ld(q + 3) : 0u;
                const uint32_t b0 = __funnelshift_r(w0, w1, sh), b1 = __funnelshift_r(w1, w2, sh), b2 = __funnelshift_r(w2, w3, sh);
                dst[c] = b0 & m; dst[c + 1] = __funnelshift_r(b0, b1, 24) & m; dst[c + 2] = __funnelshift_r(b1, b2, 16) & m; dst[c + 3] = b2 >> 8;
            } else {
                for (int k = 0; k < 4; ++k)
                    if (x + k >= 0 && x + k < a.W) dst[c + k] = load_pixel(row + (size_t)(x + k) * 3, a.prev, a.prev_end);
            }
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
// Points around a centre: 0-7 the large diamond, 8 the centre, 9-12 the small diamond.  A round of the diamond search
// scores one of ten sets: after the move along point `kind` (0-7) the points of the large diamond that are new (the
// others lost to the new centre already and cannot win), 8 the first round, 9 the small diamond.
__host__ __device__ constexpr int pt_x(int i) { constexpr int t[13] = {0, -1, 1, -2, 2, -1, 1, 0, 0, 0, -1, 1, 0}; return t[i]; }
__host__ __device__ constexpr int pt_y(int i) { constexpr int t[13] = {-2, -1, -1, 0, 0, 1, 1, 2, 0, -1, 0, 0, 1}; return t[i]; }
__constant__ int c_pt_x[13] = {0, -1, 1, -2, 2, -1, 1, 0, 0, 0, -1, 1, 0};
__constant__ int c_pt_y[13] = {-2, -1, -1, 0, 0, 1, 1, 2, 0, -1, 0, 0, 1};
constexpr int KIND_FIRST = 8, KIND_SMALL = 9;
__host__ __device__ constexpr uint32_t set_of(int kind)
{
    constexpr uint32_t t[10] = {31u, 11u, 21u, 171u, 213u, 168u, 208u, 248u, 0x1ffu, 0x1e00u};
    return t[kind];
}
__constant__ uint32_t c_set[10] = {31u, 11u, 21u, 171u, 213u, 168u, 208u, 248u, 0x1ffu, 0x1e00u};
// kind of a move (mx, my), indexed by ((my + 2) * 5 + (mx + 2)) >> 1
__constant__ int c_kind[13] = {0, 0, 0, 1, 2, 3, 0, 4, 5, 6, 0, 7, 0};

template <int OFF>
__device__ __forceinline__ uint32_t lds_off(uint32_t p)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(p), "n"(OFF) : "memory");
    return v;
}

// FAR: the window holds fewer than R pixels around the tile.
template <int ITERS, bool FAR>
struct Walk {
    uint32_t base;                  // shared-memory byte address of displacement (0, 0)
    int pitch4;                     // window row in bytes
    int dx_lo, dx_hi, dy_lo, dy_hi; // displacements that keep the block inside the frame and the range
    const dc_win_args* args;        // FAR: where candidates outside the window come from:
    const uint8_t* home;            // the block's position in the previous frame
    uint32_t cw[ITERS], off[ITERS]; // this lane's pixels and their byte offsets in the window
    uint32_t on;                    // which of them exist
    bool whole;                     // the block is not clipped: the first FULL exist in every lane
    static constexpr int FULL = ITERS <= 8 ? ITERS - 1 : ITERS / 2;
    int bx, by; uint32_t bs;        // best point so far and its SSE

    __device__ __forceinline__ bool staged(int cx, int cy, int reach) const
    {
        return !FAR || (abs(cx) + reach <= kWalkReach && abs(cy) + reach <= kWalkReach);
    }
    __device__ __forceinline__ bool inside(int cx, int cy, int reach) const
    {
        return cx - reach >= dx_lo && cx + reach <= dx_hi && cy - reach >= dy_lo && cy + reach <= dy_hi && staged(cx, cy, reach);
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
        if (FAR && !staged(dx, dy, 0)) return far(dx, dy);
        const uint32_t p = base + (uint32_t)(dy * pitch4 + dx * 4);
        uint32_t acc = 0;
#pragma unroll
        for (int i = 0; i < ITERS; ++i) {
            const uint32_t d = ((on >> i) & 1u) ? __vabsdiffu4(cw[i], lds_off<0>(p + off[i])) : 0u;
            acc = __dp4a(d, d, acc);
        }
        return __reduce_add_sync(0xffffffffu, acc);
    }
    // One point under the full order (SSE, |dx| + |dy|, dy, dx).
    __device__ __forceinline__ void consider(int dx, int dy, uint32_t& ns, int& nx, int& ny) const
    {
        if (dx < dx_lo || dx > dx_hi || dy < dy_lo || dy > dy_hi) return;
        const uint32_t s = score(dx, dy);
        if (s < ns || (s == ns && tie_of(dx, dy) < tie_of(nx, ny))) { ns = s; nx = dx; ny = dy; }
    }
    // The points of SET around (cx, cy), all valid, as straight-line code: smallest SSE and its point; tie: two scores
    // that matter were equal, the round has to be redone under the full order.
    template <uint32_t SET>
    __device__ __forceinline__ void fast_set(int cx, int cy, uint32_t& ms, int& mi, bool& tie) const
    {
        const uint32_t pc = base + (uint32_t)(cy * pitch4 + cx * 4);
        uint32_t s[13];
#pragma unroll
        for (int k = 0; k < 13; ++k) s[k] = 0;
#pragma unroll
        for (int i = 0; i < ITERS; ++i) add_point<SET, 0>(i, pc + off[i], s);
        pick<SET, 0>(s, ms, mi, tie);
    }
    template <uint32_t SET, int I>
    __device__ __forceinline__ void add_point(int i, uint32_t p, uint32_t (&s)[13]) const
    {
        if constexpr (I < 13) {
            if constexpr (((SET >> I) & 1u) != 0) {
                uint32_t d = __vabsdiffu4(cw[i], lds_off<pt_x(I) * 4>(p + (uint32_t)(pt_y(I) * pitch4)));
                if (i >= FULL) d &= 0u - ((on >> i) & 1u);
                s[I] = __dp4a(d, d, s[I]);
            }
            add_point<SET, I + 1>(i, p, s);
        }
    }
    template <uint32_t SET, int I>
    __device__ __forceinline__ void pick(const uint32_t (&s)[13], uint32_t& ms, int& mi, bool& tie) const
    {
        if constexpr (I < 13) {
            if constexpr (((SET >> I) & 1u) != 0) {
                const uint32_t v = __reduce_add_sync(0xffffffffu, s[I]);
                tie |= v == ms;
                mi = v < ms ? I : mi;
                ms = min(ms, v);
            }
            pick<SET, I + 1>(s, ms, mi, tie);
        }
    }
    // large diamond until its centre wins, then one small diamond
    __device__ __forceinline__ void diamond(int R, int32_t* status)
    {
        bx = by = 0; bs = 0xffffffffu;
        int kind = KIND_FIRST;
        const int max_moves = (2 * R + 1) * (2 * R + 1);              // every move strictly lowers the key: never reached
#pragma unroll 1
        for (int m = 0;; ++m) {
            const int cx = bx, cy = by;
            uint32_t ms = 0xffffffffu; int mi = 8; bool tie = true;
            if (whole && inside(cx, cy, 2)) {
                tie = false;
                switch (kind) {
                case 0: fast_set<set_of(0)>(cx, cy, ms, mi, tie); break;
                case 1: fast_set<set_of(1)>(cx, cy, ms, mi, tie); break;
                case 2: fast_set<set_of(2)>(cx, cy, ms, mi, tie); break;
                case 3: fast_set<set_of(3)>(cx, cy, ms, mi, tie); break;
                case 4: fast_set<set_of(4)>(cx, cy, ms, mi, tie); break;
                case 5: fast_set<set_of(5)>(cx, cy, ms, mi, tie); break;
                case 6: fast_set<set_of(6)>(cx, cy, ms, mi, tie); break;
                case 7: fast_set<set_of(7)>(cx, cy, ms, mi, tie); break;
                case KIND_FIRST: fast_set<set_of(KIND_FIRST)>(cx, cy, ms, mi, tie); break;
                default: fast_set<set_of(KIND_SMALL)>(cx, cy, ms, mi, tie); break;
                }
                tie |= ms == bs;
            }
            if (!tie) {
                if (ms < bs) { bs = ms; bx = cx + c_pt_x[mi]; by = cy + c_pt_y[mi]; }
            } else {
                uint32_t set = c_set[kind], ns = bs; int nx = cx, ny = cy;
                if (kind == KIND_FIRST) { ns = score(0, 0); set &= ~0x100u; }     // the centre is the first candidate
#pragma unroll 1
                while (set) {
                    const int i = __ffs(set) - 1;
                    set &= set - 1;
                    consider(cx + c_pt_x[i], cy + c_pt_y[i], ns, nx, ny);
                }
                bs = ns; bx = nx; by = ny;
            }
            if (kind == KIND_SMALL) return;
            if (bx == cx && by == cy) { kind = KIND_SMALL; continue; }
            if (m >= max_moves) { if ((threadIdx.x & 31) == 0 && status) atomicExch(status, (int)DC_ERR_TIMEOUT); return; }
            kind = c_kind[((by - cy + 2) * 5 + (bx - cx + 2)) >> 1];
        }
    }
    // nine-point passes with step S0, S0/2, ..., 1; S0 = largest power of two with 2 S0 - 1 <= R
    __device__ __forceinline__ void three_step(int R)
    {
        bx = by = 0; bs = score(0, 0);
        int step = R < 1 ? 0 : 1;
        while (step > 0 && 4 * step - 1 <= R) step *= 2;
#pragma unroll 1
        for (; step >= 1; step >>= 1) {
            const int cx = bx, cy = by;
            bool tie = true;
            uint32_t ms = 0xffffffffu; int mi = 4;
            if (whole && inside(cx, cy, step)) {
                tie = false;
                const uint32_t pc = base + (uint32_t)(cy * pitch4 + cx * 4);
                uint32_t s[9];
#pragma unroll
                for (int k = 0; k < 9; ++k) s[k] = 0;
#pragma unroll
                for (int i = 0; i < ITERS; ++i)
#pragma unroll
                    for (int k = 0; k < 9; ++k)
                        if (k != 4) {
                            uint32_t d = __vabsdiffu4(cw[i], lds_off<0>(pc + off[i] + (uint32_t)((k / 3 - 1) * step * pitch4 + (k % 3 - 1) * step * 4)));
                            if (i >= FULL) d &= 0u - ((on >> i) & 1u);
                            s[k] = __dp4a(d, d, s[k]);
                        }
#pragma unroll
                for (int k = 0; k < 9; ++k)
                    if (k != 4) {
                        const uint32_t v = __reduce_add_sync(0xffffffffu, s[k]);
                        tie |= v == ms;
                        mi = v < ms ? k : mi;
                        ms = min(ms, v);
                    }
                tie |= ms == bs;
            }
            if (!tie) {
                if (ms < bs) { bs = ms; bx = cx + (mi % 3 - 1) * step; by = cy + (mi / 3 - 1) * step; }
            } else {
                uint32_t ns = bs; int nx = cx, ny = cy;
#pragma unroll 1
                for (int k = 0; k < 9; ++k)
                    if (k != 4) consider(cx + (k % 3 - 1) * step, cy + (k / 3 - 1) * step, ns, nx, ny);
                bs = ns; bx = nx; by = ny;
            }
        }
    }
};

// three CTAs per SM where the lane's pixels leave the registers for it (10-pixel blocks, 720p, 4 streams: 78 us, 90 with
// two; 16-pixel blocks with three: twice as slow)
template <int ITERS, bool FAR>
__global__ void __launch_bounds__(kMaxWarps * 32, ITERS <= 4 && !FAR ? 3 : ITERS <= 8 ? 2 : 1) k_win_walk(const __grid_constant__ dc_win_args a)
{
    extern __shared__ __align__(16) uint32_t win[];
    __shared__ int32_t sums[4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    dc_pdl_wait();
    dc_pdl_release();
    const Tile t = tile_of(a);
    if (!any_mine(a, t)) return;
    const int ly = warp / a.TX, lx = warp - ly * a.TX, bx = t.bx0 + lx, by = t.by0 + ly;
    const bool block = ly < a.TY && lx < t.nbx && ly < t.nby && mine(a, bx, by), walk = block && searched(a, bx, by);
    Walk<ITERS, FAR> w;
    const int x0 = bx * a.B, y0 = by * a.B, bw = min(a.B, a.W - x0), bh = min(a.B, a.H - y0);
    w.on = 0;
#pragma unroll
    for (int i = 0; i < ITERS; ++i) {                                 // issued first: in flight while the window is staged
        const int p = i * 32 + lane, r = p / a.B, c = p - r * a.B;
        w.cw[i] = 0;
        w.off[i] = p < a.B * a.B ? (uint32_t)(r * a.win_pitch + c) * 4u : 0u;   // a lane without a last pixel reads the block's first one, masked
        if (walk && r < bh && c < bw) {
            w.on |= 1u << i;
            w.cw[i] = load_pixel(a.cur + (size_t)t.s * a.cur_stream + (size_t)(y0 + r) * a.cur_pitch + (size_t)(x0 + c) * 3, a.cur, a.cur_end);
        }
    }
    if (threadIdx.x < 4) sums[threadIdx.x] = 0;
    stage_window(a, t, win);
    __syncthreads();
    if (walk) {
        w.base = (uint32_t)__cvta_generic_to_shared(win) + (uint32_t)((ly * a.B + a.Rw) * a.win_pitch + lx * a.B + a.Rw) * 4u;
        if (FAR) { w.args = &a; w.home = a.prev + (size_t)t.s * a.prev_stream + (size_t)y0 * a.prev_pitch + (size_t)x0 * 3; }
        w.pitch4 = a.win_pitch * 4;
        w.dx_lo = max(-a.R, -x0); w.dx_hi = min(a.R, a.W - bw - x0); w.dy_lo = max(-a.R, -y0); w.dy_hi = min(a.R, a.H - bh - y0);
        w.whole = bw == a.B && bh == a.B;
        if (a.search == DC_SEARCH_THREE_STEP) w.three_step(a.R); else w.diamond(a.R, a.status);
        if (lane == 0) publish(a, t, bx, by, w.bx, w.by, w.bs, sums);
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
                const unsigned long long v = ((unsigned long long)acc[d] << 32) | tie_of(dx, dy);
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
    DC_CUDA(dc_launch_pdl(kernel, dim3((unsigned)(a.tiles_x * a.tiles_y * a.S)), threads, smem, stream, a));
    return DC_OK;
}

}  // namespace

int dc_launch_search_win(dc_win_args a, int num_sms, int device, cudaStream_t stream)
{
    const bool all = a.search == DC_SEARCH_EXHAUSTIVE;
    size_t smem = 0;
    auto shape = [&](int TX, int TY) {
        a.TX = TX; a.TY = TY;
        a.tiles_x = dc_div_up(a.Gx, TX); a.tiles_y = dc_div_up(a.Gy, TY);
        a.win_cols = (TX * a.B + 2 * a.Rw + 3) & ~3;                  // staged in groups of four
        a.win_rows = TY * a.B + 2 * a.Rw + (all ? E_ROWS - 1 : 0);    // rows only touched by displacements beyond R (scored, never compared)
        a.win_pitch = a.win_cols + ((a.B - a.win_cols) % 32 + 32) % 32;   // = B modulo 32
        smem = (size_t)a.win_rows * a.win_pitch * 4 + (all ? (size_t)TX * TY * a.B * a.B * 4 : 0);
    };
    // Wide tiles stage fewer window pixels per block; they shrink while the window is too large for three CTAs per SM, and
    // while the frames have fewer tiles than the machine has SMs (down to two blocks, one for the exhaustive search).
    int TX = 0, TY = 0;
    auto fit = [&](int Rw) {                                          // returns the window pixels staged per block
        a.Rw = Rw;
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
    if (all) { static dc_once_per_device set; return launch(k_win_all, a, warps * 32, smem, device, set, stream); }
    // one instance per number of pixels a lane owns, up to 16-pixel blocks
#define DC_WALK_(n, f) { static dc_once_per_device set; return launch(k_win_walk<n, f>, a, warps * 32, smem, device, set, stream); }
#define DC_WALK(n) { if (far) DC_WALK_(n, true) DC_WALK_(n, false) }
    switch (dc_div_up(a.B * a.B, 32)) {
    case 1: DC_WALK(1)
    case 2: DC_WALK(2)
    case 3: DC_WALK(3)
    case 4: DC_WALK(4)
    case 5: DC_WALK(5)
    case 6: DC_WALK(6)
    case 7: DC_WALK(7)
    case 8: DC_WALK(8)
    default: if (a.B * a.B <= 512) DC_WALK(16) DC_WALK(32)
    }
#undef DC_WALK
#undef DC_WALK_
}
