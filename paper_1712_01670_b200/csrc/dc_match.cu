// Image block matching (Section 4, Steps 1-5) on the GPU.  Integer arithmetic only.
//
//   dc_search_win.cu  Step 2 for other block sizes and for blocks clipped by the frame's edge.  Candidates are ordered
//              by (SSE, |dx|+|dy|, dy, dx).  Blocks that pass the PSNR bound add their vector to the Step 3 sums.
//   k_search_dsw  Step 2 for 16-pixel blocks with diamond search (the common case): one CTA per 8 x 2
//              blocks, the previous frame's window staged once in shared memory as one word per pixel; one
//              warp per block, lane 2r + h scoring every other pixel of block row r, so that loads are free of
//              bank conflicts and of byte realignment; points already scored by the previous diamond are
//              skipped (they cannot win).  Walks that leave the window continue in k_search_dsw_long with
//              private windows.
//   k_search_tss16  Step 2 for 16-pixel blocks with three step search: the same lane layout, one window that
//              covers the whole reach of the search.
//   k_verify   Steps 3-4: rounds the mean vector M, scores every block at M (reusing the Step 2
//              score when the block's own best vector is M); k_verify16_prep / k_verify16_list, or k_verify16_few, for 16-pixel blocks.
//   k_merge    Step 5: maximal horizontal runs per block row, merged vertically when the
//              spans are identical, emitted in (y, x) order by a CTA-wide ordered compaction.
#include "dc_common.cuh"
#include "dc_search_win.cuh"
#include "dc_walk.cuh"

namespace {


struct MatchArgs {
    const uint8_t* cur;  size_t cur_pitch;  size_t cur_stream;
    const uint8_t* prev; size_t prev_pitch; size_t prev_stream;
    uint8_t* copy; size_t copy_pitch, copy_stream;   // where the search of 16-pixel blocks leaves the new frame in key-frame layout, or NULL
    int W, H, B, R, Gx, Gy, S, search, skip_k, region_mode;
    uint32_t limit[4];
    int16_t* mv; uint32_t* sse; uint8_t* matched; int32_t* acc; int32_t* gmv;
    int32_t* status;                     // device status word: a walk ended by its step limit records DC_ERR_TIMEOUT
};

// (SSE, |dx| + |dy|, dy, dx) packed into one integer: tie_key behind the SSE, in 64-bit steps, which the exhaustive search is 2% faster with.
__device__ __forceinline__ unsigned long long cand_key(uint32_t sse, int dx, int dy)
{
    return ((unsigned long long)sse << 32) | ((unsigned long long)(abs(dx) + abs(dy)) << 16) |
           ((unsigned long long)(dy + 128) << 8) | (unsigned long long)(dx + 128);
}

__device__ __forceinline__ int limit_index(const MatchArgs& a, int bw, int bh)
{
    return (bh < a.B ? 2 : 0) + (bw < a.B ? 1 : 0);
}

// mean of n values with sum `sum`, rounded to nearest, halves away from zero
__device__ __forceinline__ int round_mean(int sum, int n)
{
    int m = (2 * abs(sum) + n) / (2 * n);
    return sum < 0 ? -m : m;
}

// Per-block mode, in place of Step 4: a searched block is accepted with its own vector when that match passed
// the PSNR test of Step 2.  One thread per block.  The global vector is still reported.
__global__ void k_accept_own(MatchArgs a)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int per = a.Gx * a.Gy;
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= per * a.S) return;
    const int s = gi / per, b = gi - s * per, by = b / a.Gx, bx = b - by * a.Gx;
    const int bw = min(a.B, a.W - bx * a.B), bh = min(a.B, a.H - by * a.B);
    const uint32_t v = a.sse[gi];
    const int ok = v != 0xffffffffu && v <= a.limit[limit_index(a, bw, bh)];
    a.matched[gi] = (uint8_t)ok;
    if (ok) atomicAdd(&a.acc[4 * s + 3], 1);
    if (b == 0) {
        const int K = a.acc[4 * s + 2];
        a.gmv[3 * s] = K > 0 ? round_mean(a.acc[4 * s + 0], K) : 0;
        a.gmv[3 * s + 1] = K > 0 ? round_mean(a.acc[4 * s + 1], K) : 0;
        a.gmv[3 * s + 2] = K;
    }
}

struct Step4 { int Mx, My, K; bool settled; int ok; };
// The global motion of stream s, and block b (number gi in all) where no pixels are needed to settle it.
__device__ __forceinline__ Step4 settle(const MatchArgs& a, int B, unsigned gi, int s, int b, bool in_grid)
{
    const int by = b / a.Gx, bx = b - by * a.Gx, x0 = bx * B, y0 = by * B, bw = min(B, a.W - x0), bh = min(B, a.H - y0);
    const int4 sums = __ldcg((const int4*)a.acc + s);                            // Step 3: sum dx, sum dy, K (one 16-byte load)
    Step4 r = {0, 0, sums.z, false, 0};
    if (r.K > 0) { r.Mx = round_mean(sums.x, r.K); r.My = round_mean(sums.y, r.K); }
    const bool cand_ok = in_grid && r.K > 0 && abs(r.Mx) <= a.R && abs(r.My) <= a.R && x0 + r.Mx >= 0 && y0 + r.My >= 0 &&
                         x0 + r.Mx + bw <= a.W && y0 + r.My + bh <= a.H;
    bool known = false; uint32_t v = 0;
    if (cand_ok) {
        const uint32_t own = ((const uint32_t*)a.mv)[gi];                         // (dx, dy) as one word
        v = a.sse[gi];
        known = (int16_t)(own & 0xffffu) == r.Mx && (int16_t)(own >> 16) == r.My && v != 0xffffffffu;
    }
    r.settled = in_grid && (!cand_ok || known);
    r.ok = known && v <= a.limit[limit_index(a, bw, bh)];
    return r;
}
// The SSE of row r of block b displaced by (Mx, My), for any block size: the aligned words that hold the row in the new frame, the previous
// frame's bytes shifted to their places, five words in flight.
__device__ __forceinline__ uint32_t row_sse(const MatchArgs& a, int s, int b, int Mx, int My, int r, bool on)
{
    const int by = b / a.Gx, bx = b - by * a.Gx, x0 = bx * a.B, y0 = by * a.B, bw = min(a.B, a.W - x0), bh = min(a.B, a.H - y0);
    if (!on || r >= bh) return 0;
    const uint8_t* c = a.cur + (size_t)s * a.cur_stream + (size_t)(y0 + r) * a.cur_pitch + (size_t)x0 * 3;
    const int skip = (int)((uintptr_t)c & 3u), words = (skip + bw * 3 + 3) >> 2, tail = skip + bw * 3 - 4 * (words - 1);   // 1 to 4 bytes of the last word
    const uint8_t* p = a.prev + (size_t)s * a.prev_stream + (size_t)(y0 + My + r) * a.prev_pitch + (size_t)(x0 + Mx) * 3 - skip;
    const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u;
    const uint32_t* cq = (const uint32_t*)(c - skip);
    const uint32_t* pq = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
    uint32_t acc = 0, lo = (const uint8_t*)pq >= a.prev ? dc_ld(pq) : 0u;        // bytes before the row are masked; none lie before the buffer
    for (int j0 = 0; j0 < words; j0 += 5) {
        uint32_t cw[5], hi[5];
#pragma unroll
        for (int j = 0; j < 5; ++j) { const bool in = j0 + j < words; cw[j] = in ? dc_ld(cq + j0 + j) : 0u; hi[j] = in ? dc_ld(pq + j0 + j + 1) : 0u; }
#pragma unroll
        for (int j = 0; j < 5; ++j) {
            uint32_t m = j0 + j < words ? 0xffffffffu : 0u;
            if (j0 + j == words - 1) m >>= 8 * (4 - tail);
            if (j0 + j == 0) m &= 0xffffffffu << (8 * skip);
            const uint32_t d = __vabsdiffu4(cw[j], __funnelshift_r(lo, hi[j], sh)) & m;
            acc = __dp4a(d, d, acc);
            lo = hi[j];
        }
    }
    return acc;
}

// The same of a whole block, for blocks of more than 16 pixels, by a warp: a lane has a word of a row, of every second row where a row has at
// most 16 words, so that the lanes of a load lie side by side; eight rows in flight.
__device__ __forceinline__ uint32_t wide_sse(const MatchArgs& a, int s, int b, int Mx, int My, int lane)
{
    const int by = b / a.Gx, bx = b - by * a.Gx, x0 = bx * a.B, y0 = by * a.B, bw = min(a.B, a.W - x0), bh = min(a.B, a.H - y0);
    const uint8_t* c = a.cur + (size_t)s * a.cur_stream + (size_t)y0 * a.cur_pitch + (size_t)x0 * 3;
    // the pitches of key frames are multiples of 16: every row starts at the same place in its word
    const int skip = (int)((uintptr_t)c & 3u), words = (skip + bw * 3 + 3) >> 2, tail = skip + bw * 3 - 4 * (words - 1);     // 1 to 4 bytes of the last word
    const uint8_t* p = a.prev + (size_t)s * a.prev_stream + (size_t)(y0 + My) * a.prev_pitch + (size_t)(x0 + Mx) * 3 - skip;
    const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u;
    const bool two = words <= 16;
    const int j = two ? lane & 15 : lane, first = two ? lane >> 4 : 0, step = two ? 2 : 1;
    uint32_t m = j < words ? 0xffffffffu : 0u;
    if (j == words - 1) m >>= 8 * (4 - tail);
    if (j == 0) m &= 0xffffffffu << (8 * skip);
    const uint8_t* cq = c - skip + 4 * j;
    const uint8_t* pq = (const uint8_t*)((uintptr_t)p & ~(uintptr_t)3) + 4 * j;
    uint32_t acc = 0;
    for (int r0 = first; r0 < bh; r0 += 8 * step) {
        uint32_t cw[8], lo[8], hi[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int r = r0 + k * step;
            const bool in = r < bh && j < words;
            const uint32_t* q = (const uint32_t*)(pq + (size_t)r * a.prev_pitch);
            cw[k] = in ? dc_ld((const uint32_t*)(cq + (size_t)r * a.cur_pitch)) : 0u;
            lo[k] = in && (const uint8_t*)q >= a.prev ? dc_ld(q) : 0u;           // bytes before the row are masked; none lie before the buffer
            hi[k] = in ? dc_ld(q + 1) : 0u;
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const uint32_t d = __vabsdiffu4(cw[k], __funnelshift_r(lo[k], hi[k], sh)) & m;
            acc = __dp4a(d, d, acc);
        }
    }
    return __reduce_add_sync(0xffffffffu, acc);
}

// Steps 3-4 for any block size (16-pixel blocks have kernels of their own).  A warp takes `share` blocks: a lane settles one from its own
// vector where that is M, or where M leaves the frame or the range, then the warp scores the others: two at a time, 16 lanes each, one per row,
// or (WIDE: more than 16 pixels) one at a time.
// What bounds it: the latency of a row's loads.  us with a warp per block that fetched every block byte by byte, with a lane per row also of large
// blocks, and so: 720p, 4 streams, 10 pixels, 29, 12.5, 12.5; 1080p, 2 streams, 20 pixels, 30, 210 (a load's rows in as many lines), 22.
template <bool WIDE>
__global__ void __launch_bounds__(256) k_verify(MatchArgs a, int share)
{
    dc_pdl_wait();
    dc_pdl_release();
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31, r = lane & 15, half = lane >> 4, per = a.Gx * a.Gy;
    const unsigned gi = (blockIdx.x * 8u + (threadIdx.x >> 5)) * (unsigned)share + (unsigned)lane;
    const bool in_grid = lane < share && gi < (unsigned)(per * a.S);
    const int s = in_grid ? (int)(gi / (unsigned)per) : a.S - 1, b = in_grid ? (int)(gi - (unsigned)s * per) : 0;
    const Step4 v = settle(a, a.B, gi, s, b, in_grid);
    int ok = v.ok;
    if (in_grid && b == 0) { a.gmv[3 * s] = v.Mx; a.gmv[3 * s + 1] = v.My; a.gmv[3 * s + 2] = v.K; }
    const int by = b / a.Gx, bx = b - by * a.Gx;
    const uint32_t limit = a.limit[limit_index(a, min(a.B, a.W - bx * a.B), min(a.B, a.H - by * a.B))];
    unsigned todo = __ballot_sync(all, in_grid && !v.settled);
    while (todo) {                                                               // the same in all lanes
        const int mine = __ffs(todo) - 1;
        todo &= todo - 1;
        if constexpr (WIDE) {
            const uint32_t sse = wide_sse(a, __shfl_sync(all, s, mine), __shfl_sync(all, b, mine), __shfl_sync(all, v.Mx, mine), __shfl_sync(all, v.My, mine), lane);
            if (lane == mine) ok = sse <= limit;
        } else {
            const int second = todo ? __ffs(todo) - 1 : -1, i = half && second >= 0 ? second : mine;
            todo &= todo - 1;
            const bool on = !half || second >= 0;
            const int Mx = __shfl_sync(all, v.Mx, i), My = __shfl_sync(all, v.My, i), si = __shfl_sync(all, s, i), bi = __shfl_sync(all, b, i);
            uint32_t sse = row_sse(a, si, bi, Mx, My, r, on);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) sse += __shfl_xor_sync(all, sse, o);
            const uint32_t other = __shfl_xor_sync(all, sse, 16);                // every lane knows both halves' sums
            if (lane == mine) ok = (half ? other : sse) <= limit;
            if (lane == second) ok = (half ? sse : other) <= limit;
        }
    }
    if (in_grid) a.matched[gi] = (uint8_t)ok;
    // matched count: one atomic per warp and stream
    const unsigned same = __match_any_sync(all, s), oks = __ballot_sync(all, in_grid && ok);
    if (lane == __ffs(same) - 1 && (oks & same)) atomicAdd(&a.acc[4 * s + 3], __popc(oks & same));
}

// Step 5: maximal horizontal runs of matched blocks per block row; a run continues the rectangle above it only when the
// run directly above starts and ends at the same columns; every other run heads a rectangle that extends down while
// that holds.  One CTA per stream; heads are emitted in (y, x) order by a CTA-wide ordered compaction.
// In per-block mode (mv != nullptr) neighbours of a run, the run above and the runs below must also carry the same
// vector, and the rectangle's source is displaced by that vector instead of the global one.
struct MergeArgs {
    const uint8_t* matched; const int16_t* mv; const int32_t* gmv;
    int W, H, B, Gx, Gy, max_regions;
    uint16_t* run_end;
    dc_region* regions; int32_t* n_regions; int32_t* status;
    int32_t* gmv_out; int32_t* n_out; dc_region* regions_out;                            // the caller's, or null
};
__device__ __forceinline__ void emit_region(const MergeArgs& a, int s, int idx, int r, int c0, int c1, int h, int Mx, int My)
{
    if (idx >= a.max_regions) { atomicExch(a.status, (int)DC_ERR_OVERFLOW); return; }
    const int x = c0 * a.B, y = r * a.B, x1 = min(c1 * a.B, a.W), y1 = min((r + h) * a.B, a.H);
    const dc_region g = { x, y, x1 - x, y1 - y, x + Mx, y + My };
    a.regions[(size_t)s * a.max_regions + idx] = g;
    if (a.regions_out) a.regions_out[(size_t)s * a.max_regions + idx] = g;
}
__device__ __forceinline__ void finish_merge(const MergeArgs& a, int s, int count)
{
    if (threadIdx.x == 0) {
        a.n_regions[s] = min(count, a.max_regions);
        if (a.n_out) a.n_out[s] = min(count, a.max_regions);
    }
    if (a.gmv_out && threadIdx.x < 3) a.gmv_out[3 * s + threadIdx.x] = a.gmv[3 * s + threadIdx.x];
}
// Exclusive sum of `mine` over the CTA's 1024 threads, and the total (sums: 32 words, free again after the next barrier).
__device__ __forceinline__ int block_exclusive(int mine, int* sums, int& total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, inc, o); inc += lane >= o ? t : 0; }
    if (lane == 31) sums[wid] = inc;
    __syncthreads();
    const int w = sums[lane];
    total = __reduce_add_sync(0xffffffffu, w);
    return __reduce_add_sync(0xffffffffu, lane < wid ? w : 0) + inc - mine;
}
// Length of the run of ones that starts at bit `from` of a row of `words` words (bits past the row are zero).
__device__ __forceinline__ int ones_from(const uint32_t* row, int words, int from)
{
    int w = from >> 5;
    if (w >= words) return 0;
    uint32_t zeros = ~row[w] & (0xffffffffu << (from & 31));
    while (zeros == 0) { if (++w == words) return words * 32 - from; zeros = ~row[w]; }
    return w * 32 + __ffs(zeros) - 1 - from;
}

// The blocks of a row are bits of words in shared memory, built by ballots: a run's end is a search for the first zero
// bit, and the passes over runs take a thread per word and visit set bits alone.  What bounds it: one SM per stream, so
// the instructions of its passes and the barriers between them.  Measured on 120 x 68 blocks, 8 streams: 31 us with a
// thread and its scans for every block, 19 us with bit strings but still a thread per block, 11.6 us so.
// Dynamic shared memory: merge_smem_bytes().
__host__ __device__ constexpr size_t merge_smem_bytes(int Gx, int Gy, bool own)
{
    const size_t n = (size_t)Gx * Gy, words = (size_t)(Gx + 31) / 32 * Gy;
    return n * (own ? 4 : 0) + 4 * words * 4 + n * 2;
}
__global__ void __launch_bounds__(1024) k_merge(const MergeArgs a)
{
    extern __shared__ __align__(16) uint32_t merge_smem[];
    __shared__ int sums[32];
    const int s = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, Gx = a.Gx, Gy = a.Gy, n = Gx * Gy;
    const int rw = (Gx + 31) >> 5, words = rw * Gy;
    uint32_t* starts = merge_smem + (a.mv ? n : 0);           // bit c of row r: a run starts here
    uint32_t* joined = starts + words;                        // the block continues its left neighbour's run; later: the run that starts here continues the one above
    uint32_t* heads = joined + words;                         // the run that starts here heads a rectangle
    uint32_t* first = heads + words;                          // rectangles before this word of heads
    uint16_t* e = (uint16_t*)(first + words);                 // end column of the run that starts here
    uint32_t* v = a.mv ? merge_smem : nullptr;                // (dx, dy) as one word
    dc_pdl_wait();
    dc_pdl_release();
    const int Mx = a.gmv[3 * s], My = a.gmv[3 * s + 1];
    const uint8_t* gm = a.matched + (size_t)s * n;
    const uint32_t* gv = (const uint32_t*)a.mv + (size_t)s * n;
    for (int r = wid; r < Gy; r += 32) {
        uint32_t left_on = 0, left_v = 0;                     // last block of the word before
        for (int w0 = 0; w0 < rw; w0 += 4) {
            uint32_t on[4], u[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {                     // four words' loads in flight
                const int c = (w0 + k) * 32 + lane;
                on[k] = c < Gx ? gm[r * Gx + c] : 0;
                u[k] = v && c < Gx ? gv[r * Gx + c] : 0;
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int c = (w0 + k) * 32 + lane;
                if (w0 + k >= rw) break;
                const uint32_t word = __ballot_sync(0xffffffffu, on[k] != 0);
                uint32_t join = word & ((word << 1) | left_on);
                left_on = word >> 31;
                if (v) {
                    uint32_t pv = __shfl_up_sync(0xffffffffu, u[k], 1);
                    if (lane == 0) pv = left_v;
                    join &= __ballot_sync(0xffffffffu, pv == u[k]);
                    left_v = __shfl_sync(0xffffffffu, u[k], 31);
                    if (c < Gx) v[r * Gx + c] = u[k];
                }
                if (lane == 0) { joined[r * rw + w0 + k] = join; starts[r * rw + w0 + k] = word & ~join; }
            }
        }
    }
    __syncthreads();
    for (int t = tid; t < words; t += 1024) {
        const int r = t / rw, w = t - r * rw;
        for (uint32_t left = starts[t]; left; left &= left - 1) {
            const int c = w * 32 + __ffs(left) - 1;
            e[r * Gx + c] = (uint16_t)(c + 1 + ones_from(joined + r * rw, rw, c + 1));
        }
    }
    __syncthreads();
    int mine = 0, total;
    for (int t = tid; t < words; t += 1024) {
        const int r = t / rw, w = t - r * rw;
        const uint32_t here = starts[t];
        uint32_t down = 0;
        for (uint32_t left = r > 0 ? here & starts[t - rw] : 0; left; left &= left - 1) {
            const int b = r * Gx + w * 32 + __ffs(left) - 1;
            if (e[b - Gx] == e[b] && (!v || v[b - Gx] == v[b])) down |= left & (0u - left);
        }
        joined[t] = down;
        heads[t] = here & ~down;
    }
    __syncthreads();
    const int per = (words + 1023) / 1024, lo = min(tid * per, words), hi = min(lo + per, words);
    for (int t = lo; t < hi; ++t) mine += __popc(heads[t]);
    int before = block_exclusive(mine, sums, total);
    for (int t = lo; t < hi; ++t) { first[t] = (uint32_t)before; before += __popc(heads[t]); }
    __syncthreads();
    for (int r = wid; r < Gy; r += 32)
        for (int w = 0; w < rw; ++w) {
            const int t = r * rw + w;
            const uint32_t word = heads[t];
            if (!((word >> lane) & 1u)) continue;
            int h = 1;
            while (r + h < Gy && ((joined[t + h * rw] >> lane) & 1u)) ++h;
            const int c = w * 32 + lane, b = r * Gx + c;
            const uint32_t own = v ? v[b] : 0u;
            emit_region(a, s, (int)first[t] + __popc(word & ((1u << lane) - 1u)), r, c, e[b], h,
                        v ? (int16_t)(own & 0xffffu) : Mx, v ? (int16_t)(own >> 16) : My);
        }
    finish_merge(a, s, total);
}

// The same for block grids beyond shared memory: block by block, the runs in global memory.
__global__ void __launch_bounds__(1024) k_merge_large(const MergeArgs a)
{
    __shared__ int sums[32];
    const int s = blockIdx.x, tid = threadIdx.x, Gx = a.Gx, Gy = a.Gy, n = Gx * Gy;
    dc_pdl_wait();
    dc_pdl_release();
    const uint8_t* m = a.matched + (size_t)s * n;
    const uint32_t* v = a.mv ? (const uint32_t*)a.mv + (size_t)s * n : nullptr;          // (dx, dy) as one word
    uint16_t* e = a.run_end + (size_t)s * n;
    for (int b = tid; b < n; b += 1024) {
        const int c = b % Gx;
        int end = 0;
        if (m[b] && (c == 0 || !m[b - 1] || (v && v[b - 1] != v[b]))) {
            end = c + 1;
            const uint8_t* row = m + (b - c);
            while (end < Gx && row[end] && (!v || v[b - c + end] == v[b])) ++end;
        }
        e[b] = (uint16_t)end;
    }
    __syncthreads();
    int Mx = a.gmv[3 * s], My = a.gmv[3 * s + 1];
    int base = 0;                                                     // rectangles emitted so far, the same in all threads
    for (int start = 0; start < n; start += 1024) {
        const int b = start + tid;
        int head = 0, c1 = 0, h = 0, r = 0, c0 = 0, total;
        if (b < n) {
            r = b / Gx; c0 = b - r * Gx;
            c1 = e[b];
            if (c1 != 0 && !(r > 0 && e[b - Gx] == c1 && (!v || v[b - Gx] == v[b]))) {
                head = 1; h = 1;
                while (r + h < Gy && e[b + h * Gx] == c1 && (!v || v[b + h * Gx] == v[b])) ++h;
            }
        }
        const int idx = base + block_exclusive(head, sums, total);
        if (head) {
            if (v) { const uint32_t own = v[b]; Mx = (int16_t)(own & 0xffffu); My = (int16_t)(own >> 16); }
            emit_region(a, s, idx, r, c0, c1, h, Mx, My);
        }
        base += total;
        __syncthreads();                                              // sums is free again
    }
    finish_merge(a, s, base);
}

// ---------------------------------------------------------------------------------------------
// Fast Steps 2 and 4: 16-pixel blocks, diamond search
// ---------------------------------------------------------------------------------------------

__device__ __forceinline__ void publish_block(const MatchArgs& a, int s, size_t g, int bw, int bh, unsigned long long bk)
{
    const int fx = (int)(bk & 0xff) - 128, fy = (int)((bk >> 8) & 0xff) - 128;
    const uint32_t fs = (uint32_t)(bk >> 32);
    a.mv[2 * g] = (int16_t)fx; a.mv[2 * g + 1] = (int16_t)fy; a.sse[g] = fs;
    if (fs <= a.limit[limit_index(a, bw, bh)]) {              // PSNR > T: member of Step 3's set S
        atomicAdd(&a.acc[4 * s + 0], fx);
        atomicAdd(&a.acc[4 * s + 1], fy);
        atomicAdd(&a.acc[4 * s + 2], 1);
    }
}

// ---------------------------------------------------------------------------------------------
// Step 2 for 16-pixel blocks, diamond search: one warp per block
// ---------------------------------------------------------------------------------------------
// The previous frame's window is staged in shared memory with one 32-bit word per pixel (R, G, B, 0), so a candidate
// displaced by (dx, dy) starts at a word whatever dx is: no byte realignment, and a candidate's address is the lane's
// base plus dy * pitch + dx.  Lane 2 r + h scores pixels h, h + 2, ..., h + 14 of block row r: its 8 pixels of the
// current block stay in registers, a candidate costs 8 loads at fixed offsets, 8 absolute differences, 8 multiply-
// accumulates and one warp sum.  With a row pitch of p words, p = 2 (mod 4), the 32 lanes of a load fall in 32
// different banks for every displacement (bank = r p + h + const, and r p / 2 runs through all residues mod 16),
// so shared memory is read without conflicts, and all lanes of a warp follow the same walk, so no lane waits for
// another block.  The points of the two diamonds sit at compile-time offsets from the centre's address.
// displacements that keep the block inside the previous frame and the search range
struct WalkBounds { int dx_lo, dx_hi, dy_lo, dy_hi; };

__device__ __forceinline__ WalkBounds walk_bounds(const MatchArgs& a, int x0, int y0, int bw, int bh)
{
    WalkBounds b = {max(-a.R, -x0), min(a.R, a.W - bw - x0), max(-a.R, -y0), min(a.R, a.H - bh - y0)};
    return b;
}
// The 8 pixels of row r (48 bytes at `row`, 16-byte aligned) that lane parity h scores, one word each.  copy (or NULL): where the row goes.
__device__ __forceinline__ void load_lane_pixels(const uint8_t* row, int h, bool on, uint32_t (&cw)[8], uint8_t* copy = nullptr)
{
    uint32_t w[12];
    const uint4* p = (const uint4*)row;
    uint4 v0 = make_uint4(0, 0, 0, 0), v1 = v0, v2 = v0;
    if (on) { v0 = dc_ld(p); v1 = dc_ld(p + 1); v2 = dc_ld(p + 2); }
    if (copy && on && h == 0) { uint4* o = (uint4*)copy; o[0] = v0; o[1] = v1; o[2] = v2; }
    w[0] = v0.x; w[1] = v0.y; w[2] = v0.z; w[3] = v0.w; w[4] = v1.x; w[5] = v1.y; w[6] = v1.z; w[7] = v1.w;
    w[8] = v2.x; w[9] = v2.y; w[10] = v2.z; w[11] = v2.w;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        uint32_t px[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = 2 * j + q, wi = (3 * k) >> 2, sh = ((3 * k) & 3) * 8;      // pixel k: bytes 3k .. 3k + 2
            px[q] = (sh == 0 ? w[wi] : sh == 8 ? w[wi] >> 8 : __funnelshift_r(w[wi], w[wi + 1 < 12 ? wi + 1 : wi], sh)) & 0x00ffffffu;
        }
        cw[j] = h ? px[1] : px[0];
    }
}

// Expands 4 packed pixels (12 bytes in a, b, c) to 4 words and stores them at dst (8-byte aligned).
__device__ __forceinline__ void store_pixels4(uint32_t* dst, uint32_t a, uint32_t b, uint32_t c)
{
    const uint32_t m = 0x00ffffffu;
    *(uint2*)dst = make_uint2(a & m, __funnelshift_r(a, b, 24) & m);
    *(uint2*)(dst + 2) = make_uint2(__funnelshift_r(b, c, 16) & m, c >> 8);
}
// 4 pixels starting at pixel px0 (a multiple of 4) of frame row gy, zeros outside the frame copy
__device__ __forceinline__ void load_pixels4(const uint8_t* prev, size_t pitch, int H, int gy, int px0, uint32_t& a, uint32_t& b, uint32_t& c)
{
    a = b = c = 0;
    if (gy >= 0 && gy < H && px0 >= 0 && (size_t)px0 * 3 + 12 <= pitch) {
        const uint32_t* q = (const uint32_t*)(prev + (size_t)gy * pitch + (size_t)px0 * 3);     // px0 * 3 is a multiple of 12
        a = dc_ld(q); b = dc_ld(q + 1); c = dc_ld(q + 2);
    }
}

// Candidates of one window row, at compile-time displacements LO + 2 m for the set bits m of DXS: they are shifted by whole words against
// one another, so a word is loaded once for all of them.  p: the address of displacement 0 in that row; n_px: how many of the lane's pixels
// lie inside the frame.  sum(m, value) takes the scores.
__host__ __device__ constexpr int high_bit(unsigned long long m) { int n = -1; for (; m; m >>= 1) ++n; return n; }
__host__ __device__ constexpr int bits_of(unsigned long long m) { int n = 0; for (; m; m &= m - 1) ++n; return n; }
template <int LO, unsigned long long DXS>
struct RowWords {
    static constexpr int N = 8 + high_bit(DXS);
    uint32_t w[N];
    template <int K = 0>
    __device__ __forceinline__ void load(uint32_t p)
    {
        if constexpr (K < N) {
            if constexpr (((DXS << 7) >> K & 0xffull) != 0) w[K] = lds_at<(LO + 2 * K) * 4>(p);         // some m with 0 <= K - m < 8
            load<K + 1>(p);
        }
    }
    template <bool CLIP, typename Sum>
    __device__ __forceinline__ void score(const uint32_t (&cw)[8], bool row_on, int n_px, const Sum& sum) const
    {
        constexpr int C = bits_of(DXS);
        uint32_t acc[C];
#pragma unroll
        for (int c = 0; c < C; ++c) acc[c] = 0;
#pragma unroll
        for (int k = 0; k < N; ++k) {
            int c = 0;
#pragma unroll
            for (int m = 0; m <= high_bit(DXS); ++m)
                if (DXS >> m & 1) {
                    if (k - m >= 0 && k - m < 8) {
                        const uint32_t d = !CLIP || k - m < n_px ? __vabsdiffu4(cw[(k - m) & 7], w[k]) : 0u;
                        acc[c] = __dp4a(d, d, acc[c]);
                    }
                    ++c;
                }
        }
        int c = 0;
#pragma unroll
        for (int m = 0; m <= high_bit(DXS); ++m)
            if (DXS >> m & 1) { sum(m, __reduce_add_sync(0xffffffffu, row_on ? acc[c] : 0u)); ++c; }
    }
};

// The points of the compile-time set MASK around the centre whose candidate starts at pc, row by row: straight-line code, every load at a
// fixed offset.  Lane i keeps the score of point i.  AHEAD: the words of all rows are on their way before the first is used.
__host__ __device__ constexpr int point_at(uint32_t mask, int x, int y)
{
    for (int i = 0; i < 13; ++i) if ((mask >> i & 1) && point_x(i) == x && point_y(i) == y) return i;
    return -1;
}
__host__ __device__ constexpr int row_lo(uint32_t mask, int y)                     // smallest x of the row's points, 3: none
{
    for (int x = -2; x <= 2; ++x) if (point_at(mask, x, y) >= 0) return x;
    return 3;
}
__host__ __device__ constexpr unsigned long long row_dxs(uint32_t mask, int y)
{
    unsigned long long b = 0;
    for (int m = 0; row_lo(mask, y) + 2 * m <= 2; ++m) if (point_at(mask, row_lo(mask, y) + 2 * m, y) >= 0) b |= 1ull << m;
    return b;
}
template <uint32_t MASK, int PITCH, bool AHEAD, int Y = -2>
__device__ __forceinline__ void score_set(uint32_t pc, const uint32_t (&cw)[8], bool row_on, int lane, uint32_t& mine)
{
    if constexpr (Y <= 2) {
        if constexpr (row_lo(MASK, Y) <= 2) {
            constexpr int LO = row_lo(MASK, Y);
            RowWords<LO + Y * PITCH, row_dxs(MASK, Y)> row;
            row.load(pc);
            if constexpr (AHEAD) score_set<MASK, PITCH, AHEAD, Y + 1>(pc, cw, row_on, lane, mine);
            row.template score<false>(cw, row_on, 8, [&](int m, uint32_t v) { mine = lane == point_at(MASK, LO + 2 * m, Y) ? v : mine; });
            if constexpr (!AHEAD) score_set<MASK, PITCH, AHEAD, Y + 1>(pc, cw, row_on, lane, mine);
        } else {
            score_set<MASK, PITCH, AHEAD, Y + 1>(pc, cw, row_on, lane, mine);
        }
    }
}

// One block's walk, by one warp, for as long as it stays inside the staged window.
//
// Outside the first round the centre is the best point so far and bs its SSE.  Every point around the centre is staged, so a round runs as
// straight-line code for its set whatever the frame's edge and the range allow; lane i then drops point i where it is no valid candidate, and
// the smallest score wins, or the smallest (|dx| + |dy|, dy, dx) among equal ones.  (With a path for cut sets and ties, point by point, the
// walks at the edges set the time of a small frame.)
__device__ __forceinline__ Within walk_range(const WalkBounds& b) { return Within{disp(b.dx_lo, b.dy_lo), disp(b.dx_hi, b.dy_hi)}; }

struct WalkW {
    int at, kind;               // centre, and how it was reached
    uint32_t bs;                // SSE of the best point so far (the centre, after the first round)
    int left;                   // moves left; every one strictly lowers the key, so (2 R + 1)^2 are never used up
    int next, nk; uint32_t ns;  // on return 2: the centre the walk has chosen and not yet moved to, the kind of that move, and its SSE
};

// Blocks that the frame's right edge cuts: the points of a set three at a time; n_px: how many of the lane's eight pixels lie inside.
template <int PITCH>
__device__ __forceinline__ void score_clipped(uint32_t set, uint32_t pc, uint32_t off, const uint32_t (&cw)[8], bool row_on, int n_px, int lane, uint32_t& mine)
{
#pragma unroll 1
    while (set) {                                                 // the same in all lanes
        uint32_t p[3], acc[3] = {0, 0, 0}; int at[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            at[k] = set ? __ffs(set) - 1 : -1;                    // none left: the centre once more, kept by no lane
            p[k] = pc + __shfl_sync(0xffffffffu, off, set ? at[k] : 8);
            set &= set - 1;
        }
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const uint32_t w = lds_at<0>(p[k] + 8u * j), d = j < n_px ? __vabsdiffu4(cw[j], w) : 0u;
                acc[k] = __dp4a(d, d, acc[k]);
            }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const uint32_t sum = __reduce_add_sync(0xffffffffu, row_on ? acc[k] : 0u);
            mine = lane == at[k] ? sum : mine;
        }
    }
}

// Shared-memory bytes from a candidate to the one displaced by a pair.
template <int PITCH>
__device__ __forceinline__ uint32_t bytes_of(int p)
{
    const int y = (p + 0x8000) >> 16;
    return (uint32_t)(4 * p + y * (4 * PITCH - 4 * 65536));
}

//   lane_base  shared-memory address of this lane's first word of the candidate at displacement (0, 0);
//              (dx, dy) is at lane_base + (dy * PITCH + dx) * 4
//   valid  displacements that keep the block inside the previous frame and the search range
//   reach  centres around which every point is staged
//   AHEAD  the loads of a whole round travel together
// Returns 1 when the walk has finished (result: w.at, w.bs), 2 when the next centre is out of reach.
template <int PITCH, bool AHEAD>
__device__ __forceinline__ int warp_walk(const MatchArgs& a, uint32_t lane_base, const uint32_t (&cw)[8], bool row_on, int n_px, bool clipped,
                                         Within valid, WalkW& w, Within reach)
{
    const unsigned all = 0xffffffffu;
    const int lane = threadIdx.x & 31, point = lane_point(lane);
    uint32_t pc = lane_base + bytes_of<PITCH>(w.at - disp(0, 0));
#pragma unroll 1
    for (;; --w.left) {
        uint32_t mine = 0xffffffffu;
        if (!clipped) {
            switch (w.kind) {
            case 0: score_set<kind_mask(0), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 1: score_set<kind_mask(1), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 2: score_set<kind_mask(2), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 3: score_set<kind_mask(3), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 4: score_set<kind_mask(4), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 5: score_set<kind_mask(5), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 6: score_set<kind_mask(6), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case 7: score_set<kind_mask(7), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            case KIND_FIRST: score_set<kind_mask(KIND_FIRST), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            default: score_set<kind_mask(KIND_SMALL), PITCH, AHEAD>(pc, cw, row_on, lane, mine); break;
            }
        } else {
            score_clipped<PITCH>(c_kind_mask[w.kind], pc, bytes_of<PITCH>(point), cw, row_on, n_px, lane, mine);
        }
        if (lane == 8 && w.kind != KIND_FIRST) mine = w.bs;       // the centre
        const int d = w.at + point;
        if (!within(d, valid)) mine = 0xffffffffu;
        uint32_t ns;
        const int g = best_lane(mine, d, ns);                     // the best point after this round
        const int next = __shfl_sync(all, d, g);
        if (w.kind == KIND_SMALL) { w.at = next; w.bs = ns; return 1; }                // the small diamond's best is the result
        if (g == 8) { w.bs = ns; w.kind = KIND_SMALL; continue; }                      // centre won: small diamond, then done
        if (w.left <= 0) {                                        // a walk cut here is not valid: say so
            if (lane == 0) atomicExch(a.status, (int)DC_ERR_TIMEOUT);
            w.bs = ns;
            return 1;
        }
        if (!within(next, reach)) { w.next = next; w.nk = g; w.ns = ns; --w.left; return 2; }
        pc += bytes_of<PITCH>(next - w.at);
        w.kind = g; w.at = next; w.bs = ns;
    }
}
// how many of a lane's pixels h, h + 2, ... of a block row of bw pixels exist
__device__ __forceinline__ int lane_pixel_count(int bw, int h) { return (bw - h + 1) >> 1; }

// Phase 1: one CTA per 8 x W_VS blocks, one warp per block.  The window reaches W_WRY rows above and below the tile
// and 12 pixels to its left and right (its left edge stays a multiple of 4 pixels, so that 4 pixels are 12 aligned
// bytes of the packed frame).  A walk whose next centre is out of reach is handed to phase 2.  Launched without k-skip
// only (every block is searched).
// What bounds it: instruction issue (3.3 of 4 per clock and SM on 8 full-HD streams, 105 us; 126 while cut point sets and ties had a path
// of their own), or, with few tiles, the longest walk: a round is a trip to shared memory and back.  Up to two tiles per SM the instance
// with AHEAD runs, which has the loads of a whole round in flight (64 registers a thread): one stream of 227 x 227, 8.7 -> 5.5 us, with noise
// in it and the walks of phase 2 28 -> 17.  (A whole pass, us, without and with it: VGG, two 640 x 360 streams 218 and 210; AlexNet, 18
// streams, 142 and 140.)
constexpr int W_VS = 2, W_WRY = 10, W_SIDE = 12;
constexpr int W_COLS = 128 + 2 * W_SIDE;                    // staged pixels per window row
constexpr int W_PITCH = 154;                                // words per window row
constexpr int W_ROWS = 16 * W_VS + 2 * W_WRY;
static_assert(W_PITCH % 4 == 2 && W_PITCH >= W_COLS && W_COLS % 4 == 0, "conflict-free pitch, whole groups of 4 pixels");

template <bool AHEAD>
__global__ void __launch_bounds__(W_VS * 8 * 32, AHEAD ? 2 : 3) k_search_dsw(MatchArgs a, uint4* long_list, int32_t* long_count)
{
    dc_pdl_wait();
    dc_pdl_release();
    constexpr int THREADS = W_VS * 8 * 32, GROUPS = W_COLS / 4;
    constexpr int ROWS_PER_PASS = THREADS / GROUPS, PASSES = (W_ROWS + ROWS_PER_PASS - 1) / ROWS_PER_PASS;
    __shared__ __align__(16) uint32_t win[W_ROWS * W_PITCH];
    __shared__ int32_t sums[3];
    const int strip = blockIdx.x, vg = blockIdx.y, s = blockIdx.z;        // grid: strips of 8 blocks x groups of W_VS block rows x streams
    const int xs = strip * 128, yb = vg * 16 * W_VS;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31, r = lane >> 1, h = lane & 1;
    const int by = vg * W_VS + (warp >> 3), bx = strip * 8 + (warp & 7);
    const int x0 = bx * 16, y0 = by * 16;
    const bool searched = bx < a.Gx && by < a.Gy;
    const int bh = searched ? min(16, a.H - y0) : 0, bw = min(16, a.W - x0);
    const bool row_on = r < bh;
    uint32_t cw[8];                                            // issued first: in flight while the window is staged
    {
        const int row = row_on ? y0 + r : 0, at = (row_on ? x0 : 0) * 3;
        load_lane_pixels(a.cur + (size_t)s * a.cur_stream + (size_t)row * a.cur_pitch + at, h, row_on, cw,
                         a.copy ? a.copy + (size_t)s * a.copy_stream + (size_t)row * a.copy_pitch + at : nullptr);
    }
    if (threadIdx.x < 3) sums[threadIdx.x] = 0;
    {   // the window: a thread keeps its group of 4 pixels (one column position) and goes down the rows, 13 rows apart
        const int gq = threadIdx.x % GROUPS, row0 = threadIdx.x / GROUPS, px0 = xs - W_SIDE + 4 * gq;
        const bool col_ok = row0 < ROWS_PER_PASS && px0 >= 0 && (size_t)px0 * 3 + 12 <= a.prev_pitch;
        const uint8_t* src = a.prev + (size_t)s * a.prev_stream + (size_t)px0 * 3;       // px0 * 3 is a multiple of 12
        uint32_t* dst = win + row0 * W_PITCH + 4 * gq;
        uint32_t pa[PASSES], pb[PASSES], pc[PASSES];
#pragma unroll
        for (int k = 0; k < PASSES; ++k) {                         // all loads first
            const int row = row0 + k * ROWS_PER_PASS, gy = yb - W_WRY + row;
            pa[k] = pb[k] = pc[k] = 0;
            if (col_ok && row < W_ROWS && gy >= 0 && gy < a.H) {
                const uint32_t* q = (const uint32_t*)(src + (size_t)gy * a.prev_pitch);
                pa[k] = dc_ld(q); pb[k] = dc_ld(q + 1); pc[k] = dc_ld(q + 2);
            }
        }
        if (row0 < ROWS_PER_PASS) {
#pragma unroll
            for (int k = 0; k < PASSES; ++k)
                if (row0 + k * ROWS_PER_PASS < W_ROWS) store_pixels4(dst + k * ROWS_PER_PASS * W_PITCH, pa[k], pb[k], pc[k]);
        }
    }
    __syncthreads();
    const size_t g = (size_t)s * a.Gx * a.Gy + (size_t)by * a.Gx + bx;
    if (searched) {
        const WalkBounds wb = walk_bounds(a, x0, y0, bw, bh);
        const uint32_t lane_base = (uint32_t)__cvta_generic_to_shared(win) +
                                   (uint32_t)((((warp >> 3) * 16 + r + W_WRY) * W_PITCH + (x0 - xs + W_SIDE) + h) * 4);
        WalkW w = {disp(0, 0), KIND_FIRST, 0xffffffffu, (2 * a.R + 1) * (2 * a.R + 1), 0, 0, 0u};
        const Within reach = {disp(2 - W_SIDE, 2 - W_WRY), disp(W_SIDE - 2, W_WRY - 2)};
        const int st = warp_walk<W_PITCH, AHEAD>(a, lane_base, cw, row_on, lane_pixel_count(bw, h), bw < 16, walk_range(wb), w, reach);
        if (lane == 0) {
            if (st == 1) {
                const int dx = disp_x(w.at), dy = disp_y(w.at);
                a.mv[2 * g] = (int16_t)dx; a.mv[2 * g + 1] = (int16_t)dy; a.sse[g] = w.bs;
                if (w.bs <= a.limit[limit_index(a, bw, bh)]) {        // PSNR > T: member of Step 3's set S
                    atomicAdd(&sums[0], dx); atomicAdd(&sums[1], dy); atomicAdd(&sums[2], 1);
                }
            } else {                                                  // block, chosen next centre, its SSE, the kind of that move
                const int slot = atomicAdd(long_count, 1);
                long_list[slot] = make_uint4((uint32_t)g, (uint32_t)w.next, w.ns, (uint32_t)w.nk);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sums[2]) {                                // Step 3's sums once per CTA (one stream per CTA)
        atomicAdd(&a.acc[4 * s + 0], sums[0]);
        atomicAdd(&a.acc[4 * s + 1], sums[1]);
        atomicAdd(&a.acc[4 * s + 2], sums[2]);
    }
}

// ---------------------------------------------------------------------------------------------
// Step 2 for 16-pixel blocks, three step search (Section 7.5): one warp per block
// ---------------------------------------------------------------------------------------------
// Layout of the diamond kernel: one word per pixel, lane 2 r + h scores every other pixel of block row r, no bank
// conflicts.  The window reaches `side` pixels (2 S0 - 1, rounded up to four) to the left and right and wr = 2 S0 - 1
// rows up and down, so every point of the search is staged.  A step scores its eight points row by row and decides by SSE alone; when
// two of the scores that matter are equal the exact order (SSE, |dx| + |dy|, dy, dx) picks from the same scores.
// What bounds it: issue slots - 8 differences, 8 multiply-adds and a warp sum per point and block, and the loads, which the points of a
// row share where the step is 8 or less.  Measured on 8 full-HD frames, range 16: 140 us with 4 lanes per block and byte-aligned rows (a
// bank conflict and a realignment per word), 126 with 8 loads per point and two CTAs per SM, 114 so.  AHEAD (up to two tiles per SM):
// the loads of a step travel together; two 640 x 360 streams 9.9 -> 5.8 us, eight of 300 x 200 (1.1 tiles per SM) 8.4 -> 7.7, and 11.6
// without it and with the points of blocks that the right edge cuts one by one.
constexpr int TSS_VS = 2;
struct TssShape { int s0, wr, side, pitch; };
static TssShape tss_shape(int R)
{
    TssShape t;
    t.s0 = R < 1 ? 0 : 1;                                       // first step: the largest power of two with 2 S0 - 1 <= R
    while (t.s0 > 0 && 4 * t.s0 - 1 <= R) t.s0 *= 2;
    t.wr = t.s0 > 0 ? 2 * t.s0 - 1 : 0;
    t.side = (t.wr + 3) & ~3;
    t.pitch = 128 + 2 * t.side + 2;                             // 2 modulo 4: conflict-free
    return t;
}
static size_t tss_window_bytes(const TssShape& t) { return (size_t)(16 * TSS_VS + 2 * t.wr) * t.pitch * sizeof(uint32_t); }

// The eight points of a step of compile-time length, row by row (the middle of the centre's row is the best point so far).  CLIP: blocks that
// the frame's right edge cuts; n_px: how many of the lane's eight pixels lie inside.
template <int STEP, bool CLIP, bool AHEAD, int Y = -1>
__device__ __forceinline__ void tss_score(uint32_t pc, uint32_t row_bytes, const uint32_t (&cw)[8], bool row_on, int n_px, int lane, uint32_t& mine)
{
    if constexpr (Y <= 1) {
        const uint32_t p = pc + (uint32_t)Y * row_bytes;
        constexpr int G = 3 * (Y + 1);
        if constexpr (STEP == 1) {                                // an odd step: its sides are no whole words from its middle
            RowWords<-1, 3ull> sides;
            RowWords<0, 1ull> middle;
            sides.load(p);
            if constexpr (Y != 0) middle.load(p);
            if constexpr (AHEAD) tss_score<STEP, CLIP, AHEAD, Y + 1>(pc, row_bytes, cw, row_on, n_px, lane, mine);
            sides.template score<CLIP>(cw, row_on, n_px, [&](int m, uint32_t v) { mine = lane == G + 2 * m ? v : mine; });
            if constexpr (Y != 0) middle.template score<CLIP>(cw, row_on, n_px, [&](int m, uint32_t v) { mine = lane == G + 1 ? v : mine; });
        } else {
            constexpr unsigned long long DXS = 1ull | (Y != 0 ? 1ull << (STEP / 2) : 0ull) | 1ull << STEP;
            RowWords<-STEP, DXS> row;
            row.load(p);
            if constexpr (AHEAD) tss_score<STEP, CLIP, AHEAD, Y + 1>(pc, row_bytes, cw, row_on, n_px, lane, mine);
            row.template score<CLIP>(cw, row_on, n_px, [&](int m, uint32_t v) { mine = lane == G + 2 * m / STEP ? v : mine; });
        }
        if constexpr (!AHEAD) tss_score<STEP, CLIP, AHEAD, Y + 1>(pc, row_bytes, cw, row_on, n_px, lane, mine);
    }
}

// Lane g < 9 settles point g of the 3 x 3 grid (4: its centre, the best so far): its displacement, validity and tie key
// are computed once per step and not point by point.
template <bool CLIP, bool AHEAD>
__device__ __forceinline__ void tss_walk(uint32_t lane_base, int pitch, int s0, const uint32_t (&cw)[8], bool row_on, int n_px,
                                         Within valid, int& at, uint32_t& bs)
{
    const int lane = threadIdx.x & 31, point = pair(lane % 3 - 1, lane / 3 - 1);
    {   // the zero vector
        RowWords<0, 1ull> zero;
        zero.load(lane_base);
        zero.template score<CLIP>(cw, row_on, n_px, [&](int, uint32_t v) { bs = v; });
    }
    at = disp(0, 0);
    uint32_t pc = lane_base;
#pragma unroll 1
    for (int step = s0; step > 0; step >>= 1) {
        const uint32_t row_bytes = (uint32_t)(step * pitch) * 4u;
        uint32_t mine = lane == 4 ? bs : 0xffffffffu;
        switch (step) {
        case 1: tss_score<1, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        case 2: tss_score<2, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        case 4: tss_score<4, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        case 8: tss_score<8, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        case 16: tss_score<16, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        default: tss_score<32, CLIP, AHEAD>(pc, row_bytes, cw, row_on, n_px, lane, mine); break;
        }
        const int d = at + step * point;
        if (!within(d, valid)) mine = 0xffffffffu;
        const int g = best_lane(mine, d, bs), my = g / 3 - 1, mx = g - 3 * (my + 1) - 1;
        at += step * pair(mx, my);
        pc += (uint32_t)((my * pitch + mx) * step * 4);
    }
}

template <bool AHEAD>
__global__ void __launch_bounds__(TSS_VS * 8 * 32, AHEAD ? 2 : 3) k_search_tss16(MatchArgs a, TssShape t)
{
    dc_pdl_wait();
    dc_pdl_release();
    extern __shared__ __align__(16) uint32_t tss_win[];
    __shared__ int32_t sums[3];
    constexpr int THREADS = TSS_VS * 8 * 32;
    const int strip = blockIdx.x, vg = blockIdx.y, s = blockIdx.z;
    const int xs = strip * 128, yb = vg * 16 * TSS_VS;
    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31, r = lane >> 1, h = lane & 1;
    const int by = vg * TSS_VS + (warp >> 3), bx = strip * 8 + (warp & 7);
    const int x0 = bx * 16, y0 = by * 16;
    const bool searched = bx < a.Gx && by < a.Gy;
    const int bh = searched ? min(16, a.H - y0) : 0, bw = min(16, a.W - x0);
    const bool row_on = r < bh;
    uint32_t cw[8];                                            // issued first: in flight while the window is staged
    {
        const int row = row_on ? y0 + r : 0, at = (row_on ? x0 : 0) * 3;
        load_lane_pixels(a.cur + (size_t)s * a.cur_stream + (size_t)row * a.cur_pitch + at, h, row_on, cw,
                         a.copy ? a.copy + (size_t)s * a.copy_stream + (size_t)row * a.copy_pitch + at : nullptr);
    }
    if (threadIdx.x < 3) sums[threadIdx.x] = 0;
    const uint8_t* prev = a.prev + (size_t)s * a.prev_stream;
    // groups of 4 pixels, five in flight per thread; a thread's next group is THREADS further: rows and columns by addition
    const int groups = (128 + 2 * t.side) / 4, rows = 16 * TSS_VS + 2 * t.wr, row_add = THREADS / groups, col_add = THREADS - row_add * groups;
    constexpr int UNR = AHEAD ? 5 : 3;
    for (int row = threadIdx.x / groups, gq = threadIdx.x - row * groups; row < rows;) {
        uint32_t pa[UNR], pb[UNR], pc[UNR];
        uint32_t* dst[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u) {
            load_pixels4(prev, a.prev_pitch, a.H, yb - t.wr + row, xs - t.side + 4 * gq, pa[u], pb[u], pc[u]);
            dst[u] = row < rows ? tss_win + row * t.pitch + 4 * gq : nullptr;
            row += row_add; gq += col_add;
            if (gq >= groups) { gq -= groups; ++row; }
        }
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (dst[u]) store_pixels4(dst[u], pa[u], pb[u], pc[u]);
    }
    __syncthreads();
    if (searched) {
        const size_t g = (size_t)s * a.Gx * a.Gy + (size_t)by * a.Gx + bx;
        const WalkBounds wb = walk_bounds(a, x0, y0, bw, bh);
        const uint32_t lane_base = (uint32_t)__cvta_generic_to_shared(tss_win) +
                                   (uint32_t)((((warp >> 3) * 16 + r + t.wr) * t.pitch + (x0 - xs + t.side) + h) * 4);
        int at; uint32_t bs;
        if (bw == 16) tss_walk<false, AHEAD>(lane_base, t.pitch, t.s0, cw, row_on, 8, walk_range(wb), at, bs);
        else tss_walk<true, AHEAD>(lane_base, t.pitch, t.s0, cw, row_on, lane_pixel_count(bw, h), walk_range(wb), at, bs);
        const int cx = disp_x(at), cy = disp_y(at);
        if (lane == 0) {
            a.mv[2 * g] = (int16_t)cx; a.mv[2 * g + 1] = (int16_t)cy; a.sse[g] = bs;
            if (bs <= a.limit[limit_index(a, bw, bh)]) {          // PSNR > T: member of Step 3's set S
                atomicAdd(&sums[0], cx); atomicAdd(&sums[1], cy); atomicAdd(&sums[2], 1);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && sums[2]) {                            // Step 3's sums once per CTA (one stream per CTA)
        atomicAdd(&a.acc[4 * s + 0], sums[0]);
        atomicAdd(&a.acc[4 * s + 1], sums[1]);
        atomicAdd(&a.acc[4 * s + 2], sums[2]);
    }
}

// Section 4, k-skip: blocks that are not searched report vector (0, 0) and SSE 2^32 - 1.  One thread per block.
__global__ void k_mark_unsearched(MatchArgs a)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int gi = blockIdx.x * blockDim.x + threadIdx.x;
    if (gi >= a.S * a.Gx * a.Gy) return;
    const int b = gi % (a.Gx * a.Gy), by = b / a.Gx, bx = b - by * a.Gx;
    if (bx % a.skip_k != 0 || by % a.skip_k != 0) { a.mv[2 * gi] = 0; a.mv[2 * gi + 1] = 0; a.sse[gi] = 0xffffffffu; }
}

// Phase 2: the walks that left their tile's window.  A warp takes walks off the list one after the other (atomic
// cursor); the walk gets a private window of P_ROWS x P_COLS pixels, re-staged whenever the next centre is out of reach, its middle two
// moves ahead of the centre in the walk's direction.  A continued walk makes exactly the move it had chosen (new points only),
// so the sequence of scored candidates is the uninterrupted walk's.
// With k-skip (Section 4) the searched blocks lie k blocks apart and share no window: there is no phase 1 then,
// and this kernel walks every searched block from its start (long_list == nullptr; item i is the
// i-th searched block in stream / row / column order).
constexpr int P_WARPS = 8;
constexpr int P_REACH = 8;                                  // staged pixels above and left of the block at the window's centre
constexpr int P_ROWS = 16 + 2 * P_REACH, P_COLS = 36, P_PITCH = 38;
// Four CTAs per SM: 8 full-HD streams 58 us, 74 with five, whose registers spill.
static_assert(P_PITCH % 4 == 2 && P_PITCH >= P_COLS && P_COLS % 4 == 0 && P_COLS >= 16 + 2 * P_REACH + 3, "window of a walk");

template <bool AHEAD>
__global__ void __launch_bounds__(P_WARPS * 32, AHEAD ? 2 : 4) k_search_dsw_long(MatchArgs a, const uint4* long_list, const int32_t* long_count, int32_t* cursor)
{
    dc_pdl_wait();
    dc_pdl_release();
    __shared__ __align__(16) uint32_t win_all[P_WARPS][P_ROWS * P_PITCH];
    const int lane = threadIdx.x & 31, r = lane >> 1, h = lane & 1;
    uint32_t* win = win_all[threadIdx.x >> 5];
    const int per = a.Gx * a.Gy;
    const bool direct = long_list == nullptr;
    const int sgx = (a.Gx + a.skip_k - 1) / a.skip_k, sgy = (a.Gy + a.skip_k - 1) / a.skip_k;       // searched columns, rows
    const int n = direct ? a.S * sgx * sgy : *long_count;
#pragma unroll 1
    for (;;) {
        int idx = 0;
        if (lane == 0) idx = atomicAdd(cursor, 1);
        idx = __shfl_sync(0xffffffffu, idx, 0);
        if (idx >= n) break;
        unsigned g;                                               // S * Gx * Gy < 2^31
        WalkW w = {disp(0, 0), KIND_FIRST, 0xffffffffu, (2 * a.R + 1) * (2 * a.R + 1), 0, 0, 0u};
        if (direct) {
            const int ss = idx / (sgx * sgy), q = idx - ss * sgx * sgy, sby = q / sgx, sbx = q - sby * sgx;
            g = (unsigned)(ss * per + sby * a.skip_k * a.Gx + sbx * a.skip_k);
        } else {
            const uint4 e = long_list[idx];
            g = e.x; w.bs = e.z;
            w.at = (int)e.y;                                                                  // the move it had chosen: make it
            w.kind = (int)e.w;
        }
        const int s = (int)(g / (unsigned)per), b = (int)g - s * per, by = b / a.Gx, bx = b - by * a.Gx;
        const int x0 = bx * 16, y0 = by * 16, bh = min(16, a.H - y0), bw = min(16, a.W - x0);
        const bool row_on = r < bh;
        uint32_t cw[8];
        load_lane_pixels(a.cur + (size_t)s * a.cur_stream + (size_t)(row_on ? y0 + r : y0) * a.cur_pitch + (size_t)x0 * 3, h, row_on, cw);
        const uint8_t* prev = a.prev + (size_t)s * a.prev_stream;
        const Within valid = walk_range(walk_bounds(a, x0, y0, bw, bh));
#pragma unroll 1
        for (;;) {                                                       // ends: every window takes a move, of which warp_walk counts the rest
            // the window for the centre that is scored next
            constexpr int AROUND = P_REACH - 2;
            const int centre = w.at + 2 * lane_point(w.kind);
            const Within reach = {centre - pair(AROUND, AROUND), centre + pair(AROUND, AROUND)};
            const int wx0 = (x0 + disp_x(centre) - P_REACH) & ~3, wy0 = y0 + disp_y(centre) - P_REACH;
            {   // a lane keeps its group of 4 pixels (one column position) and goes down the rows, 3 rows apart
                constexpr int GROUPS = P_COLS / 4, RPP = 32 / GROUPS, PASSES = (P_ROWS + RPP - 1) / RPP, HALF = (PASSES + 1) / 2;
                const int gq = lane % GROUPS, row0 = lane / GROUPS, px0 = wx0 + 4 * gq;
                const bool col_ok = row0 < RPP && px0 >= 0 && (size_t)px0 * 3 + 12 <= a.prev_pitch;
                const uint8_t* src = prev + (size_t)px0 * 3;                          // px0 * 3 is a multiple of 12
                uint32_t* dst = win + row0 * P_PITCH + 4 * gq;
#pragma unroll
                for (int half = 0; half < 2; ++half) {                               // loads of half the passes, then their stores
                    uint32_t pa[HALF], pb[HALF], pc[HALF];
#pragma unroll
                    for (int k = 0; k < HALF; ++k) {
                        const int row = row0 + (half * HALF + k) * RPP, gy = wy0 + row;
                        pa[k] = pb[k] = pc[k] = 0;
                        if (col_ok && row < P_ROWS && gy >= 0 && gy < a.H) {
                            const uint32_t* q = (const uint32_t*)(src + (size_t)gy * a.prev_pitch);
                            pa[k] = dc_ld(q); pb[k] = dc_ld(q + 1); pc[k] = dc_ld(q + 2);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < HALF; ++k) {
                        const int row = row0 + (half * HALF + k) * RPP;
                        if (row0 < RPP && row < P_ROWS) store_pixels4(dst + (half * HALF + k) * RPP * P_PITCH, pa[k], pb[k], pc[k]);
                    }
                }
            }
            __syncwarp();
            // this lane's first word at displacement (0, 0): frame row y0 + r, pixel x0 + h, relative to the window's
            // origin (it may lie outside the window; only displacements near the centre are ever addressed)
            const uint32_t lane_base = (uint32_t)__cvta_generic_to_shared(win) + (uint32_t)(((r + y0 - wy0) * P_PITCH + (x0 - wx0) + h) * 4);
            const int st = warp_walk<P_PITCH, AHEAD>(a, lane_base, cw, row_on, lane_pixel_count(bw, h), bw < 16, valid, w, reach);
            if (st == 1) break;
            // make the chosen move; the next round scores its new points in a window around the new centre
            w.kind = w.nk;
            w.at = w.next; w.bs = w.ns;
            __syncwarp();                                                // every lane has finished reading the old window
        }
        if (lane == 0) publish_block(a, s, g, bw, bh, ((unsigned long long)w.bs << 32) | tie_key(disp_x(w.at), disp_y(w.at)));
    }
}

// Step 4 for 16-pixel blocks, in two launches.
// k_verify16_prep (one thread per block) rounds M, settles every block that needs no pixels -- M leaves the frame
// or the range for it, or its own best vector is M, so that Step 2 already holds the score (Section 4's second
// acceleration, exact in that case) -- and lists the others.  k_verify16_list scores the listed blocks, one
// half-warp per block and one lane per block row, so that no warp idles on blocks that were settled.

// Lane r of 16: the SSE of row r of block b displaced by (Mx, My).
__device__ __forceinline__ uint32_t score16(const MatchArgs& a, int s, int b, int Mx, int My, int r, bool on)
{
    const int by = b / a.Gx, bx = b - by * a.Gx, x0 = bx * 16, y0 = by * 16, bw = min(16, a.W - x0), bh = min(16, a.H - y0);
    if (!on || r >= bh) return 0;
    const uint4* c16 = (const uint4*)(a.cur + (size_t)s * a.cur_stream + (size_t)(y0 + r) * a.cur_pitch + (size_t)x0 * 3);   // 16-byte aligned
    const uint4 v0 = dc_ld(c16), v1 = dc_ld(c16 + 1), v2 = dc_ld(c16 + 2);
    uint32_t cw[12] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w, v2.x, v2.y, v2.z, v2.w};
    // the bytes of word j inside a block that the frame's right edge cuts
    auto inside = [&](int j) { const int nb = bw * 3 - 4 * j; return nb >= 4 ? 0xffffffffu : nb <= 0 ? 0u : (1u << (8 * nb)) - 1u; };
    if (bw < 16) {
#pragma unroll
        for (int j = 0; j < 12; ++j) cw[j] &= inside(j);
    }
    // the 48 bytes of the displaced row lie in four aligned 16-byte chunks (rows of the frame copy are padded):
    // four wide loads instead of thirteen narrow ones, then a word offset that is the same for a whole stream
    const uint8_t* p = a.prev + (size_t)s * a.prev_stream + (size_t)(y0 + My + r) * a.prev_pitch + (size_t)(x0 + Mx) * 3;
    const uint4* p16 = (const uint4*)((uintptr_t)p & ~(uintptr_t)15);
    const uint4 c0 = dc_ld(p16), c1 = dc_ld(p16 + 1), c2 = dc_ld(p16 + 2), c3 = dc_ld(p16 + 3);
    const uint32_t ww[16] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w, c2.x, c2.y, c2.z, c2.w, c3.x, c3.y, c3.z, c3.w};
    const uint32_t boff = (uint32_t)(uintptr_t)p & 15u, sh = (boff & 3u) * 8u;
    uint32_t w[13];
    switch (boff >> 2) {
    case 0:
#pragma unroll
        for (int j = 0; j < 13; ++j) w[j] = ww[j];
        break;
    case 1:
#pragma unroll
        for (int j = 0; j < 13; ++j) w[j] = ww[j + 1];
        break;
    case 2:
#pragma unroll
        for (int j = 0; j < 13; ++j) w[j] = ww[j + 2];
        break;
    default:
#pragma unroll
        for (int j = 0; j < 13; ++j) w[j] = ww[j + 3];
        break;
    }
    uint32_t acc[3] = {0, 0, 0};                                // three chains hide the dp4a latency
    if (bw == 16) {
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            const uint32_t d = __vabsdiffu4(cw[j], __funnelshift_r(w[j], w[j + 1], sh));
            acc[j % 3] = __dp4a(d, d, acc[j % 3]);
        }
    } else {
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            const uint32_t d = __vabsdiffu4(cw[j], __funnelshift_r(w[j], w[j + 1], sh) & inside(j));
            acc[j % 3] = __dp4a(d, d, acc[j % 3]);
        }
    }
    return acc[0] + acc[1] + acc[2];
}

__global__ void __launch_bounds__(256) k_verify16_prep(MatchArgs a, uint32_t* list, int32_t* list_count)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int lane = threadIdx.x & 31;
    const int per = a.Gx * a.Gy;
    const unsigned gi = blockIdx.x * 256u + threadIdx.x;                          // S * Gx * Gy < 2^31
    const bool in_grid = gi < (unsigned)(per * a.S);
    const int s = in_grid ? (int)(gi / (unsigned)per) : a.S - 1, b = in_grid ? (int)(gi - (unsigned)s * per) : 0;
    const Step4 r = settle(a, 16, gi, s, b, in_grid);
    if (r.settled) a.matched[gi] = (uint8_t)r.ok;
    if (in_grid && b == 0) { a.gmv[3 * s] = r.Mx; a.gmv[3 * s + 1] = r.My; a.gmv[3 * s + 2] = r.K; }
    // matched count: one atomic per warp and stream
    const unsigned same = __match_any_sync(0xffffffffu, s);
    const unsigned oks = __ballot_sync(0xffffffffu, r.ok);
    if (lane == __ffs(same) - 1 && (oks & same)) atomicAdd(&a.acc[4 * s + 3], __popc(oks & same));
    // the blocks whose pixels must be read
    const bool todo = in_grid && !r.settled;
    const unsigned tm = __ballot_sync(0xffffffffu, todo);
    if (tm) {
        int base = 0;
        if (lane == 0) base = atomicAdd(list_count, __popc(tm));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (todo) list[base + __popc(tm & ((1u << lane) - 1u))] = gi;
    }
}

__global__ void __launch_bounds__(256) k_verify16_list(MatchArgs a, const uint32_t* list, const int32_t* list_count)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int lane = threadIdx.x & 31, r = lane & 15, half = lane >> 4;
    const int per = a.Gx * a.Gy, n = *list_count;
    const int stride = gridDim.x * 16;
    for (int i0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 2; i0 < n; i0 += stride) {      // both halves of a warp stay in the loop together
        const int i = i0 + half;
        const bool on = i < n;
        const unsigned gi = on ? list[i] : 0u;
        const int s = (int)(gi / (unsigned)per), b = (int)(gi - (unsigned)s * per);
        const uint32_t sse = __reduce_add_sync(half ? 0xffff0000u : 0x0000ffffu, score16(a, s, b, a.gmv[3 * s], a.gmv[3 * s + 1], r, on));
        if (r == 0 && on) {
            const int by = b / a.Gx, bx = b - by * a.Gx;
            const int ok = sse <= a.limit[limit_index(a, min(16, a.W - bx * 16), min(16, a.H - by * 16))];
            a.matched[gi] = (uint8_t)ok;
            if (ok) atomicAdd(&a.acc[4 * s + 3], 1);
        }
    }
}

// Both in one launch, a half-warp per block from the start, where the blocks are few and a launch counts.  With more blocks than the SMs
// hold such warps the list deals the work out better (a whole pass in us, one launch and two: 8 full-HD streams, 65 280 blocks, 345
// and 315; 32 of them 1891 and 1818; 720p, 6 streams, 21 600 blocks, 436 and 418).
__global__ void __launch_bounds__(256) k_verify16_few(MatchArgs a)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int lane = threadIdx.x & 31, r = lane & 15, half = lane >> 4, per = a.Gx * a.Gy;
    const unsigned gi = (blockIdx.x * 8u + (threadIdx.x >> 5)) * 2u + half;
    const bool in_grid = gi < (unsigned)(per * a.S);
    const int s = in_grid ? (int)(gi / (unsigned)per) : a.S - 1, b = in_grid ? (int)(gi - (unsigned)s * per) : 0;
    const Step4 v = settle(a, 16, gi, s, b, in_grid);
    const bool todo = in_grid && !v.settled;
    const uint32_t sse = __reduce_add_sync(half ? 0xffff0000u : 0x0000ffffu, score16(a, s, b, v.Mx, v.My, r, todo));
    if (r != 0 || !in_grid) return;
    if (b == 0) { a.gmv[3 * s] = v.Mx; a.gmv[3 * s + 1] = v.My; a.gmv[3 * s + 2] = v.K; }
    const int by = b / a.Gx, bx = b - by * a.Gx;
    const int ok = todo ? sse <= a.limit[limit_index(a, min(16, a.W - bx * 16), min(16, a.H - by * 16))] : v.ok;
    a.matched[gi] = (uint8_t)ok;
    if (ok) atomicAdd(&a.acc[4 * s + 3], 1);
}

// ---------------------------------------------------------------------------------------------
// Fast Step 2: 16-pixel blocks, exhaustive search (plain integer ALU work: every displacement is scored)
// ---------------------------------------------------------------------------------------------
// One CTA per strip of 8 blocks, one warp per block.  The strip's search window (16 + 2R rows) is staged in
// shared memory once.  A lane owns one horizontal displacement dx; for one 4-byte column of the block it
// keeps the 16 rows of the current block in registers and walks down the window: every previous-frame word
// it loads is scored against all block rows it can pair with, i.e. for E_DY vertical displacements at once,
// so one (unaligned) load feeds up to 16 difference/accumulate pairs.  Displacements beyond the last full
// group of 32 dx values are scored one candidate per lane.  Blocks clipped by the frame edge are left to
// the generic kernel.
constexpr int E_DY = 13;                        // vertical displacements scored together (65 = 5 * 13 for R = 32)
constexpr int E_MAXR = 32;
constexpr int E_PITCH = 152;                    // window row in words: (128 + 64) px * 3 B + 15 B alignment + one spare word, 16-byte multiple
constexpr int E_MAXROWS = 16 + 2 * E_MAXR + E_DY - 1;   // plus rows only touched by displacements beyond R (scored, never compared)

__global__ void __launch_bounds__(256, 3) k_search_es16(MatchArgs a)
{
    dc_pdl_wait();
    dc_pdl_release();
    extern __shared__ uint32_t es_sm[];
    const int R = a.R, n_d = 2 * R + 1;
    const int chunks = (n_d + E_DY - 1) / E_DY;
    const int rows = 16 + chunks * E_DY - 1;                     // <= E_MAXROWS
    uint32_t* win = es_sm;
    uint32_t* cur_all = es_sm + rows * E_PITCH;
    const int strips = (a.Gx + 7) >> 3;
    const int strip = blockIdx.x % strips, by = (blockIdx.x / strips) % a.Gy, s = blockIdx.x / (strips * a.Gy);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int xs = strip * 128, y0 = by * 16;
    const int wx0 = ((xs - R) * 3) & ~15;                        // byte column of the window origin (may be < 0)
    const uint8_t* prev = a.prev + (size_t)s * a.prev_stream;
    const bool row_searched = (a.skip_k <= 1 || by % a.skip_k == 0) && a.H - y0 >= 16;
    for (int i = threadIdx.x; row_searched && i < rows * (E_PITCH / 4); i += 256) {
        const int row = i / (E_PITCH / 4), ci = i - row * (E_PITCH / 4);
        const int gy = y0 - R + row, gb = wx0 + ci * 16;
        uint4 v = make_uint4(0, 0, 0, 0);
        if (gy >= 0 && gy < a.H && gb >= 0 && gb + 16 <= (int)a.prev_pitch)
            v = dc_ld((const uint4*)(prev + (size_t)gy * a.prev_pitch + gb));
        *(uint4*)(win + row * E_PITCH + ci * 4) = v;
    }
    const int bx = strip * 8 + warp, x0 = bx * 16;
    const bool full = bx < a.Gx && a.W - x0 >= 16 && a.H - y0 >= 16;
    const bool skipped = a.skip_k > 1 && (bx % a.skip_k != 0 || by % a.skip_k != 0);
    uint32_t* curw = cur_all + warp * 192;
    if (full && !skipped) {                                       // the current block: 16 rows of 48 bytes
        const uint8_t* cb = a.cur + (size_t)s * a.cur_stream + (size_t)y0 * a.cur_pitch + (size_t)x0 * 3;
        for (int i = lane; i < 16 * 3; i += 32) {
            const int r = i / 3, q = i - r * 3;
            *(uint4*)(curw + r * 12 + q * 4) = dc_ld((const uint4*)(cb + (size_t)r * a.cur_pitch) + q);
        }
    }
    __syncthreads();
    if (bx >= a.Gx) return;
    const size_t g = (size_t)s * a.Gx * a.Gy + (size_t)by * a.Gx + bx;
    if (skipped) {
        if (lane == 0) { a.mv[2 * g] = 0; a.mv[2 * g + 1] = 0; a.sse[g] = 0xffffffffu; }
        return;
    }
    if (!full) return;                                            // clipped block: the generic kernel scores it

    unsigned long long bk = ~0ull;
    const int full_passes = n_d / 32;
    for (int pass = 0; pass < full_passes; ++pass) {
        const int dx = -R + pass * 32 + lane;
        const int boff = (x0 + dx) * 3 - wx0;
        const uint32_t sh = (boff & 3) * 8;
        const bool x_ok = x0 + dx >= 0 && x0 + dx + 16 <= a.W;
        for (int c = 0; c < chunks; ++c) {
            const int dy0 = -R + c * E_DY;
            uint32_t acc[E_DY];
#pragma unroll
            for (int d = 0; d < E_DY; ++d) acc[d] = 0;
            const uint32_t* col = win + (c * E_DY) * E_PITCH + (boff >> 2);      // window row of displacement dy0, block row 0
#pragma unroll 1
            for (int j = 0; j < 12; ++j) {
                uint32_t cw[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) cw[r] = curw[r * 12 + j];
#pragma unroll
                for (int p = 0; p < 16 + E_DY - 1; ++p) {
                    const uint32_t w = __funnelshift_r(col[p * E_PITCH + j], col[p * E_PITCH + j + 1], sh);
#pragma unroll
                    for (int r = 0; r < 16; ++r) {
                        if (p - r >= 0 && p - r < E_DY) {
                            const uint32_t t = __vabsdiffu4(cw[r], w);
                            acc[p - r] = __dp4a(t, t, acc[p - r]);
                        }
                    }
                }
            }
#pragma unroll
            for (int d = 0; d < E_DY; ++d) {
                const int dy = dy0 + d;
                if (x_ok && dy <= R && y0 + dy >= 0 && y0 + dy + 16 <= a.H) {
                    const unsigned long long k = cand_key(acc[d], dx, dy);
                    if (k < bk) bk = k;
                }
            }
        }
    }
    // the remaining dx columns: one candidate per lane and round
    const int dx_first = -R + full_passes * 32, n_left = (n_d - full_passes * 32) * n_d;
    for (int i = lane; i < n_left; i += 32) {
        const int dx = dx_first + i / n_d, dy = -R + i % n_d;
        if (x0 + dx < 0 || x0 + dx + 16 > a.W || y0 + dy < 0 || y0 + dy + 16 > a.H) continue;
        const int boff = (x0 + dx) * 3 - wx0;
        const uint32_t sh = (boff & 3) * 8;
        const uint32_t* col = win + (dy + R) * E_PITCH + (boff >> 2);
        uint32_t acc = 0;
#pragma unroll 2
        for (int r = 0; r < 16; ++r) {
            uint32_t lo = col[r * E_PITCH];
#pragma unroll
            for (int j = 0; j < 12; ++j) {
                const uint32_t hi = col[r * E_PITCH + j + 1];
                const uint32_t t = __vabsdiffu4(curw[r * 12 + j], __funnelshift_r(lo, hi, sh));
                acc = __dp4a(t, t, acc);
                lo = hi;
            }
        }
        const unsigned long long k = cand_key(acc, dx, dy);
        if (k < bk) bk = k;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long other = __shfl_xor_sync(0xffffffffu, bk, o);
        if (other < bk) bk = other;
    }
    if (lane == 0) publish_block(a, s, g, 16, 16, bk);            // the zero vector is always valid, so bk is set
}

// Step 3's sums and the list counters of a search that no frame copy precedes.  A kernel, not a memset: the search behind it is launched while it
// runs (the search without a cache, 720p, 85 -> 82 us a call).
__global__ void k_clear(int32_t* p, int n)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (int i = threadIdx.x; i < n; i += blockDim.x) p[i] = 0;
}

// Frame -> the library's aligned copy, one 16-byte vector of a row per thread.  Rows of any alignment are read as aligned
// 32-bit words and shifted; bytes beyond a row's end become zeros; the last words of the caller's buffer are read byte
// by byte.  Also zeroes the Step 3 sums and list counters of the search that follows (zero: n_zero words, or NULL).
__global__ void __launch_bounds__(256) k_copy_frame(const uint8_t* src, const uint8_t* src_end, size_t src_pitch, uint8_t* dst, size_t dst_pitch, int row_bytes,
                                                    unsigned total, int chunks, int32_t* zero, int n_zero)
{
    dc_pdl_wait();
    dc_pdl_release();
    if (zero && blockIdx.x == 0)
        for (int i = threadIdx.x; i < n_zero; i += blockDim.x) zero[i] = 0;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned row = i / (unsigned)chunks, c = i - row * (unsigned)chunks;
        const uint8_t* p = src + (size_t)row * src_pitch + c * 16u;
        const uint32_t sh = ((uint32_t)(uintptr_t)p & 3u) * 8u;
        const int left = row_bytes - (int)c * 16;                     // bytes of the row from here on
        uint4 v;
        if (((uintptr_t)p & 15u) == 0 && p + 16 <= src_end) {
            v = dc_ld((const uint4*)p);
        } else if (p + 20 <= src_end) {
            const uint32_t* q = (const uint32_t*)((uintptr_t)p & ~(uintptr_t)3);
            const uint32_t w0 = dc_ld(q), w1 = dc_ld(q + 1), w2 = dc_ld(q + 2), w3 = dc_ld(q + 3), w4 = sh ? dc_ld(q + 4) : 0u;
            v = make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh), __funnelshift_r(w3, w4, sh));
        } else {
            uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < 16; ++k) if (k < left) w[k >> 2] |= (uint32_t)dc_ld(p + k) << (8 * (k & 3));
            v = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (left < 16) {
            const uint32_t keep[4] = {left >= 4 ? ~0u : (1u << (8 * left)) - 1u, left >= 8 ? ~0u : left <= 4 ? 0u : (1u << (8 * (left - 4))) - 1u,
                                      left >= 12 ? ~0u : left <= 8 ? 0u : (1u << (8 * (left - 8))) - 1u, left <= 12 ? 0u : (1u << (8 * (left - 12))) - 1u};
            v.x &= keep[0]; v.y &= keep[1]; v.z &= keep[2]; v.w &= keep[3];
        }
        *(uint4*)(dst + (size_t)row * dst_pitch + c * 16u) = v;
    }
}

// Few blocks per warp where the frames have few.  us with 2, 4 and 8 (from launch to end): 640 x 360, 6 streams, 24 pixels (16 blocks per SM) 38, 43,
// 49; 227 x 227, 64 streams, 12 pixels (156) 18.6, 19.9, 24.7; 1080p, 2 streams, 10 pixels (280) 40, 26, 25, 8 pixels (438) 56, 33, 23.
void launch_verify(dc_cache* c, const MatchArgs& a)
{
    dc_prof_scope ps(c, DC_ST_VERIFY);
    const int blocks = a.S * a.Gx * a.Gy, share = blocks <= c->num_sms * 64 ? 2 : blocks <= c->num_sms * 280 ? 4 : 8;
    const dim3 grid((unsigned)dc_div_up(blocks, 8 * share));
    dc_launch_pdl(a.B <= 16 ? k_verify<false> : k_verify<true>, grid, 256, 0, c->stream, a, share);       // errors: cudaGetLastError below
}

// Step 2 over staged windows: every block, or (only_clipped, see dc_win_args) those that the 16-pixel kernels leave out
int search_win(dc_cache* c, const MatchArgs& a, int only_clipped)
{
    dc_win_args w;
    const size_t bytes = c->key_pitch * (size_t)c->cfg.height * c->S + 256;      // the library's copies and their spare tail
    w.cur = a.cur; w.cur_end = a.cur + bytes; w.cur_pitch = a.cur_pitch; w.cur_stream = a.cur_stream;
    w.prev = a.prev; w.prev_end = a.prev + bytes; w.prev_pitch = a.prev_pitch; w.prev_stream = a.prev_stream;
    w.W = a.W; w.H = a.H; w.B = a.B; w.R = a.R; w.Gx = a.Gx; w.Gy = a.Gy; w.S = a.S; w.search = a.search; w.skip_k = a.skip_k;
    w.only_clipped = only_clipped;
    for (int i = 0; i < 4; ++i) w.limit[i] = a.limit[i];
    w.mv = a.mv; w.sse = a.sse; w.acc = a.acc; w.status = a.status;
    dc_prof_scope ps(c, DC_ST_SEARCH);
    c->launches += 1;
    return dc_launch_search_win(w, c->num_sms, c->device, c->stream);
}

}  // namespace

// zero: the Step 3 sums of the match set that the search after this copy will use, or NULL
int dc_launch_clear(int32_t* p, int n, cudaStream_t stream)
{
    DC_CUDA(dc_launch_pdl(k_clear, dim3(1), 256, 0, stream, p, n));
    return DC_OK;
}

int dc_launch_copy_frame(dc_cache* c, const uint8_t* frame, size_t pitch, uint8_t* dst, int32_t* zero)
{
    const int row_bytes = c->cfg.width * 3, rows = c->cfg.height * c->S, chunks = (row_bytes + 15) / 16;
    const uint8_t* end = frame + pitch * (size_t)(rows - 1) + row_bytes;
    const size_t work = (size_t)rows * chunks;
    if (work > 0xffffffffull) return DC_ERR_CONFIG;                   // 64 GB of pixels
    size_t grid = (work + 255) / 256;
    if (grid > (size_t)c->num_sms * 32) grid = (size_t)c->num_sms * 32;
    dc_prof_scope ps(c, DC_ST_KEY_UPDATE);
    DC_CUDA(dc_launch_pdl(k_copy_frame, dim3((unsigned)grid), 256, 0, c->stream, frame, end, pitch, dst, c->key_pitch, row_bytes, (unsigned)work, chunks,
                          zero, 4 * c->S + 4));
    c->launches += 1;
    return DC_OK;
}

// The searches of 16-pixel blocks read a block's row as three aligned vectors: frames whose rows are whole blocks and start on 16 bytes
// need no copy to be matched, and the one that the next frame is matched against is written from the same registers.  Passes in us with the
// copy first and so: VGG, 32 full-HD streams 1803 and 1723; step by step, 8 full-HD streams 296 and 270; ResNet-50, 24 streams, 850 both.
// (Announced frames, whose match runs beside an inference, are copied first: VGG, 6 streams of 720p, 364 so and 379 in place, 32 full-HD
// streams 1665 both.)
bool dc_match_in_place(const dc_cache* c, const uint8_t* frame, size_t pitch)
{
    const bool walks = c->cfg.search == DC_SEARCH_DIAMOND || c->cfg.search == DC_SEARCH_THREE_STEP;
    return c->cfg.block == 16 && walks && c->cfg.skip_k <= 1 && c->cfg.width % 16 == 0 && (uintptr_t)frame % 16 == 0 && pitch % 16 == 0;
}

int dc_launch_match(dc_cache* c, uint8_t* cur_key, const uint8_t* prev_key, const dc_match_out* out, const uint8_t* frame, size_t pitch)
{
    MatchArgs a;
    a.cur = cur_key; a.cur_pitch = c->key_pitch; a.cur_stream = c->key_pitch * (size_t)c->cfg.height;
    a.copy = nullptr; a.copy_pitch = a.cur_pitch; a.copy_stream = a.cur_stream;
    if (frame) {
        a.copy = cur_key;
        a.cur = frame; a.cur_pitch = pitch; a.cur_stream = pitch * (size_t)c->cfg.height;
        dc_prof_scope ps(c, DC_ST_KEY_UPDATE);
        const int rc = dc_launch_clear(c->mv_acc, 4 * c->S + 4, c->stream);
        if (rc != DC_OK) return rc;
        c->launches += 1;
    }
    a.prev = prev_key; a.prev_pitch = c->key_pitch; a.prev_stream = c->key_pitch * (size_t)c->cfg.height;
    a.W = c->cfg.width; a.H = c->cfg.height; a.B = c->cfg.block; a.R = c->cfg.range;
    a.Gx = c->Gx; a.Gy = c->Gy; a.S = c->S; a.search = c->cfg.search; a.skip_k = c->cfg.skip_k; a.region_mode = c->cfg.region_mode;
    for (int i = 0; i < 4; ++i) a.limit[i] = c->sse_limit[i];
    // the caller's arrays, where given, take the place of the library's
    a.mv = out && out->mv ? out->mv : c->blk_mv; a.sse = out && out->sse ? out->sse : c->blk_sse;
    a.matched = out && out->matched ? out->matched : c->matched; a.acc = c->mv_acc; a.gmv = c->gmv;
    a.status = c->status;
    // Step 3 sums and, behind them, the counter of walks handed to the second search phase: zeroed by the frame copy
    int32_t* long_count = c->mv_acc + 4 * c->S;
    // walks that phase 2 may get: no more warps than blocks
    const dim3 long_grid((unsigned)min(c->num_sms * 4, dc_div_up(a.S * a.Gx * a.Gy, P_WARPS)));
    if (a.B == 16 && a.search == DC_SEARCH_DIAMOND) {
        {
            dc_prof_scope ps(c, DC_ST_SEARCH);
            const bool few = (long long)((a.Gx + 7) / 8) * ((a.Gy + W_VS - 1) / W_VS) * a.S <= 2 * c->num_sms;
            if (a.skip_k <= 1) {
                const dim3 tiles((a.Gx + 7) / 8, (a.Gy + W_VS - 1) / W_VS, a.S);
                DC_CUDA(dc_launch_pdl(few ? k_search_dsw<true> : k_search_dsw<false>, tiles, W_VS * 8 * 32, 0, c->stream, a, c->long_list, long_count));
                DC_CUDA(dc_launch_pdl(few ? k_search_dsw_long<true> : k_search_dsw_long<false>, long_grid, P_WARPS * 32, 0, c->stream, a, (const uint4*)c->long_list, (const int32_t*)long_count, long_count + 1));
            } else {
                DC_CUDA(dc_launch_pdl(k_mark_unsearched, dim3((unsigned)dc_div_up(a.S * a.Gx * a.Gy, 256)), 256, 0, c->stream, a));
                DC_CUDA(dc_launch_pdl(few ? k_search_dsw_long<true> : k_search_dsw_long<false>, long_grid, P_WARPS * 32, 0, c->stream, a, (const uint4*)nullptr, (const int32_t*)long_count, long_count + 1));
            }
            c->launches += 1;
        }
    } else if (a.B == 16 && a.search == DC_SEARCH_THREE_STEP && a.skip_k <= 1) {
        const TssShape t = tss_shape(a.R);
        static dc_once_per_device attr_set;
        if (attr_set.first(c->device)) {
            const int most = (int)tss_window_bytes(tss_shape(64));
            DC_CUDA(cudaFuncSetAttribute(k_search_tss16<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
            DC_CUDA(cudaFuncSetAttribute(k_search_tss16<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
        }
        dc_prof_scope ps(c, DC_ST_SEARCH);
        const dim3 tiles((unsigned)((a.Gx + 7) / 8), (unsigned)((a.Gy + TSS_VS - 1) / TSS_VS), (unsigned)a.S);
        DC_CUDA(dc_launch_pdl((long long)tiles.x * tiles.y * tiles.z <= 2 * c->num_sms ? k_search_tss16<true> : k_search_tss16<false>, tiles, TSS_VS * 8 * 32,
                              tss_window_bytes(t), c->stream, a, t));
    } else if (a.B == 16 && a.search == DC_SEARCH_EXHAUSTIVE && a.R <= E_MAXR && a.W >= 16 && a.H >= 16) {
        const int chunks = (2 * a.R + 1 + E_DY - 1) / E_DY;
        const size_t smem = ((size_t)(16 + chunks * E_DY - 1) * E_PITCH + 8 * 192) * sizeof(uint32_t);
        static dc_once_per_device attr_set;
        if (attr_set.first(c->device)) {
            DC_CUDA(cudaFuncSetAttribute(k_search_es16, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(((size_t)E_MAXROWS * E_PITCH + 8 * 192) * sizeof(uint32_t))));
        }
        {
            dc_prof_scope ps(c, DC_ST_SEARCH);
            DC_CUDA(dc_launch_pdl(k_search_es16, dim3((unsigned)(((a.Gx + 7) / 8) * a.Gy * a.S)), 256, smem, c->stream, a));
        }
        if (a.W % 16 != 0 || a.H % 16 != 0) {                   // blocks clipped by the right / bottom edge
            const int rc = search_win(c, a, 1);
            if (rc != DC_OK) return rc;
        }
    } else {
        const int rc = search_win(c, a, 0);
        if (rc != DC_OK) return rc;
    }
    if (a.region_mode == DC_REGIONS_PER_BLOCK) {
        dc_prof_scope ps(c, DC_ST_VERIFY);
        DC_CUDA(dc_launch_pdl(k_accept_own, dim3((unsigned)dc_div_up(a.S * a.Gx * a.Gy, 256)), 256, 0, c->stream, a));
    } else if (a.B == 16) {
        dc_prof_scope ps(c, DC_ST_VERIFY);
        const int blocks = a.S * a.Gx * a.Gy;
        if (blocks <= c->num_sms * 64) {
            DC_CUDA(dc_launch_pdl(k_verify16_few, dim3((unsigned)dc_div_up(blocks, 16)), 256, 0, c->stream, a));
        } else {
            int32_t* todo_count = long_count + 2;                       // zeroed with the Step 3 sums; the walk list is free again
            DC_CUDA(dc_launch_pdl(k_verify16_prep, dim3((unsigned)dc_div_up(a.S * a.Gx * a.Gy, 256)), 256, 0, c->stream, a, (uint32_t*)c->long_list, todo_count));
            DC_CUDA(dc_launch_pdl(k_verify16_list, dim3((unsigned)min(c->num_sms * 8, dc_div_up(a.S * a.Gx * a.Gy, 16))), 256, 0, c->stream, a,
                                  (const uint32_t*)c->long_list, (const int32_t*)todo_count));
            c->launches += 1;
        }
    } else {
        launch_verify(c, a);
    }
    {
        dc_prof_scope ps(c, DC_ST_MERGE);
        const bool own = a.region_mode == DC_REGIONS_PER_BLOCK;
        const size_t need = merge_smem_bytes(a.Gx, a.Gy, own);
        static dc_once_per_device attr_set;
        if (attr_set.first(c->device)) DC_CUDA(cudaFuncSetAttribute(k_merge, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
        const MergeArgs ma = {a.matched, own ? a.mv : nullptr, c->gmv, a.W, a.H, a.B, a.Gx, a.Gy, c->max_regions, c->run_end, c->regions0, c->n_regions,
                              c->status, out ? out->gmv : nullptr, out ? out->n_regions : nullptr, out ? out->regions : nullptr};
        if (need <= 160 * 1024) DC_CUDA(dc_launch_pdl(k_merge, dim3((unsigned)c->S), 1024, need, c->stream, ma));
        else DC_CUDA(dc_launch_pdl(k_merge_large, dim3((unsigned)c->S), 1024, 0, c->stream, ma));
    }
    c->launches += 3;
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}
