// What the kernels that walk (dc_match.cu, dc_search_win.cu) share: the points of the diamond search, and displacements as pairs.
#pragma once
#include "dc_common.cuh"

// Points around a centre: 0-7 the large diamond, 8 its centre, 9-12 the small diamond.
__host__ __device__ constexpr int point_x(int i)
{
    constexpr int t[13] = {0, -1, 1, -2, 2, -1, 1, 0, 0, 0, -1, 1, 0};
    return t[i];
}
__host__ __device__ constexpr int point_y(int i)
{
    constexpr int t[13] = {-2, -1, -1, 0, 0, 1, 1, 2, 0, -1, 0, 0, 1};
    return t[i];
}
// A round of the diamond search scores one of ten point sets around the current centre: kind 0-7, the points of the large diamond that are
// new after the move along diamond point `kind` (the others lost to the new centre already and cannot win); kind 8, the first round
// (centre and all eight points); kind 9, the small diamond.
constexpr int KIND_FIRST = 8, KIND_SMALL = 9;
__host__ __device__ constexpr uint32_t kind_mask(int kind)
{
    constexpr uint32_t t[10] = {31u, 11u, 21u, 171u, 213u, 168u, 208u, 248u, 0x1ffu, 0x1e00u};
    return t[kind];
}
static __constant__ uint32_t c_kind_mask[10] = {31u, 11u, 21u, 171u, 213u, 168u, 208u, 248u, 0x1ffu, 0x1e00u};

// Displacements in a walk are pairs of 16-bit numbers in one register, dy + kBias above dx + kBias: both axes are compared at once, and
// a lane's registers are what bounds the warps per SM.
constexpr int kBias = 128;
__host__ __device__ constexpr int pair(int dx, int dy) { return dy * 65536 + dx; }                 // a difference of displacements
__host__ __device__ constexpr int disp(int dx, int dy) { return pair(dx + kBias, dy + kBias); }
__device__ __forceinline__ int disp_x(int d) { return (d & 0xffff) - kBias; }
__device__ __forceinline__ int disp_y(int d) { return (d >> 16) - kBias; }
struct Within { int lo, hi; };                                                                     // a range of displacements
__device__ __forceinline__ bool within(int d, Within r) { return (int)__vminu2(__vmaxu2((unsigned)d, (unsigned)r.lo), (unsigned)r.hi) == d; }

// Candidates are ordered by (SSE, |dx| + |dy|, dy, dx); this is the order behind the SSE.
__device__ __forceinline__ uint32_t tie_key(int dx, int dy)
{
    return ((uint32_t)(abs(dx) + abs(dy)) << 16) | ((uint32_t)(dy + 128) << 8) | (uint32_t)(dx + 128);
}
// The best of the candidates that the lanes hold: lane `d`'s displacement, `mine` its score (2^32 - 1: none).  Returns its lane.
__device__ __forceinline__ int best_lane(uint32_t mine, int d, uint32_t& score)
{
    const unsigned all = 0xffffffffu;
    score = __reduce_min_sync(all, mine);
    unsigned best = __ballot_sync(all, mine == score);
    if (best & (best - 1)) {                                      // equal scores: the exact order among them
        const uint32_t kt = tie_key(disp_x(d), disp_y(d)), kb = __reduce_min_sync(all, mine == score ? kt : 0xffffffffu);
        best = __ballot_sync(all, mine == score && kt == kb);
    }
    return __ffs(best) - 1;
}
// This lane's point (lanes 0 to 12), from the centre.
__device__ __forceinline__ int lane_point(int lane)
{
    // x + 2 and y + 2 of the points, three bits each
    constexpr auto pack = [](bool y) { unsigned long long v = 0; for (int i = 0; i < 13; ++i) v |= (unsigned long long)((y ? point_y(i) : point_x(i)) + 2) << (3 * i); return v; };
    constexpr unsigned long long X = pack(false), Y = pack(true);
    const int i = lane < 13 ? lane : 8;
    return pair((int)(X >> (3 * i) & 7) - 2, (int)(Y >> (3 * i) & 7) - 2);
}

template <int OFF>
__device__ __forceinline__ uint32_t lds_at(uint32_t p)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(p), "n"(OFF) : "memory");
    return v;
}
