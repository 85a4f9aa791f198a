// Partial convolution on CUDA cores for stride-1 1x1, 3x3 and 5x5 layers (float32 and bfloat16 channel counts that the
// tensor-core kernels do not take), grouped ones included, and for layers with one output pixel per stream.
//   k_conv_simt  register-blocked, packed fp32 FMAs
//   k_dense      fully-connected layers: one warp per slice of the reduction
// Only pixels whose bit in the tile's reuse bitmap is clear are written.
#include "dc_common.cuh"

namespace {

template <typename T> __device__ __forceinline__ T to_elt(float v);
template <> __device__ __forceinline__ float to_elt<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_elt<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// ---------------------------------------------------------------------------------------------
// Stride-1 KW x KW convolution, register blocked
// ---------------------------------------------------------------------------------------------
// A work item is one dirty 16 x 8 tile times BN output channels.  A thread owns one tile row (8 pixels) and TC channels:
// 8 x TC sums in registers, as pairs of neighbouring channels for the packed FMA (fma.rn.f32x2: each half rounded like
// fmaf; half the instructions).  Per chunk of CI input channels the (16 + KW - 1) x (8 + KW - 1) input patch lies in
// shared memory channel-major ([ci][row][12]) and the weights as [tap][ci][BN]: a thread loads the 8 + KW - 1 values of
// a patch row once and uses them for all KW taps of that row, so an FMA costs 1/10 of a shared-memory load (3 x 3,
// TC = 8).  lane = 8 * channel group + row: with a row pitch of 12 words the eight rows of a 16-byte load fall in
// different banks and the weights are broadcast.  Both operands are double buffered (patch through registers, weights
// by cp.async), one barrier per chunk.  A warp whose eight rows are all reused skips the arithmetic.
// KS > 1: the CTA holds KS such groups of warps, each takes every KS-th chunk with buffers and a named barrier of its
// own, and their sums meet in shared memory at the end: for layers with so few tiles that one group's serial walk over
// the channels would set the time.
// What bounds it: the FMA pipe where the layer fills the machine, else the walk of one warp (see simt_shape for both).
constexpr int kSimtPitch = 12;

__host__ __device__ constexpr int simt_threads(int BN, int TC) { return 16 * BN / TC; }
__host__ __device__ constexpr int simt_patch_floats(int KW, int CI) { return CI * (DC_TILE_H + KW - 1) * kSimtPitch; }
__host__ __device__ constexpr int simt_weight_floats(int KW, int CI, int BN) { return KW * KW * CI * BN; }
// Shared memory of one group of warps: two buffers of both operands (one when the group has a single chunk: more CTAs per
// SM then), and with KS > 1 at least the room its sums take when the groups meet.
__host__ __device__ constexpr int simt_group_floats(int KW, int CI, int BN, int KS, int bufs)
{
    const int f = bufs * (simt_patch_floats(KW, CI) + simt_weight_floats(KW, CI, BN));
    return KS > 1 && 128 * BN > f ? 128 * BN : f;
}
// input channels per chunk: enough arithmetic between two barriers, two buffers within 51 KB
__host__ __device__ constexpr int simt_ci(int KW, bool few) { return KW == 1 ? 16 : KW == 3 && !few ? 8 : 4; }

struct SimtArgs {
    const void* in; const float* w; const float* bias; void* out;     // w: [groups * nb_g][chunks][KW * KW][CI][BN], zero padded
    const int32_t* tile_list; const int32_t* tile_count; const uint32_t* masks;
    int Hi, Wi, Ci, Ho, Wo, Co, p, relu, tiles_x, tiles_y;
    int Cig, Cog, nb_g, NB, chunks;                                   // channels per group, blocks per group, blocks in all
    int early;                                                        // dc_lists_settled()
    int vec;                                                          // four channels of a pixel are one aligned load
};

__device__ __forceinline__ unsigned long long pack2(float lo, float hi)
{
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b)
{
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)), "l"(src) : "memory");
}
// four channels of one pixel as floats; n < 4: the channels that exist
__device__ __forceinline__ float4 ld_quad(const float* p, int n, bool vec)
{
    if (vec) return dc_ld((const float4*)p);
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) v.x = dc_ld(p);
    if (n > 1) v.y = dc_ld(p + 1);
    if (n > 2) v.z = dc_ld(p + 2);
    if (n > 3) v.w = dc_ld(p + 3);
    return v;
}
__device__ __forceinline__ float4 ld_quad(const __nv_bfloat16* p, int n, bool vec)
{
    if (vec) {
        const uint2 u = dc_ld((const uint2*)p);
        return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
    }
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) v.x = __bfloat162float(p[0]);
    if (n > 1) v.y = __bfloat162float(p[1]);
    if (n > 2) v.z = __bfloat162float(p[2]);
    if (n > 3) v.w = __bfloat162float(p[3]);
    return v;
}
__device__ __forceinline__ void st_quad(float* p, float4 v) { *(float4*)p = v; }
__device__ __forceinline__ void st_quad(__nv_bfloat16* p, float4 v)
{
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    *(uint2*)p = make_uint2(*(const uint32_t*)&a, *(const uint32_t*)&b);
}

template <typename T, int KW, int CI, int BN, int TC, int KS>
__global__ void __launch_bounds__(KS * simt_threads(BN, TC)) k_conv_simt(const SimtArgs a)
{
    constexpr int THREADS = simt_threads(BN, TC), PH = DC_TILE_H + KW - 1, PW = DC_TILE_W + KW - 1, PX = PH * PW;
    constexpr int PLANE = PH * kSimtPitch, ABUF = simt_patch_floats(KW, CI), BBUF = simt_weight_floats(KW, CI, BN);
    constexpr int QUADS = PX * (CI / 4), QPT = (QUADS + THREADS - 1) / THREADS;
    constexpr int UNROLL = KW == 3 && TC == 8 ? 4 : 2;                // measured: 1, 2, 4 channels per turn 464, 456, 449 us (64 -> 64, 113 x 113, 24 streams)
    extern __shared__ __align__(16) float simt_smem_raw[];
    const int ks = threadIdx.x / THREADS, tid = threadIdx.x % THREADS, warp = tid >> 5, lane = tid & 31;
    const int bufs = KS == 1 || a.chunks > KS ? 2 : 1;
    float* As = simt_smem_raw + ks * simt_group_floats(KW, CI, BN, KS, bufs);   // [bufs][CI][PH][12]
    float* Bs = As + bufs * ABUF;                                     // [bufs][KW * KW][CI][BN]
    const int prow = (warp & 1) * 8 + (lane & 7), coff = (warp >> 1) * (4 * TC) + (lane >> 3) * TC;

    const int nb = blockIdx.x % a.NB, ti = blockIdx.x / a.NB;
    const float* wsrc = a.w + (size_t)nb * a.chunks * BBUF;
    auto fetch_weights = [&](int chunk, int buf) {
        const float* src = wsrc + (size_t)chunk * BBUF;
        float* dst = Bs + buf * BBUF;
        for (int e = tid * 4; e < BBUF; e += THREADS * 4) cp_async16(dst + e, src + e);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    if (ks < a.chunks) fetch_weights(ks, 0);                                              // the weights are nobody's output: before the wait
    // the previous kernel's output is read only after the wait; the tile list and the bitmaps too, unless they are older than it
    if (!a.early) { dc_pdl_wait(); dc_pdl_release(); }
    const bool present = ti < __ldcg(a.tile_count);
    const int tile = present ? __ldcg(a.tile_list + ti) : 0;
    const int per = a.tiles_x * a.tiles_y, s = tile / per, t = tile - s * per, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
    const int grp = nb / a.nb_g, cb = (nb - grp * a.nb_g) * BN;       // group, first channel of the block inside it
    const int oy = ty * DC_TILE_H + prow, ox0 = tx * DC_TILE_W;
    // the row's pixels that this item has to write: inside the map and not reused
    uint32_t todo = ~(__ldcg(a.masks + (size_t)tile * 4 + (prow >> 2)) >> (8 * (prow & 3))) & 0xffu;
    if (a.Wo - ox0 < DC_TILE_W) todo &= (1u << (a.Wo - ox0)) - 1u;
    if (oy >= a.Ho) todo = 0;
    const bool busy = __any_sync(0xffffffffu, todo != 0);
    if (a.early) { dc_pdl_wait(); dc_pdl_release(); }
    if (!present) { asm volatile("cp.async.wait_all;" ::: "memory"); return; }

    const T* in = (const T*)a.in + (size_t)s * a.Hi * a.Wi * a.Ci + grp * a.Cig;
    const bool vec = a.vec != 0;
    float4 stage[QPT];
    auto load_patch = [&](int chunk) {
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            const int i = tid + u * THREADS, q = i / PX, px = i - q * PX, y = px / PW, x = px - y * PW;
            const int iy = ty * DC_TILE_H - a.p + y, ix = ox0 - a.p + x, c0 = chunk * CI + 4 * q;
            stage[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < QUADS && iy >= 0 && iy < a.Hi && ix >= 0 && ix < a.Wi && c0 < a.Cig)
                stage[u] = ld_quad(in + ((size_t)iy * a.Wi + ix) * a.Ci + c0, a.Cig - c0, vec);
        }
    };
    auto store_patch = [&](int buf) {
#pragma unroll
        for (int u = 0; u < QPT; ++u) {
            const int i = tid + u * THREADS, q = i / PX, px = i - q * PX, y = px / PW, x = px - y * PW;
            if (i < QUADS) {
                float* d = As + buf * ABUF + 4 * q * PLANE + y * kSimtPitch + x;
                d[0] = stage[u].x; d[PLANE] = stage[u].y; d[2 * PLANE] = stage[u].z; d[3 * PLANE] = stage[u].w;
            }
        }
    };
    unsigned long long acc[DC_TILE_W][TC / 2];
#pragma unroll
    for (int i = 0; i < DC_TILE_W; ++i)
#pragma unroll
        for (int j = 0; j < TC / 2; ++j) acc[i][j] = 0ull;

    if (ks < a.chunks) { load_patch(ks); store_patch(0); }
    int buf = 0;
    for (int chunk = ks; chunk < a.chunks; chunk += KS, buf ^= 1) {
        asm volatile("cp.async.wait_all;" ::: "memory");
        // chunk staged by the whole group; the other buffers are free
        if (KS == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(ks + 1), "r"(THREADS) : "memory");
        const bool more = chunk + KS < a.chunks;
        if (more) { fetch_weights(chunk + KS, buf ^ 1); load_patch(chunk + KS); }
        if (busy) {
            const float* ap = As + buf * ABUF + prow * kSimtPitch;
            const float* bp = Bs + buf * BBUF + coff;
#pragma unroll UNROLL
            for (int ci = 0; ci < CI; ++ci) {
#pragma unroll
                for (int ky = 0; ky < KW; ++ky) {
                    unsigned long long av[PW];
                    {
                        const float4* r = (const float4*)(ap + ci * PLANE + ky * kSimtPitch);
                        float v[12];
#pragma unroll
                        for (int k = 0; k < (PW + 3) / 4; ++k) { const float4 q = r[k]; v[4 * k] = q.x; v[4 * k + 1] = q.y; v[4 * k + 2] = q.z; v[4 * k + 3] = q.w; }
#pragma unroll
                        for (int k = 0; k < PW; ++k) av[k] = pack2(v[k], v[k]);
                    }
#pragma unroll
                    for (int kx = 0; kx < KW; ++kx) {
                        const ulonglong2* wv = (const ulonglong2*)(bp + ((ky * KW + kx) * CI + ci) * BN);
#pragma unroll
                        for (int j = 0; j < TC / 4; ++j) {
                            const ulonglong2 b = wv[j];
#pragma unroll
                            for (int i = 0; i < DC_TILE_W; ++i) { fma2(acc[i][2 * j], av[i + kx], b.x); fma2(acc[i][2 * j + 1], av[i + kx], b.y); }
                        }
                    }
                }
            }
        }
        if (more) store_patch(buf ^ 1);
    }
    // with KS groups, each finishes 8 / KS of the row's pixels
    constexpr int PPG = DC_TILE_W / KS;
    unsigned long long sum[PPG][TC / 2];
    if constexpr (KS == 1) {
#pragma unroll
        for (int i = 0; i < DC_TILE_W; ++i)
#pragma unroll
            for (int j = 0; j < TC / 2; ++j) sum[i][j] = acc[i][j];
    } else {
        unsigned long long* part = (unsigned long long*)simt_smem_raw;  // [KS][8][TC / 2][THREADS]
        __syncthreads();
#pragma unroll
        for (int i = 0; i < DC_TILE_W; ++i)
#pragma unroll
            for (int j = 0; j < TC / 2; ++j) part[((ks * DC_TILE_W + i) * (TC / 2) + j) * THREADS + tid] = acc[i][j];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < PPG; ++i)
#pragma unroll
            for (int j = 0; j < TC / 2; ++j) {
                unsigned long long v = part[((ks * PPG + i) * (TC / 2) + j) * THREADS + tid];
#pragma unroll
                for (int g = 1; g < KS; ++g) v = add2(v, part[((g * DC_TILE_W + ks * PPG + i) * (TC / 2) + j) * THREADS + tid]);
                sum[i][j] = v;
            }
        todo = (todo >> (ks * PPG)) & ((1u << PPG) - 1u);
    }
    if (todo) {
        const int c0 = cb + coff;                                     // channel inside the group
        T* out = (T*)a.out + (((size_t)s * a.Ho + oy) * a.Wo + ox0 + ks * PPG) * a.Co + grp * a.Cog + c0;
        const float* bias = a.bias + grp * a.Cog + c0;
#pragma unroll
        for (int j = 0; j < TC / 4; ++j) {
            if (c0 + 4 * j >= a.Cog) continue;                        // channels come in fours
            const float b0 = __ldg(bias + 4 * j), b1 = __ldg(bias + 4 * j + 1), b2 = __ldg(bias + 4 * j + 2), b3 = __ldg(bias + 4 * j + 3);
#pragma unroll
            for (int i = 0; i < PPG; ++i) {
                if (!((todo >> i) & 1u)) continue;
                float4 v;
                unpack2(sum[i][2 * j], v.x, v.y); unpack2(sum[i][2 * j + 1], v.z, v.w);
                v.x += b0; v.y += b1; v.z += b2; v.w += b3;
                if (a.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
                st_quad(out + (size_t)i * a.Co + 4 * j, v);
            }
        }
    }
}

// weights [cout][taps][Cig] -> [groups * nb_g][chunks][taps][CI][BN], zeros beyond the last channel
template <typename T>
__global__ void k_pack_simt(const T* w, int taps, int Cig, int Cog, int nb_g, int NB, int chunks, int CI, int BN, float* out)
{
    const size_t total = (size_t)NB * chunks * taps * CI * BN;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i;
        const int n = (int)(r % BN); r /= BN;
        const int ci = (int)(r % CI); r /= CI;
        const int tap = (int)(r % taps); r /= taps;
        const int chunk = (int)(r % chunks), nb = (int)(r / chunks);
        const int grp = nb / nb_g, co = (nb - grp * nb_g) * BN + n, c = chunk * CI + ci;
        out[i] = co < Cog && c < Cig ? (float)w[((size_t)(grp * Cog + co) * taps + tap) * Cig + c] : 0.f;
    }
}

// ---------------------------------------------------------------------------------------------
// One output pixel per stream (fully-connected layers): out[s][n] = sum over K of in[s][k] w[n][k]
// ---------------------------------------------------------------------------------------------
// A CTA takes 4 streams x 4 outputs, its eight warps a slice of K each, a lane every 32nd vector of 4 values of the
// slice: 8 vector loads feed 64 FMAs, and even a small layer spreads over S * N / 16 CTAs (a tile of the convolution
// kernels would hold one useful pixel of 128 and walk K alone).
constexpr int DN_S = 4, DN_N = 4, DN_WARPS = 8;

struct DenseArgs { const void* in; const void* w; const float* bias; void* out; const uint32_t* masks; int S, N, K, relu, vec; };

template <typename T>
__global__ void __launch_bounds__(DN_WARPS * 32) k_dense(const DenseArgs a)
{
    __shared__ float part[DN_WARPS][DN_S * DN_N];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * DN_N, s0 = blockIdx.y * DN_S;
    dc_pdl_wait();
    dc_pdl_release();
    const int nv = (a.K + 3) / 4, per = (nv + DN_WARPS - 1) / DN_WARPS, lo = warp * per, hi = min(nv, lo + per);
    const bool vec = a.vec != 0;
    float acc[DN_S * DN_N];
#pragma unroll
    for (int i = 0; i < DN_S * DN_N; ++i) acc[i] = 0.f;
    const T* in = (const T*)a.in; const T* w = (const T*)a.w;
    for (int v = lo + lane; v < hi; v += 32) {
        float4 x[DN_S], y[DN_N];
#pragma unroll
        for (int i = 0; i < DN_S; ++i) x[i] = ld_quad(in + (size_t)min(s0 + i, a.S - 1) * a.K + 4 * v, a.K - 4 * v, vec);
#pragma unroll
        for (int j = 0; j < DN_N; ++j) y[j] = ld_quad(w + (size_t)min(n0 + j, a.N - 1) * a.K + 4 * v, a.K - 4 * v, vec);
#pragma unroll
        for (int i = 0; i < DN_S; ++i)
#pragma unroll
            for (int j = 0; j < DN_N; ++j) {
                float& c = acc[i * DN_N + j];
                c = fmaf(x[i].x, y[j].x, c); c = fmaf(x[i].y, y[j].y, c); c = fmaf(x[i].z, y[j].z, c); c = fmaf(x[i].w, y[j].w, c);
            }
    }
#pragma unroll
    for (int i = 0; i < DN_S * DN_N; ++i) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
        if (lane == 0) part[warp][i] = acc[i];
    }
    __syncthreads();
    if (threadIdx.x < DN_S * DN_N) {
        const int s = s0 + threadIdx.x / DN_N, n = n0 + threadIdx.x % DN_N;
        if (s < a.S && n < a.N && !(a.masks[(size_t)s * 4] & 1u)) {
            float v = __ldg(a.bias + n);
            for (int k = 0; k < DN_WARPS; ++k) v += part[k][threadIdx.x];
            if (a.relu) v = fmaxf(v, 0.f);
            ((T*)a.out)[(size_t)s * a.N + n] = to_elt<T>(v);
        }
    }
}

}  // namespace

static bool simt_ok(const dc_cache* c, const dc_layer_desc& d)
{
    const int G = d.groups > 1 ? d.groups : 1;
    return d.kind == DC_CONV && d.sh == 1 && d.sw == 1 && d.kh == d.kw && d.ph == d.pw && (d.cout / G) % 4 == 0 &&
           (d.kw == 1 || d.kw == 3 || (d.kw == 5 && c->cfg.dtype == DC_FP32));
}
// one output pixel and no padding: the reduction is the layer's whole input, in memory order
bool dc_dense_ok(const dc_layer_rt& L)
{
    const dc_layer_desc& d = L.d;
    return d.kind == DC_CONV && d.out_h == 1 && d.out_w == 1 && d.kh == L.in_h && d.kw == L.in_w && d.ph == 0 && d.pw == 0 && d.groups <= 1;
}

struct SimtShape { int CI, BN, TC, KS; };
// 8 x 8 sums per thread everywhere but in narrow layers (8 x 4 needs twice the shared-memory loads per FMA).  A layer
// fills the machine when it has 16 warps per SM with every tile dirty (cached frames leave a part of that): then one
// group of warps per CTA and wide blocks (64 -> 64 channels at 113 x 113, 24 streams: 449 us, 50 TFLOP/s of useful work
// in tiles that are 83 % full; the one-pixel-per-thread kernel took 1.9 ms).  With fewer, four groups share the chunks (the
// small CNN on one stream: convolutions 395 -> 108 us; capping registers for two such CTAs per SM spills: 121 us).
static SimtShape simt_shape(const dc_cache* c, const dc_layer_rt& L)
{
    const int G = L.d.groups > 1 ? L.d.groups : 1, cog = L.d.cout / G, cig = L.d.cin / G;
    const long long tiles = (long long)L.tiles_x * L.tiles_y * c->S * G;
    SimtShape s;
    s.CI = simt_ci(L.d.kw, cig <= 4);
    s.BN = cog <= 16 ? 16 : c->cfg.dtype == DC_FP32 && (cog % 64 == 0 || cog > 96) ? 64 : 32;
    s.TC = s.BN == 16 ? 4 : 8;
    s.KS = 1;
    if (tiles * dc_div_up(cog, s.BN) * (simt_threads(s.BN, s.TC) / 32) < (long long)c->num_sms * 16) {
        if (s.BN == 64) s.BN = 32;
        if (dc_div_up(cig, s.CI) >= 4) s.KS = 4;
    }
    return s;
}

void dc_simt_order(const dc_cache* c, const dc_layer_rt& L, int* ci, int* ks)
{
    const SimtShape s = simt_shape(c, L);
    *ci = s.CI; *ks = s.KS;
}

template <typename T, int KW, int CI, int BN, int TC, int KS>
static int launch_simt(dc_cache* c, const SimtArgs& a, int max_tiles)
{
    const int smem = 4 * KS * simt_group_floats(KW, CI, BN, KS, KS == 1 || a.chunks > KS ? 2 : 1);
    constexpr int most = 4 * KS * simt_group_floats(KW, CI, BN, KS, 2);
    if (most > 48 * 1024) {
        static dc_once_per_device attr_set;
        if (attr_set.first(c->device)) DC_CUDA(cudaFuncSetAttribute(k_conv_simt<T, KW, CI, BN, TC, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    }
    // one CTA per item: the hardware hands items out as CTAs finish, those beyond the device-side count leave at once
    DC_CUDA(dc_launch_pdl(k_conv_simt<T, KW, CI, BN, TC, KS>, dim3((unsigned)(max_tiles * a.NB)), KS * simt_threads(BN, TC), smem, c->stream, a));
    return DC_OK;
}
template <typename T, int KW, int CI>
static int launch_simt_shape(dc_cache* c, const SimtArgs& a, const SimtShape& s, int max_tiles)
{
    if constexpr (KW != 3 || CI != 4)                                 // few input channels are one chunk
        if (s.KS == 4) return s.BN == 16 ? launch_simt<T, KW, CI, 16, 4, 4>(c, a, max_tiles) : launch_simt<T, KW, CI, 32, 8, 4>(c, a, max_tiles);
    if (s.BN == 16) return launch_simt<T, KW, CI, 16, 4, 1>(c, a, max_tiles);
    if constexpr (sizeof(T) == 4) if (s.BN == 64) return launch_simt<T, KW, CI, 64, 8, 1>(c, a, max_tiles);
    return launch_simt<T, KW, CI, 32, 8, 1>(c, a, max_tiles);
}
template <typename T>
static int launch_simt_kw(dc_cache* c, const SimtArgs& a, int kw, const SimtShape& s, int max_tiles)
{
    if (kw == 1) return launch_simt_shape<T, 1, simt_ci(1, false)>(c, a, s, max_tiles);
    if constexpr (sizeof(T) == 4) if (kw == 5) return launch_simt_shape<T, 5, simt_ci(5, false)>(c, a, s, max_tiles);
    if (s.CI == 4) return launch_simt_shape<T, 3, 4>(c, a, s, max_tiles);
    return launch_simt_shape<T, 3, simt_ci(3, false)>(c, a, s, max_tiles);
}

// A caller's map may start at any element: four of them are one load or store only where they lie on a boundary of four.
static bool quads(const dc_cache* c, const void* map) { return (uintptr_t)map % (4u * (unsigned)c->elt) == 0; }
bool dc_conv_simt_stores(const dc_cache* c, const void* out) { return quads(c, out); }

int dc_launch_conv_simt(dc_cache* c, int layer, const void* in, void* out, const int32_t* tile_list, const int32_t* tile_count,
                        const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const SimtShape sh = simt_shape(c, L);
    const int G = L.d.groups > 1 ? L.d.groups : 1;
    SimtArgs a;
    a.in = in; a.w = L.weight_simt; a.bias = L.bias; a.out = out;
    a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks; a.early = dc_lists_settled(c);
    a.Hi = L.in_h; a.Wi = L.in_w; a.Ci = L.d.cin; a.Ho = L.d.out_h; a.Wo = L.d.out_w; a.Co = L.d.cout; a.p = L.d.ph; a.relu = L.d.relu;
    a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.Cig = L.d.cin / G; a.Cog = L.d.cout / G; a.nb_g = dc_div_up(a.Cog, sh.BN); a.NB = G * a.nb_g; a.chunks = dc_div_up(a.Cig, sh.CI);
    a.vec = a.Ci % 4 == 0 && a.Cig % 4 == 0 && quads(c, in);
    dc_prof_scope ps(c, DC_ST_CONV);
    c->launches += 1;
    return c->cfg.dtype == DC_BF16 ? launch_simt_kw<__nv_bfloat16>(c, a, L.d.kw, sh, max_tiles) : launch_simt_kw<float>(c, a, L.d.kw, sh, max_tiles);
}

int dc_launch_dense(dc_cache* c, int layer, const void* in, void* out, const uint32_t* masks)
{
    dc_layer_rt& L = c->L[layer];
    DenseArgs a = {in, L.weight, L.bias, out, masks, c->S, L.d.cout, L.d.kh * L.d.kw * L.d.cin, L.d.relu, 0};
    a.vec = a.K % 4 == 0 && quads(c, in);
    const dim3 grid(dc_div_up(a.N, DN_N), dc_div_up(a.S, DN_S));
    dc_prof_scope ps(c, DC_ST_CONV);
    if (c->cfg.dtype == DC_BF16) DC_CUDA(dc_launch_pdl(k_dense<__nv_bfloat16>, grid, DN_WARPS * 32, 0, c->stream, a));
    else DC_CUDA(dc_launch_pdl(k_dense<float>, grid, DN_WARPS * 32, 0, c->stream, a));
    c->launches += 1;
    return DC_OK;
}

// The packed weights of a layer that runs on k_conv_simt (L.weight holds them as [cout][kh][kw][cin / groups]).
int dc_pack_weights_simt(dc_cache* c, int layer)
{
    dc_layer_rt& L = c->L[layer];
    if (!simt_ok(c, L.d) || dc_dense_ok(L)) return DC_OK;
    const SimtShape sh = simt_shape(c, L);
    const int G = L.d.groups > 1 ? L.d.groups : 1, cig = L.d.cin / G, cog = L.d.cout / G, taps = L.d.kh * L.d.kw;
    const int nb_g = dc_div_up(cog, sh.BN), chunks = dc_div_up(cig, sh.CI);
    const size_t floats = (size_t)G * nb_g * chunks * taps * sh.CI * sh.BN;
    DC_CUDA(cudaMalloc((void**)&L.weight_simt, floats * sizeof(float)));
    c->bytes += floats * sizeof(float);
    int grid = (int)((floats + 255) / 256); if (grid > c->num_sms * 8) grid = c->num_sms * 8;
    if (c->cfg.dtype == DC_BF16)
        k_pack_simt<__nv_bfloat16><<<grid, 256, 0, c->stream>>>((const __nv_bfloat16*)L.weight, taps, cig, cog, nb_g, G * nb_g, chunks, sh.CI, sh.BN, L.weight_simt);
    else
        k_pack_simt<float><<<grid, 256, 0, c->stream>>>((const float*)L.weight, taps, cig, cog, nb_g, G * nb_g, chunks, sh.CI, sh.BN, L.weight_simt);
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}
