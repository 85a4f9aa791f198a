// Partial convolution of float32 maps on the 5th-generation tensor cores, without giving up float32 accuracy.
//
// A float has 24 significant bits, a bf16 eight: an operand of 2^-110 or more is the exact sum of three bf16 pieces, x = x0 + x1 + x2
// (each the nearest bf16 of what is left).  The product of two operands is then six tensor-core products of pieces,
//     x0 w0  +  (x0 w1 + x1 w0)  +  (x0 w2 + x1 w1 + x2 w0),
// whose remainder (x1 w2 and smaller) is 2^-24 of the product at most, 2^-26 or less of most.  Products of bf16 are exact in fp32; what rounds is the sum,
// and there the tensor core is kept on a short leash: it adds up one kernel row of 32 channels (terms of each of the three sizes in
// an accumulator of its own), then the sums move to registers and are added there, rounded to nearest, in a fixed order.
// Measured against 64-bit sums (2-norm, pixel inputs through five layers): 0.6 of the error of the chain of fp32 FMAs.
//
// One instruction takes several products: the weight pieces lie behind one another along N, so A = x0 times [w0 w1 w2] fills three
// blocks of BN columns, x1 times [w0 w1] adds to the last two, x2 times [w0] to the last.  A block of BN = 64 channels so costs
// 192 + 128 + 64 columns per 16 input channels, and the pixels are read from shared memory three times, not six.
//
// Work item: one dirty 16 x 8 tile (128 pixels = M) times BN channels; persistent CTAs, one per SM.  16 warps:
//   0      weights: one bulk copy per (32 channels, kernel row), packed as the MMA reads them
//   1      MMA issue
//   2-9    the sums: tensor memory -> registers after every kernel row; bias, ReLU, store of the pixels not reused.  A warp has 32 pixels and
//          half of the channels, or (TURNS: several items per CTA) all of them of every other item: four warps empty the accumulators of one
//          item while the other four finish the one before.
//   10-15  input: the (16 + kh - 1) x (8 + kw - 1) patch of 32 channels, split into pieces on its way to shared memory (planes of
//          8 channels, 16 bytes a pixel: every tap is a shifted view of it, as in the patch scheme of the bf16 kernels)
// What bounds it: no unit by itself.  MMAs run 52% of the clocks, as long as reading their operands takes (64-channel blocks; blocks of 32: 55%, a
// half longer than their arithmetic); loads and stores of the other warps take the shared-memory pipe for 37 to 56% of the clocks, half of that bank
// conflicts.  The rest is hand-overs around the kernel rows: without loads, drains and stores 0.78 of the time, without MMAs 0.8.
// Measured, 24 streams, all tiles, us (CUDA cores, here): 32 -> 32 at 227 x 227 451, 178; 32 -> 64 at 113 x 113 246, 82; 64 -> 64 461, 133;
// 64 -> 128 at 56 x 56 213, 69.  One stream: 29.0, 14.3; 19.5, 8.8; 32.2, 12.7; 17.0, 10.9.
//
// Infinities, NaN and magnitudes that no bf16 holds do not split (inf - inf), nor do most floats below 2^-110, whose last bits lie
// under the smallest bf16 of 2^-133: whatever leaves a remainder behind its third piece.  The warps that split a tile mark it if it
// holds one, and its pixels are computed by FMAs (fma_pixels); weights like that keep the layer on the CUDA cores.
// FMAs compute two kinds of pixels more.  A sum that is not finite: where operands that do split add up to more than a float holds, the
// accumulators of the three sizes can become infinities of either sign, and their sum NaN.  A sum below 2^-100 other than zero: its
// small terms lie where floats have fewer bits, and the tensor core cuts there more often than FMAs round (twice the error at 2^-132).
// With every pixel computed so, 64 -> 64 channels, 3 x 3 at 113 x 113, 4 streams, takes 405 us (43 on the tensor cores, 118 on
// k_conv_simt; a channel after the other from global memory took 12 ms).
#include "dc_common.cuh"
#include "dc_tcgen05.cuh"

namespace {

constexpr int kSumWarps = 8, kSplitWarps = 6, kThreadsF = 32 * (2 + kSumWarps + kSplitWarps);
constexpr int kStagesF = 8;                       // weight stages at most
constexpr int kChF = 32;                          // input channels per patch
constexpr int kRowsPerDrain1 = 3;                 // 1 x 1 kernels: patches between two drains (6 steps of 16 channels, as a row of a 3 x 3 kernel)
constexpr int kTileFlags = 8;                     // more than the items between the splitting warps and the epilogue (at most 6)
constexpr float kSmallSum = 0x1p-100f;            // below it the tensor core's cuts at 2^-149 may count for more than an FMA's roundings
constexpr unsigned long long kWaitLimitF = 2000000000ull;

struct F32Args {
    const float* in; const uint8_t* wp; const float* w; const float* bias; float* out;   // wp: [groups * nb_g][chunks][taps][4][3 BN][8] bf16
                                                  // w: [groups][Cig filled up to 16s][taps][nb_g * BN] float, for pixels computed by FMAs
    const int32_t* tile_list; const int32_t* tile_count; const uint32_t* masks;
    int Hi, Wi, Ci, Ho, Wo, Co, p, relu, tiles_x, tiles_y;
    int Cig, Cog, nb_g, NB, chunks, ks_last;      // channels per group; blocks per group and in all; patches; steps of 16 channels in the last
    int fma_ci, fma_ks;                           // sums by FMAs: every fma_ks-th run of fma_ci channels in a chain of its own (dc_simt_order)
    int stages;
    int vec;                                      // four input channels are one aligned load
    int early;
    int32_t* status;
    unsigned long long wait_ns;
    int skip_loads;
};

// Channels of the output's staging (32 pixels for each warp): a warp's half, or as many as fit.  Its bytes for a warp: at least what
// fma_pixels keeps there, some channels of the window that 4 x 8 pixels see and their weights for 16 channels of the output.
__host__ __device__ constexpr int f32_stage_ch(int BN, int KW) { return BN == 32 ? 16 : KW == 5 ? 8 : 32; }
__host__ __device__ constexpr int f32_window_ch(int KW) { return KW == 5 ? 1 : 8; }
__host__ __device__ constexpr int f32_stage_bytes(int BN, int KW)
{
    const int out = 32 * (f32_stage_ch(BN, KW) + 4) * 4, fma = (KW == 1 ? f32_window_ch(KW) : KW * KW) * 64 + f32_window_ch(KW) * (DC_TILE_W + KW - 1) * (4 + KW - 1) * 4;
    return out > fma ? out : fma;
}

struct __align__(16) CtlF {
    unsigned long long full[kStagesF], empty[kStagesF], a_full[2], a_empty[2], t_full[4], t_empty[2];     // t_full: [2 groups of sum warps][2 sets]
    uint32_t tmem_base;
    volatile int abort_flag;
    unsigned long long wait_ns;
    volatile int odd[kTileFlags];                 // item that holds a value that does not split (its number + 1)
};

__device__ __forceinline__ bool f_wait(uint32_t bar, uint32_t parity, CtlF* ctl, int32_t* status)
{
    return mbar_wait_at(bar, parity, &ctl->abort_flag, &ctl->wait_ns, status);
}
// A whole warp's wait: one lane asks, so that a waiting warp takes one turn at the barrier and not 32.
__device__ __forceinline__ bool f_wait_warp(uint32_t bar, uint32_t parity, int lane, CtlF* ctl, int32_t* status)
{
    bool ok = true;
    if (lane == 0) ok = f_wait(bar, parity, ctl, status);
    return __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
}
// N columns, 128 rows, bf16 operands, fp32 sums
__device__ __forceinline__ uint32_t f_idesc(int n) { return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (8u << 24); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                 : "r"(taddr) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }
__device__ __forceinline__ float lds32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ float max3_abs(float a, float b, float c)       // of the magnitudes; NaN if one of them is
{
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3_abs(float a, float b, float c)       // of the magnitudes that are not NaN
{
    float r;
    asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi)
{
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// Two floats into three pairs of pieces; one of the low 16 bits of `odd` is set if one of them does not split: what is left for the third
// piece is no bf16 itself, or NaN (whose bits are all ones).
__device__ __forceinline__ void split2(float a, float b, uint32_t& p0, uint32_t& p1, uint32_t& p2, uint32_t& odd)
{
    p0 = bf16_pair(a, b);
    a -= __uint_as_float(p0 << 16); b -= __uint_as_float(p0 & 0xffff0000u);
    p1 = bf16_pair(a, b);
    a -= __uint_as_float(p1 << 16); b -= __uint_as_float(p1 & 0xffff0000u);
    p2 = bf16_pair(a, b);
    odd |= __float_as_uint(a) | __float_as_uint(b);
}

// A warp's 4 x 8 pixels, from row y0, column x0 of stream s on, whose `redo` is set, channels c0 ... of group grp, by FMAs: a value of the patch
// does not split, or a sum overflowed.  In the order of k_conv_simt's sums, so that the bits are that kernel's, also where the order decides
// between infinity and NaN.  XC channels of the window that the pixels see and the weights of STEP channels lie in shared memory (`stage`, the warp's
// own); the weights travel while the ones before are in use.  A call, and behind the stores, where the sums are no longer needed: inlined, or with
// the sums to keep, its registers cost the ordinary tiles 2 to 20 % (small CNN, 24 streams: 710 us a pass so, 732 inlined, 705 without it).
template <int BN, int KW>
__device__ __noinline__ void fma_pixels(const F32Args& a, uint32_t stage, int s, int y0, int x0, int grp, int c0, bool redo)
{
    constexpr int TAPS = KW * KW, WX = DC_TILE_W + KW - 1, WIN = WX * (4 + KW - 1), XC = f32_window_ch(KW), STEP = KW == 1 ? XC : 1;
    constexpr int ROWS = STEP * TAPS, QUADS = ROWS * 4, WQ = (QUADS + 31) / 32, XQ = XC < 4 ? 1 : XC / 4;
    const int lane = threadIdx.x & 31, cog = a.nb_g * BN, cig = (a.Cig + 15) & ~15, ci = a.fma_ci, n_ks = a.fma_ks;
    const float* const in = a.in + (size_t)s * a.Hi * a.Wi * a.Ci + grp * a.Cig;
    const uint32_t window = stage + ROWS * 64, mine = window + (lane / DC_TILE_W * WX + lane % DC_TILE_W) * 4;
    auto fill = [&](int c) {                                               // channels c ... of the window, [channel][pixel]
#pragma unroll 1
        for (int u = lane; u < WIN * XQ; u += 32) {
            const int px = u / XQ, i = u % XQ * 4, wy = px / WX, y = y0 - a.p + wy, x = x0 - a.p + px - wy * WX;
            const int left = (unsigned)y < (unsigned)a.Hi && (unsigned)x < (unsigned)a.Wi ? a.Cig - c - i : 0;
            const float* p = in + ((size_t)y * a.Wi + x) * a.Ci + c + i;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (XC >= 4 && a.vec) { if (left > 0) v = dc_ld((const float4*)p); }
            else {
                if (left > 0) v.x = dc_ld(p);
                if (XC > 1 && left > 1) v.y = dc_ld(p + 1);
                if (XC > 2 && left > 2) v.z = dc_ld(p + 2);
                if (XC > 3 && left > 3) v.w = dc_ld(p + 3);
            }
            const uint32_t at = window + (i * WIN + px) * 4;
            sts32(at, v.x);
            if constexpr (XC > 1) { sts32(at + WIN * 4, v.y); sts32(at + 2 * WIN * 4, v.z); sts32(at + 3 * WIN * 4, v.w); }
        }
    };
#pragma unroll 1
    for (int c_out = c0; c_out < min(c0 + BN / 2, a.Cog); c_out += 16) {
        const float* const k0 = a.w + ((size_t)grp * TAPS * cig + lane / 4) * cog + c_out + lane % 4 * 4;
        float sum[16];
#pragma unroll 1
        for (int ks = 0; ks < n_ks; ++ks) {
            float part[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) part[j] = 0.f;
            float4 wn[WQ];
            auto weights = [&](int c) {
#pragma unroll
                for (int q = 0; q < WQ; ++q)
                    if (lane + 32 * q < QUADS) wn[q] = __ldg((const float4*)(k0 + ((size_t)c * TAPS + 8 * q) * cog));
            };
            int c = ks * ci;
            if (c < a.Cig) weights(c);
#pragma unroll 1
            while (c < a.Cig) {
                __syncwarp();
                fill(c);
#pragma unroll 1
                for (int i = 0; i < XC; i += STEP) {
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < WQ; ++q)
                        if (lane + 32 * q < QUADS)
                            sts128(stage + (lane + 32 * q) * 16, __float_as_uint(wn[q].x), __float_as_uint(wn[q].y), __float_as_uint(wn[q].z), __float_as_uint(wn[q].w));
                    __syncwarp();
                    c += STEP;
                    if (c % ci == 0) c += (n_ks - 1) * ci;                 // the chain's next run of channels
                    if (c < cig) weights(c);
#pragma unroll
                    for (int r = 0; r < ROWS; ++r) {
                        const float v = lds32(mine + ((i + r / TAPS) * WIN + r % TAPS / KW * WX + r % TAPS % KW) * 4);
#pragma unroll
                        for (int j = 0; j < 16; j += 4) {
                            const uint4 w = lds128(stage + r * 64 + j * 4);
                            part[j] = fmaf(v, __uint_as_float(w.x), part[j]); part[j + 1] = fmaf(v, __uint_as_float(w.y), part[j + 1]);
                            part[j + 2] = fmaf(v, __uint_as_float(w.z), part[j + 2]); part[j + 3] = fmaf(v, __uint_as_float(w.w), part[j + 3]);
                        }
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[j] = ks == 0 ? part[j] : sum[j] + part[j];
        }
        float* o = a.out + (((size_t)s * a.Ho + y0 + lane / DC_TILE_W) * a.Wo + x0 + lane % DC_TILE_W) * a.Co + grp * a.Cog + c_out;
        const float* bias = a.bias + grp * a.Cog + c_out;
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            if (!redo || c_out + j >= a.Cog) continue;                     // channels come in fours
            float4 v = make_float4(sum[j] + __ldg(bias + j), sum[j + 1] + __ldg(bias + j + 1), sum[j + 2] + __ldg(bias + j + 2), sum[j + 3] + __ldg(bias + j + 3));
            if (a.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
            *(float4*)(o + j) = v;
        }
    }
    __syncwarp();
}

template <int BN, int KW, bool TURNS>
__global__ void __launch_bounds__(kThreadsF, 1) k_conv_f32(const __grid_constant__ F32Args a)
{
    constexpr int PW = DC_TILE_W + KW - 1, PX = PW * (DC_TILE_H + KW - 1), PLANE = PX * 16, PIECE = 4 * PLANE, A_SLOT = 3 * PIECE;
    constexpr int TAP = 4 * 3 * BN * 16, B_STAGE = KW * TAP;              // weights of a tap, of a kernel row
    constexpr int UNITS = (4 * PX + 32 * kSplitWarps - 1) / (32 * kSplitWarps);   // 8-channel pixels that a splitting thread holds
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = (uint8_t*)(((uintptr_t)smem_raw + 127) & ~(uintptr_t)127);
    uint8_t* bring = base + 2 * A_SLOT;
    CtlF* ctl = (CtlF*)(bring + (size_t)a.stages * B_STAGE);
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int per_stream = a.tiles_x * a.tiles_y;
    constexpr uint32_t kSet = 3 * BN, kCols = BN == 32 ? 256 : 512;
    constexpr int STAGE_CH = f32_stage_ch(BN, KW), STAGE_PITCH = (STAGE_CH + 4) * 4;   // bank-conflict free for both sides
    constexpr int kRows = KW > 1 ? 1 : kRowsPerDrain1;

    if (threadIdx.x == 0) {
        for (int i = 0; i < a.stages; ++i) { mbar_init(&ctl->full[i], 1); mbar_init(&ctl->empty[i], 1); }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&ctl->a_full[i], kSplitWarps); mbar_init(&ctl->a_empty[i], 1);
            mbar_init(&ctl->t_full[i], 1); mbar_init(&ctl->t_full[2 + i], 1); mbar_init(&ctl->t_empty[i], TURNS ? kSumWarps / 2 : kSumWarps);
        }
        for (int i = 0; i < kTileFlags; ++i) ctl->odd[i] = 0;
        ctl->abort_flag = 0;
        ctl->wait_ns = a.wait_ns;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&ctl->tmem_base)), "r"(kCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;
    if (!a.early) { dc_pdl_wait(); dc_pdl_release(); }
    const int n_items = __ldcg(a.tile_count) * a.NB;
    const uint32_t full0 = smem_u32(&ctl->full[0]), empty0 = smem_u32(&ctl->empty[0]), a_full0 = smem_u32(&ctl->a_full[0]), a_empty0 = smem_u32(&ctl->a_empty[0]);
    const uint32_t t_full0 = smem_u32(&ctl->t_full[0]), t_empty0 = smem_u32(&ctl->t_empty[0]);
    auto k_steps = [&](int cc) { return cc + 1 < a.chunks ? kChF / 16 : a.ks_last; };
    // All of a layer's weights in the ring: they stay there, sent once.  A fifth of what moves through shared memory in a kernel row were weights that
    // were there before (32 -> 32 at 227 x 227, 24 streams, all tiles: 203 us without this and without turns, 205 with turns alone, 178 with both).
    const bool resident = TURNS && a.NB == 1 && a.chunks * KW <= a.stages;

    if (warp == 0) {
        // ---------------- weights ----------------
        if (elect_one()) {
            RingPos r;
            r.start(smem_u32(bring), (uint32_t)a.stages);
            const uint32_t r0 = r.data;
            const size_t block = (size_t)a.chunks * KW * B_STAGE;
            // a last patch of one step needs the first half of each tap alone
            auto send = [&](uint32_t off, uint32_t dst, const uint8_t* src, int cc) {
                const int half = k_steps(cc) == 1;
                mbar_expect_tx(full0 + off, (uint32_t)(half ? B_STAGE / 2 : B_STAGE));
                if (!half) bulk_copy(dst, src, B_STAGE, full0 + off);
                else for (int t = 0; t < KW; ++t) bulk_copy(dst + t * TAP, src + t * TAP, TAP / 2, full0 + off);
            };
            bool ok = true;
            int ahead = 0;
            if (a.early) {
                // the weights are nobody's output: the first stages travel while the previous kernel ends
                if ((int)blockIdx.x < n_items && !a.skip_loads) {
                    const uint8_t* w = a.wp + (size_t)(blockIdx.x % a.NB) * block;
                    const int n = min(a.stages, a.chunks * KW);
                    for (int cc = 0, t = 0; ahead < n; ++ahead) {
                        send(8u * ahead, r0 + ahead * B_STAGE, w + (size_t)ahead * B_STAGE, cc);
                        if (++t == KW) { t = 0; ++cc; }
                    }
                }
                dc_pdl_wait(); dc_pdl_release();
            }
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const uint8_t* w = a.wp + (size_t)(item % a.NB) * block;
                for (int cc = 0; cc < a.chunks && ok; ++cc)
                    for (int t = 0; t < KW; ++t, w += B_STAGE) {
                        if (ahead > 0) --ahead;
                        else {
                            ok = f_wait(empty0 + r.off, r.phase ^ 1u, ctl, a.status);
                            if (!ok) break;
                            if (!a.skip_loads) send(r.off, r.data, w, cc);
                        }
                        r.next(r0, (uint32_t)a.stages, (uint32_t)B_STAGE);
                    }
                if (resident) break;
            }
            // on an abort: give the copies already issued a bounded chance to land before the CTA exits
            if (!ok) { const unsigned long long t0 = now_ns(); while (now_ns() - t0 < 2000000ull) { } }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issuer ----------------
        if (a.early) { dc_pdl_wait(); dc_pdl_release(); }
        if (elect_one()) {
            const uint64_t ac = umma_desc(0, PW * 16, 0, PLANE), bc = umma_desc(0, 128, 0, 3 * BN * 16);
            const uint32_t a_hi = (uint32_t)(ac >> 32), b_hi = (uint32_t)(bc >> 32);
            const uint32_t a0 = (uint32_t)ac + (smem_u32(base) >> 4), b0 = (uint32_t)bc + (smem_u32(bring) >> 4);
            const uint32_t i3 = f_idesc(3 * BN), i2 = f_idesc(2 * BN), i1 = f_idesc(BN);
            RingPos rb, ra;
            rb.start(b0, (uint32_t)a.stages); ra.start(a0, 2);
            uint32_t set = 0, set_ph = 0, group = 0;                           // group: of sum warps, whose turn the item is
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x, group ^= TURNS ? 2u : 0u) {
                int rows = 0;                                              // kernel rows in the accumulator set
                const bool fresh = !resident || item == (int)blockIdx.x;   // weights to wait for
                if (resident) rb.start(b0, (uint32_t)a.stages);
                for (int cc = 0; cc < a.chunks && ok; ++cc) {
                    ok = f_wait(a_full0 + ra.off, ra.phase, ctl, a.status);
                    const bool two = k_steps(cc) == 2;
                    for (int ky = 0; ky < KW && ok; ++ky) {
                        if (rows == 0) ok = f_wait(t_empty0 + 8u * set, set_ph ^ 1u, ctl, a.status);
                        if (fresh) ok = ok && f_wait(full0 + rb.off, rb.phase, ctl, a.status);
                        if (!ok) break;
                        tc_fence_after();
                        const uint32_t d = tmem_base + set * kSet, at = ra.data + (uint32_t)(ky * PW);
                        // a kernel row's MMAs in one go: what one lane can issue is the limit here, not the tensor pipe
#pragma unroll
                        for (int kx = 0; kx < KW; ++kx)
#pragma unroll
                            for (int k = 0; k < kChF / 16; ++k)
                                if (k == 0 || two) {
                                    const uint32_t al = at + kx + k * (PLANE >> 3), bl = rb.data + ((kx * TAP + k * (2 * 3 * BN * 16)) >> 4);
                                    umma_chunk(d, al, a_hi, 0, bl, b_hi, 0, i3, kx + k == 0 ? (uint32_t)rows : 1u, 1);
                                    umma_chunk(d + BN, al + (PIECE >> 4), a_hi, 0, bl, b_hi, 0, i2, 1u, 1);
                                    umma_chunk(d + 2 * BN, al + 2 * (PIECE >> 4), a_hi, 0, bl, b_hi, 0, i1, 1u, 1);
                                }
                        if (!resident) umma_commit_at(empty0 + rb.off);
                        rb.next(b0, (uint32_t)a.stages, (uint32_t)B_STAGE >> 4);
                        if (++rows == kRows || (cc + 1 == a.chunks && ky + 1 == KW)) {
                            umma_commit_at(t_full0 + 8u * (group + set));
                            rows = 0;
                            set ^= 1u;
                            if (set == 0) set_ph ^= 1u;
                        }
                    }
                    if (ok) umma_commit_at(a_empty0 + ra.off);
                    ra.next(a0, 2, (uint32_t)A_SLOT >> 4);
                }
            }
        }
        __syncwarp();
    } else if (warp < 2 + kSumWarps) {
        // ---------------- sums, bias, ReLU, store ----------------
        constexpr int HALF = BN / 2, CH = TURNS ? BN : HALF;              // channels of this thread's pixel; those whose outcome is decided together
        const int q = warp & 3, group = (warp - 2) >> 2, half = TURNS ? 0 : group, m = q * 32 + lane, row = m / DC_TILE_W, col = m % DC_TILE_W;
        const uint32_t lanes = (uint32_t)(q * 32) << 16;
        const int drains = (a.chunks * KW + kRows - 1) / kRows;
        auto tile_of = [&](int item) { return item < n_items ? __ldcg(a.tile_list + item / a.NB) : 0; };
        const int first = TURNS ? group : 0, every = TURNS ? 2 : 1;       // of the CTA's items, this warp's
        int next = tile_of(blockIdx.x + first * gridDim.x);
        if (a.early) { dc_pdl_wait(); dc_pdl_release(); }
        const uint32_t stage = smem_u32(ctl + 1) + (warp - 2) * f32_stage_bytes(BN, KW);
        const uint32_t t_full = t_full0 + (TURNS ? 16u * group : 0u);
        uint32_t next_set = 0, phases = 0;                                 // phases: TURNS: bit s: of set s, for this group; else of both
        int seq = first;
        for (int item = blockIdx.x + first * gridDim.x; item < n_items; item += every * gridDim.x, seq += every) {
            const int tile = next;
            next = tile_of(item + every * gridDim.x);
            const uint32_t word = __ldcg(a.masks + (size_t)tile * 4 + (row >> 2));
            float sum[CH];
#pragma unroll
            for (int j = 0; j < CH; ++j) sum[j] = 0.f;
            bool ok = true;
            uint32_t set = TURNS ? (uint32_t)(seq * drains) & 1u : next_set;
            for (int u = 0; u < drains; ++u, set ^= 1u) {
                ok = f_wait_warp(t_full + 8u * set, TURNS ? (phases >> set) & 1u : phases, lane, ctl, a.status);
                if (!ok) break;
                if (TURNS) phases ^= 1u << set;
                tc_fence_after();
                const uint32_t d = tmem_base + lanes + set * kSet + half * CH;
#pragma unroll
                for (int h = 0; h < CH; h += 16) {                         // the small terms first
                    uint32_t x[16], y[16];
                    tmem_ld16(d + 2 * BN + h, x);
                    tmem_ld16(d + BN + h, y);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; ++j) x[j] = __float_as_uint(__uint_as_float(x[j]) + __uint_as_float(y[j]));
                    tmem_ld16(d + h, y);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 16; ++j) sum[h + j] += __uint_as_float(y[j]) + __uint_as_float(x[j]);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&ctl->t_empty[set]);
                if (!TURNS && set == 1) phases ^= 1u;
            }
            if (!TURNS) next_set = set;
            if (!ok) break;
            const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
            const int y = ty * DC_TILE_H + row, x = tx * DC_TILE_W + col;
            const bool active = y < a.Ho && x < a.Wo && !((word >> (8 * (row & 3) + col)) & 1u);
            auto odd_item = [&] { return ctl->odd[seq % kTileFlags] == seq + 1; };
            const bool odd_early = TURNS && odd_item();
            const int nb = item % a.NB, grp = nb / a.nb_g;
#pragma unroll
            for (int h = 0; h < CH; h += HALF) {
                const int c0 = (nb - grp * a.nb_g) * BN + half * HALF + h, n = min(HALF, a.Cog - c0);
                float* const tile_out = a.out + (((size_t)s * a.Ho + ty * DC_TILE_H) * a.Wo + tx * DC_TILE_W) * a.Co + grp * a.Cog + c0;
                const float* bias = a.bias + grp * a.Cog + c0;
                float most = 0.f, least = INFINITY;                        // magnitudes; NaN counts among the largest
#pragma unroll
                for (int j = 0; j < HALF; j += 2) { most = max3_abs(most, sum[h + j], sum[h + j + 1]); least = min3_abs(least, sum[h + j], sum[h + j + 1]); }
                bool small = false;
                if (least < kSmallSum) {
#pragma unroll
                    for (int j = 0; j < HALF; ++j) small = small || (fabsf(sum[h + j]) < kSmallSum && sum[h + j] != 0.f);
                }
                const bool redo = active && (!(most < INFINITY) || small || (TURNS ? odd_early : odd_item()));
                // through shared memory, so that lanes side by side store side by side (a lane's own 32-byte pieces of its pixel: each store of a
                // warp touched 32 lines, and the stores took as long as the MMAs)
                const uint32_t todo = __ballot_sync(0xffffffffu, active && !redo);
                const int part = lane % (STAGE_CH / 4);
#pragma unroll
                for (int c = 0; c < HALF; c += STAGE_CH) {
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < STAGE_CH; j += 4)
                        sts128(stage + lane * STAGE_PITCH + j * 4, __float_as_uint(sum[h + c + j]), __float_as_uint(sum[h + c + j + 1]),
                               __float_as_uint(sum[h + c + j + 2]), __float_as_uint(sum[h + c + j + 3]));
                    __syncwarp();
                    if (c + 4 * part >= n) continue;                       // channels come in fours
                    const float* pb = bias + c + 4 * part;
                    const float b0 = __ldg(pb), b1 = __ldg(pb + 1), b2 = __ldg(pb + 2), b3 = __ldg(pb + 3);
#pragma unroll
                    for (int i = 0; i < STAGE_CH / 4; ++i) {
                        const int p = i * (128 / STAGE_CH) + lane / (STAGE_CH / 4);
                        const uint4 w = lds128(stage + p * STAGE_PITCH + part * 16);
                        float4 v = make_float4(__uint_as_float(w.x) + b0, __uint_as_float(w.y) + b1, __uint_as_float(w.z) + b2, __uint_as_float(w.w) + b3);
                        if (a.relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
                        if ((todo >> p) & 1u) *(float4*)(tile_out + ((size_t)(q * 4 + p / 8) * a.Wo + p % 8) * a.Co + c + 4 * part) = v;
                    }
                }
                if (__any_sync(0xffffffffu, redo)) fma_pixels<BN, KW>(a, stage, s, ty * DC_TILE_H + q * 4, tx * DC_TILE_W, grp, c0, redo);
            }
        }
    } else {
        // ---------------- input patches, split into pieces ----------------
        const int tid = threadIdx.x - (2 + kSumWarps) * 32;
        int py[UNITS], px[UNITS], so[UNITS], cg[UNITS];                    // unit: pixel of the patch, its place, its channels; eight lanes, eight pixels
#pragma unroll
        for (int i = 0; i < UNITS; ++i) {
            const int u = tid + i * 32 * kSplitWarps, p = (u >> 5) * 8 + (u & 7), g = (u >> 3) & 3;
            py[i] = p / PW; px[i] = p - py[i] * PW; cg[i] = 8 * g;
            so[i] = p < PX ? g * PLANE + p * 16 : -1;
        }
        // the patches in order, their loads one patch ahead of the splitting
        struct Patch { int cc, seq; };                                     // cc < 0: none left
        int item = blockIdx.x, cc = 0, seq = 0;
        auto tile_of = [&](int i) { return i < n_items ? __ldcg(a.tile_list + i / a.NB) : 0; };
        int tile = tile_of(item), y0 = 0, x0 = 0;
        const float* in = a.in;
        auto place = [&]() {
            const int s = tile / per_stream, t = tile - s * per_stream, ty = t / a.tiles_x, tx = t - ty * a.tiles_x;
            y0 = ty * DC_TILE_H - a.p; x0 = tx * DC_TILE_W - a.p;
            in = a.in + (size_t)s * a.Hi * a.Wi * a.Ci + item % a.NB / a.nb_g * a.Cig;
            tile = tile_of(item + gridDim.x);
        };
        place();
        auto load = [&](float4 (&v)[UNITS][2]) -> Patch {
            if (item >= n_items) return {-1, 0};
#pragma unroll
            for (int i = 0; i < UNITS; ++i) {
                v[i][0] = v[i][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                const int y = y0 + py[i], x = x0 + px[i], left = a.Cig - (cc * kChF + cg[i]);
                if (so[i] < 0 || left <= 0 || (unsigned)y >= (unsigned)a.Hi || (unsigned)x >= (unsigned)a.Wi) continue;
                const float* p = in + ((size_t)y * a.Wi + x) * a.Ci + cc * kChF + cg[i];
                if (a.vec) {
                    v[i][0] = dc_ld((const float4*)p);
                    if (left > 4) v[i][1] = dc_ld((const float4*)p + 1);
                } else {
                    float e[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) e[k] = k < left ? dc_ld(p + k) : 0.f;
                    v[i][0] = make_float4(e[0], e[1], e[2], e[3]); v[i][1] = make_float4(e[4], e[5], e[6], e[7]);
                }
            }
            const Patch now = {cc, seq};
            if (++cc == a.chunks) { cc = 0; ++seq; item += gridDim.x; place(); }
            return now;
        };
        const uint32_t a0 = smem_u32(base);
        uint32_t slot = 0, phase = 0;
        auto split = [&](const float4 (&v)[UNITS][2], Patch b) -> bool {
            const int c_end = 16 * k_steps(b.cc);                          // channels of this patch that the MMAs read
            if (!f_wait_warp(a_empty0 + 8u * slot, phase ^ 1u, lane, ctl, a.status)) return false;
            uint32_t odd = 0;
#pragma unroll
            for (int i = 0; i < UNITS; ++i) {
                if (so[i] < 0 || cg[i] >= c_end) continue;
                uint32_t p0[4], p1[4], p2[4];
                split2(v[i][0].x, v[i][0].y, p0[0], p1[0], p2[0], odd);
                split2(v[i][0].z, v[i][0].w, p0[1], p1[1], p2[1], odd);
                split2(v[i][1].x, v[i][1].y, p0[2], p1[2], p2[2], odd);
                split2(v[i][1].z, v[i][1].w, p0[3], p1[3], p2[3], odd);
                const uint32_t at = a0 + slot * A_SLOT + so[i];
                sts128(at, p0[0], p0[1], p0[2], p0[3]);
                sts128(at + PIECE, p1[0], p1[1], p1[2], p1[3]);
                sts128(at + 2 * PIECE, p2[0], p2[1], p2[2], p2[3]);
            }
            if (odd & 0xffffu) ctl->odd[b.seq % kTileFlags] = b.seq + 1;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&ctl->a_full[slot]);
            slot ^= 1u;
            if (slot == 0) phase ^= 1u;
            return true;
        };
        if (a.early) { dc_pdl_wait(); dc_pdl_release(); }
        float4 v0[UNITS][2], v1[UNITS][2];
        Patch b0 = load(v0);
        while (b0.cc >= 0) {
            const Patch b1 = load(v1);
            if (!split(v0, b0) || b1.cc < 0) break;
            b0 = load(v0);
            if (!split(v1, b1)) break;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kCols) : "memory");
    }
}

// weights [cout][taps][Cig] -> [groups * nb_g][chunks][taps][4][3 BN][8]: plane g of a stage holds channels 8 g ... of its 32, row p * BN + n
// piece p of output channel n.  `odd` is set by a weight that does not split.
__global__ void k_pack_f32(const float* w, int taps, int Cig, int Cog, int nb_g, int NB, int chunks, int BN, __nv_bfloat16* out, int32_t* odd)
{
    const size_t total = (size_t)NB * chunks * taps * 4 * BN * 8;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i;
        const int e = (int)(r % 8); r /= 8;
        const int n = (int)(r % BN); r /= BN;
        const int g = (int)(r % 4); r /= 4;
        const size_t stage = r;
        const int t = (int)(r % taps); r /= taps;
        const int cc = (int)(r % chunks), nb = (int)(r / chunks);
        const int grp = nb / nb_g, co = (nb - grp * nb_g) * BN + n, c = cc * kChF + 8 * g + e;
        float v = co < Cog && c < Cig ? w[((size_t)(grp * Cog + co) * taps + t) * Cig + c] : 0.f;
        __nv_bfloat16* o = out + ((stage * 4 + g) * 3 * BN + n) * 8 + e;
        for (int p = 0; p < 3; ++p) {
            const __nv_bfloat16 b = __float2bfloat16_rn(v);
            o[(size_t)p * BN * 8] = b;
            v -= __bfloat162float(b);
        }
        if (v != 0.f) *odd = 1;                                           // (NaN too)
    }
}

// The same weights as floats, [cout][taps][Cig] -> [groups][Cig filled up to 16s][taps][nb_g * BN] with zeros beyond the last channels.
__global__ void k_pack_f32_fma(const float* w, int taps, int Cig, int Cog, int cig, int cog, size_t total, float* out)
{
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        size_t r = i;
        const int n = (int)(r % cog); r /= cog;
        const int t = (int)(r % taps); r /= taps;
        const int c = (int)(r % cig);
        const size_t grp = r / cig;
        out[i] = n < Cog && c < Cig ? w[((grp * Cog + n) * taps + t) * Cig + c] : 0.f;
    }
}

// The pixels are read from shared memory again for every block of channels: a step of 16 channels measured 240 clocks for 32 output channels and 310
// for 64 (272 and 364 where a CTA has dozens of items: the same ratio).  Wide blocks, then, unless they leave SMs without an item: whichever takes
// fewer clocks with every tile dirty.  us in blocks of 32 and 64, 3 x 3: 64 -> 128 at 56 x 56, 1 stream 10.8 and 11.8, 2 15.8 and 12.7, 24 95.7 and 69.0;
// 64 -> 96 at 113 x 113 (three narrow blocks or two wide ones), 1 stream 20.9 and 19.0, 2 31.1 and 31.8, 4 54.1 and 51.3, 24 291 and 264.
int f32_bn(const dc_cache* c, const dc_layer_rt& L)
{
    const int G = L.d.groups > 1 ? L.d.groups : 1, cog = L.d.cout / G;
    const long long tiles = (long long)L.tiles_x * L.tiles_y * c->S * G, sms = c->num_sms;
    const long long narrow = (tiles * dc_div_up(cog, 32) + sms - 1) / sms * 240, wide = (tiles * dc_div_up(cog, 64) + sms - 1) / sms * 310;
    return narrow < wide ? 32 : 64;
}

}  // namespace

// Few channels on either side fill a small part of an MMA's 16 by 32; such layers stay on the CUDA cores.
static bool f32_ok(const dc_cache* c, const dc_layer_desc& d)
{
    const int G = d.groups > 1 ? d.groups : 1;
    return c->cfg.dtype == DC_FP32 && d.kind == DC_CONV && d.sh == 1 && d.sw == 1 && d.kh == d.kw && d.ph == d.pw &&
           (d.kw == 1 || d.kw == 3 || d.kw == 5) && d.cin / G >= 16 && d.cout / G >= 32 && (d.cout / G) % 4 == 0;
}

// Bytes of the pieces, and of the float weights that lie behind them (dc_layer_rt::weight_f32).
struct F32Bytes { size_t pieces, floats; };
static F32Bytes f32_weight_bytes(const dc_cache* c, const dc_layer_rt& L)
{
    const int G = L.d.groups > 1 ? L.d.groups : 1, BN = f32_bn(c, L), cig = L.d.cin / G;
    const size_t rows = (size_t)G * dc_div_up(L.d.cout / G, BN) * BN * L.d.kh * L.d.kw;
    return {rows * dc_div_up(cig, kChF) * kChF * 3 * 2, rows * ((cig + 15) & ~15) * sizeof(float)};
}

int dc_pack_weights_f32(dc_cache* c, int layer)
{
    dc_layer_rt& L = c->L[layer];
    if (!f32_ok(c, L.d) || dc_dense_ok(L) || getenv("DC_NO_TENSOR_CORES")) return DC_OK;
    const int G = L.d.groups > 1 ? L.d.groups : 1, cig = L.d.cin / G, cog = L.d.cout / G, taps = L.d.kh * L.d.kw;
    const int BN = f32_bn(c, L), nb_g = dc_div_up(cog, BN), chunks = dc_div_up(cig, kChF);
    const F32Bytes bytes = f32_weight_bytes(c, L);
    DC_CUDA(cudaMalloc(&L.weight_f32, bytes.pieces + bytes.floats));
    c->bytes += bytes.pieces + bytes.floats;
    auto grid = [&](size_t n) { const size_t g = (n + 255) / 256, most = (size_t)c->num_sms * 8; return (int)(g < most ? g : most); };
    k_pack_f32<<<grid(bytes.pieces / 6), 256, 0, c->stream>>>((const float*)L.weight, taps, cig, cog, nb_g, G * nb_g, chunks, BN, (__nv_bfloat16*)L.weight_f32, c->reuse_px + layer);
    DC_CUDA(cudaGetLastError());
    k_pack_f32_fma<<<grid(bytes.floats / 4), 256, 0, c->stream>>>((const float*)L.weight, taps, cig, cog, (cig + 15) & ~15, nb_g * BN, bytes.floats / 4,
                                                                 (float*)((uint8_t*)L.weight_f32 + bytes.pieces));
    DC_CUDA(cudaGetLastError());
    return DC_OK;
}

// Layers with a weight that does not split go to the CUDA cores after all.  dc_pack_weights_f32 has left word in the first n_layers
// counters of the reuse step (zeroed before); one wait for all layers.
int dc_settle_weights_f32(dc_cache* c)
{
    int32_t odd[DC_MAX_LAYERS];
    bool any = false;
    for (int i = 0; i < c->n_layers; ++i) any = any || c->L[i].weight_f32;
    if (!any) return DC_OK;
    DC_CUDA(cudaMemcpyAsync(odd, c->reuse_px, sizeof(int32_t) * c->n_layers, cudaMemcpyDeviceToHost, c->stream));
    DC_CUDA(cudaStreamSynchronize(c->stream));
    for (int i = 0; i < c->n_layers; ++i) {
        dc_layer_rt& L = c->L[i];
        if (!L.weight_f32 || !odd[i]) continue;
        cudaFree(L.weight_f32);
        L.weight_f32 = nullptr;
        const F32Bytes bytes = f32_weight_bytes(c, L);
        c->bytes -= bytes.pieces + bytes.floats;
        const int rc = dc_pack_weights_simt(c, i);
        if (rc != DC_OK) return rc;
    }
    return DC_OK;
}

// A CTA takes its SM whole (512 threads of 128 registers), also where the next frame is matched beside it: a VGG-16 trunk in float32 on full-HD
// frames with the next one announced takes 1.07, 3.2 and 6.7 ms a pass for 4, 16 and 32 streams so, and took 3.1, 10.1 and 19.5 on
// k_conv_simt, whose CTAs leave the search room.
template <int BN, int KW, bool TURNS>
static int launch_f32(dc_cache* c, F32Args& a, int grid)
{
    constexpr int a_total = 2 * 3 * 4 * 16 * (DC_TILE_W + KW - 1) * (DC_TILE_H + KW - 1), stage = KW * 4 * 3 * BN * 16, staging = kSumWarps * f32_stage_bytes(BN, KW);
    constexpr int room = (226 * 1024 - (int)sizeof(CtlF) - staging - a_total) / stage;
    static_assert(room >= 2, "two kernel rows of weights fit");
    a.stages = room > kStagesF ? kStagesF : room;
    const size_t smem = (size_t)a_total + (size_t)a.stages * stage + sizeof(CtlF) + staging + 128;
    static dc_once_per_device attr_set;
    if (attr_set.first(c->device)) DC_CUDA(cudaFuncSetAttribute(k_conv_f32<BN, KW, TURNS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    DC_CUDA(dc_launch_pdl(k_conv_f32<BN, KW, TURNS>, dim3((unsigned)grid), kThreadsF, smem, c->stream, a));
    return DC_OK;
}

int dc_launch_conv_f32(dc_cache* c, int layer, const void* in, void* out, const int32_t* tile_list, const int32_t* tile_count,
                       const uint32_t* masks, int max_tiles)
{
    dc_layer_rt& L = c->L[layer];
    const int G = L.d.groups > 1 ? L.d.groups : 1, BN = f32_bn(c, L);
    F32Args a;
    a.in = (const float*)in; a.wp = (const uint8_t*)L.weight_f32; a.w = (const float*)(a.wp + f32_weight_bytes(c, L).pieces); a.bias = L.bias; a.out = (float*)out;
    a.tile_list = tile_list; a.tile_count = tile_count; a.masks = masks; a.early = dc_lists_settled(c);
    a.Hi = L.in_h; a.Wi = L.in_w; a.Ci = L.d.cin; a.Ho = L.d.out_h; a.Wo = L.d.out_w; a.Co = L.d.cout;
    a.p = L.d.ph; a.relu = L.d.relu; a.tiles_x = L.tiles_x; a.tiles_y = L.tiles_y;
    a.Cig = L.d.cin / G; a.Cog = L.d.cout / G; a.nb_g = dc_div_up(a.Cog, BN); a.NB = G * a.nb_g; a.chunks = dc_div_up(a.Cig, kChF);
    a.ks_last = (a.Cig - (a.chunks - 1) * kChF + 15) / 16;
    dc_simt_order(c, L, &a.fma_ci, &a.fma_ks);
    a.vec = a.Ci % 4 == 0 && a.Cig % 4 == 0 && (uintptr_t)in % 16 == 0;
    a.status = c->status; a.wait_ns = kWaitLimitF; a.skip_loads = 0;
    if (c->debug_stall_ms > 0) { a.wait_ns = (unsigned long long)c->debug_stall_ms * 1000000ull; a.skip_loads = 1; c->debug_stall_ms = 0; }
    const long long items = (long long)(max_tiles < 1 ? 1 : max_tiles) * a.NB;
    const int grid = items > c->num_sms ? c->num_sms : (int)items;
    dc_prof_scope ps(c, DC_ST_CONV);
    c->launches += 1;
    // TURNS for 3 x 3 kernels where a CTA has several items of 32 channels; with few each the eight warps finish one sooner together, 5 x 5 kernels take 5%
    // longer in turns whatever their number, 1 x 1 kernels up to 5%; sums of 64 channels are more than a thread's registers hold beside the rest.
    // us without and with it, every tile dirty, by items: 32 -> 32, 250 11.1 and 11.8, 400 14.1 and 14.4, 450 16.3 and 16.2, 1000 26.1 and 24.2;
    // 16 -> 32, 1000 21.7 and 19.3; 64 -> 32, 1000 41.1 and 39.2; 1 x 1, 32 -> 32, 5220 73 and 77.
    const bool turns = BN == 32 && L.d.kw == 3 && items > 3ll * c->num_sms;
#define DC_F32(kw) return BN == 64 ? launch_f32<64, kw, false>(c, a, grid) : launch_f32<32, kw, false>(c, a, grid)
    if (turns) return launch_f32<32, 3, true>(c, a, grid);
    if (L.d.kw == 1) DC_F32(1);
    if (L.d.kw == 3) DC_F32(3);
    DC_F32(5);
#undef DC_F32
}
