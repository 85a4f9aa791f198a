// Layers that are computed in full every frame (Section 5: only convolutions are cached):
// frame -> network input, area resize, max pooling, residual add, ReLU.  All are bandwidth
// bound: one pass over input and output.
#include "dc_common.cuh"

namespace {

template <typename T> __device__ __forceinline__ float to_f(T v);
template <> __device__ __forceinline__ float to_f<float>(float v) { return v; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Round a double to bfloat16, nearest even: first to a float that keeps a trace of what was cut off in its last bit
// (round to odd), so that the second rounding sees on which side of a tie the value lay.
__device__ __forceinline__ __nv_bfloat16 double_to_bf16(double v)
{
    float f = __double2float_rz(v);
    if ((double)f != v) f = __uint_as_float(__float_as_uint(f) | 1u);
    return __float2bfloat16_rn(f);
}
template <typename T> __device__ __forceinline__ T from_d(double v);
template <> __device__ __forceinline__ float from_d<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_d<__nv_bfloat16>(double v) { return double_to_bf16(v); }

// pixel / 255 in the map's type.  bfloat16: the product with the float nearest to 1/255, rounded, is the correctly
// rounded quotient for all 256 values; float: the division.
template <typename T> __device__ __forceinline__ T from_pixel(uint32_t v);
template <> __device__ __forceinline__ float from_pixel<float>(uint32_t v) { return __fdiv_rn((float)v, 255.f); }
template <> __device__ __forceinline__ __nv_bfloat16 from_pixel<__nv_bfloat16>(uint32_t v) { return __float2bfloat16_rn((float)v * (1.f / 255.f)); }

// Frame copy (rows 16-byte aligned) -> network input map: four values per thread, one aligned word of the row.
template <typename T>
__global__ void __launch_bounds__(256) k_input_map(const uint8_t* frame, size_t pitch, int row_elems, int words, unsigned total, T* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned row = i / (unsigned)words, w = i - row * (unsigned)words;
        const uint32_t v = dc_ld((const uint32_t*)(frame + (size_t)row * pitch) + w);
        T* o = out + (size_t)row * row_elems + 4 * w;
#pragma unroll
        for (int k = 0; k < 4; ++k) if ((int)(4 * w) + k < row_elems) o[k] = from_pixel<T>((v >> (8 * k)) & 0xffu);
    }
}

// Frame copy -> the first convolution's operand copies, without the input map in between (bfloat16 caches whose input
// map nobody else reads).  k_frame_pad8: [S][H][W][8], three channels and five zeros, one pixel per thread.
__global__ void __launch_bounds__(256) k_frame_pad8(const uint8_t* frame, size_t pitch, int W, unsigned total, uint4* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned row = i / (unsigned)W, x = i - row * (unsigned)W;
        const uint32_t* q = (const uint32_t*)(frame + (size_t)row * pitch) + (3 * x >> 2);
        const uint32_t v = __funnelshift_r(dc_ld(q), dc_ld(q + 1), (3 * x & 3) * 8);    // the copy's rows have spare bytes
        const __nv_bfloat162 rg = __halves2bfloat162(from_pixel<__nv_bfloat16>(v & 0xffu), from_pixel<__nv_bfloat16>((v >> 8) & 0xffu));
        const __nv_bfloat162 b0 = __halves2bfloat162(from_pixel<__nv_bfloat16>((v >> 16) & 0xffu), __float2bfloat16_rn(0.f));
        out[i] = make_uint4(*(const uint32_t*)&rg, *(const uint32_t*)&b0, 0u, 0u);
    }
}
// k_frame_s2d: the space-to-depth block map of dc_conv_s2d.cu.  Element e of a block pixel is byte e % (3 s) of the block's
// row e / (3 s): within a block row the bytes are consecutive in the frame.  One thread per 8 elements, which come from at
// most two rows of the frame (3 s >= 6 and 8 elements start at an even byte of a six-byte row), a CTA per 128 of a row of blocks.
// What bounds it: the instructions per element; aligned words in place of single bytes, and rows dealt to CTAs in place of
// three divisions per thread; then the writes.  96 frames of 227 x 227, blocks of 4: 27 -> 18 us; 128 of 224 x 224,
// blocks of 2: 35 -> 23.
__device__ __forceinline__ unsigned long long fetch_bytes8(const uint8_t* row, int byte, int row_bytes)   // zeros outside the row
{
    const int from = byte > 0 ? byte : 0, left = row_bytes - from;
    if (left <= 0 || byte <= -8) return 0;
    const uint32_t* q = (const uint32_t*)row + (from >> 2);           // the copy's rows have spare bytes
    const uint32_t w0 = dc_ld(q), w1 = dc_ld(q + 1), w2 = dc_ld(q + 2);
    const int sh = (from & 3) * 8;
    unsigned long long v = (unsigned long long)__funnelshift_r(w1, w2, sh) << 32 | __funnelshift_r(w0, w1, sh);
    if (left < 8) v &= (1ull << (8 * left)) - 1ull;
    return byte < 0 ? v << (-8 * byte) : v;
}
__global__ void __launch_bounds__(128) k_frame_s2d(const uint8_t* frame, size_t pitch, int W, int H, int bs, int Py, int Px, int Hs, int Ws, int chunks,
                                                   int rows, uint4* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int rb = 3 * bs, per_row = Ws * chunks, i = blockIdx.y * 128 + threadIdx.x;   // the thread's place in a row of blocks
    if (i >= per_row) return;
    const int bx = i / chunks, ch = i - bx * chunks;
    const int dy = 8 * ch / rb, b = 8 * ch - dy * rb, n1 = min(8, rb - b), x_byte = (bx * bs - Px) * 3;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int st = r / Hs, iy = (r - st * Hs) * bs - Py + dy;
        const uint8_t* src = frame + (size_t)st * H * pitch;
        unsigned long long v = 0;
        if (dy < bs && iy >= 0 && iy < H) v = fetch_bytes8(src + (size_t)iy * pitch, x_byte + b, 3 * W);
        if (n1 < 8) {
            v &= (1ull << (8 * n1)) - 1ull;
            if (dy + 1 < bs && iy + 1 >= 0 && iy + 1 < H) v |= fetch_bytes8(src + (size_t)(iy + 1) * pitch, x_byte, 3 * W) << (8 * n1);
        }
        uint32_t o[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t w = (uint32_t)(v >> (16 * k));
            const __nv_bfloat162 e = __halves2bfloat162(from_pixel<__nv_bfloat16>(w & 0xffu), from_pixel<__nv_bfloat16>((w >> 8) & 0xffu));
            o[k] = *(const uint32_t*)&e;
        }
        out[(size_t)r * per_row + i] = make_uint4(o[0], o[1], o[2], o[3]);
    }
}

// Box average of the frame: output (oy, ox) is the mean over rows [floor(oy H / Ho),
// ceil((oy + 1) H / Ho) - 1] and the like columns, divided by 255.  One CTA per output row:
// pass 1 sums the span's source rows column-wise with coalesced 16-byte loads (row starts are
// 16-byte aligned in the library's frame copy), six rows in flight, into shared memory; pass 2 sums each output
// pixel's column span.  All sums are integers; the one division is done in double.  pad8 (or NULL): the pixel once more with
// its channels padded to eight, for the few-channel convolution that follows.
template <typename T>
__global__ void __launch_bounds__(256) k_resize_area(const uint8_t* frame, size_t pitch, int W, int H, int S,
                                                     int Wo, int Ho, T* out, uint4* pad8)
{
    extern __shared__ uint16_t colsum[];                       // [ceil16(W * 3)]
    dc_pdl_wait();
    dc_pdl_release();
    const int oy = blockIdx.x % Ho, s = blockIdx.x / Ho;
    const int y0 = (int)((long long)oy * H / Ho), y1 = (int)(((long long)(oy + 1) * H + Ho - 1) / Ho) - 1;
    const int row_bytes = W * 3, chunks = (row_bytes + 15) >> 4, rows = y1 - y0 + 1;
    const uint8_t* base = frame + ((size_t)s * H + y0) * pitch;
    for (int c = threadIdx.x; c < chunks; c += blockDim.x) {
        uint32_t acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};            // 16 byte columns as 8 pairs of 16-bit sums
        for (int yb = 0; yb < rows; yb += 6) {
            uint4 v[6];
#pragma unroll
            for (int k = 0; k < 6; ++k) v[k] = yb + k < rows ? dc_ld((const uint4*)(base + (size_t)(yb + k) * pitch + c * 16)) : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    acc[2 * j] += __byte_perm(w[j], 0, 0x4140);    // bytes 0, 1 -> two 16-bit lanes
                    acc[2 * j + 1] += __byte_perm(w[j], 0, 0x4342);
                }
            }
        }
        uint4* dst = (uint4*)(colsum + c * 16);
        dst[0] = make_uint4(acc[0], acc[1], acc[2], acc[3]);
        dst[1] = make_uint4(acc[4], acc[5], acc[6], acc[7]);
    }
    __syncthreads();
    for (int ox = threadIdx.x; ox < Wo; ox += blockDim.x) {
        const int x0 = (int)((long long)ox * W / Wo), x1 = (int)(((long long)(ox + 1) * W + Wo - 1) / Wo) - 1;
        uint32_t sum[3] = {0, 0, 0};
        for (int x = x0; x <= x1; ++x) { sum[0] += colsum[x * 3]; sum[1] += colsum[x * 3 + 1]; sum[2] += colsum[x * 3 + 2]; }
        const double div = (double)(rows * (x1 - x0 + 1)) * 255.0;
        const size_t px = ((size_t)s * Ho + oy) * Wo + ox;
        T v[3];
#pragma unroll
        for (int ch = 0; ch < 3; ++ch) { v[ch] = from_d<T>((double)sum[ch] / div); out[px * 3 + ch] = v[ch]; }
        if constexpr (sizeof(T) == 2) {
            if (pad8) {
                const __nv_bfloat162 rg = __halves2bfloat162(v[0], v[1]), b0 = __halves2bfloat162(v[2], __float2bfloat16_rn(0.f));
                pad8[px] = make_uint4(*(const uint32_t*)&rg, *(const uint32_t*)&b0, 0u, 0u);
            }
        }
    }
}

// 8 (bf16) or 4 (float) channels per thread with 16-byte loads; C must be a multiple of that.
template <typename T> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    static __device__ __forceinline__ uint4 vmax(uint4 a, uint4 b)
    {
        return make_uint4(__float_as_uint(fmaxf(__uint_as_float(a.x), __uint_as_float(b.x))),
                          __float_as_uint(fmaxf(__uint_as_float(a.y), __uint_as_float(b.y))),
                          __float_as_uint(fmaxf(__uint_as_float(a.z), __uint_as_float(b.z))),
                          __float_as_uint(fmaxf(__uint_as_float(a.w), __uint_as_float(b.w))));
    }
};
template <> struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    static __device__ __forceinline__ uint32_t m2(uint32_t a, uint32_t b)
    {
        __nv_bfloat162 r = __hmax2(*reinterpret_cast<__nv_bfloat162*>(&a), *reinterpret_cast<__nv_bfloat162*>(&b));
        return *reinterpret_cast<uint32_t*>(&r);
    }
    static __device__ __forceinline__ uint4 vmax(uint4 a, uint4 b) { return make_uint4(m2(a.x, b.x), m2(a.y, b.y), m2(a.z, b.z), m2(a.w, b.w)); }
};

// masks (optional): the layer's per-tile reuse bitmaps; a pixel whose bit is set was filled from the cache.
// also: the caller's copy of the network's last map, or NULL (here and in the kernels below).
// K x K windows with K known: the loads of an output vector are independent and travel together (a tap
// outside the map is moved to the nearest row and column inside, whose tap is in the window too: the maximum is the same).  K = 0: any window, tap after tap.
template <typename T, int K>
__global__ void __launch_bounds__(256) k_maxpool_vec(const uint4* in, int Hi, int Wi, unsigned cv, dc_layer_desc L, unsigned total, uint4* out, uint4* also, const uint32_t* masks,
                                                     int tiles_x, int tiles_y)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned t = i / cv, c = i - t * cv, u = t / (unsigned)L.out_w;
        const int ox = (int)(t - u * (unsigned)L.out_w);
        const unsigned s = u / (unsigned)L.out_h;
        const int oy = (int)(u - s * (unsigned)L.out_h);
        if (masks) {
            const size_t tile = ((size_t)s * tiles_y + oy / DC_TILE_H) * tiles_x + ox / DC_TILE_W;
            const int bit = DC_TILE_BIT(oy % DC_TILE_H, ox % DC_TILE_W);
            if ((masks[tile * 4 + (bit >> 5)] >> (bit & 31)) & 1u) continue;
        }
        const int y0 = oy * L.sh - L.ph, x0 = ox * L.sw - L.pw;
        const uint4* base = in + (size_t)s * Hi * Wi * cv + c;
        uint4 m;
        if constexpr (K > 0) {
            uint4 v[K * K];
#pragma unroll
            for (int k = 0; k < K * K; ++k) {
                const int y = min(max(y0 + k / K, max(y0, 0)), Hi - 1), x = min(max(x0 + k % K, max(x0, 0)), Wi - 1);
                v[k] = dc_ld(base + ((size_t)y * Wi + x) * cv);
            }
            m = v[0];
#pragma unroll
            for (int k = 1; k < K * K; ++k) m = Vec16<T>::vmax(m, v[k]);
        } else {
            bool first = true;
            m = make_uint4(0, 0, 0, 0);
            for (int ky = 0; ky < L.kh; ++ky) {
                const int iy = y0 + ky;
                if (iy < 0 || iy >= Hi) continue;
                for (int kx = 0; kx < L.kw; ++kx) {
                    const int ix = x0 + kx;
                    if (ix < 0 || ix >= Wi) continue;
                    const uint4 v = dc_ld(base + ((size_t)iy * Wi + ix) * cv);
                    m = first ? v : Vec16<T>::vmax(m, v);
                    first = false;
                }
            }
        }
        out[i] = m;
        if (also) also[i] = m;
    }
}

// 2 x 2 windows at stride 2 without padding (every window inside the map), no reuse bitmap: the four 16-byte
// loads of an output vector are independent and issued together; 32-bit index arithmetic.
template <typename T>
__global__ void k_maxpool2x2_vec(const uint4* in, int Hi, int Wi, int cv, int out_h, int out_w, unsigned total, uint4* out, uint4* also)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned c = i % cv, t = i / cv, ox = t % out_w, u = t / out_w, oy = u % out_h, s = u / out_h;
        const uint4* p = in + (((size_t)s * Hi + 2 * oy) * Wi + 2 * ox) * cv + c;
        const size_t row = (size_t)Wi * cv;
        const uint4 v00 = dc_ld(p), v01 = dc_ld(p + cv), v10 = dc_ld(p + row), v11 = dc_ld(p + row + cv);
        const uint4 m = Vec16<T>::vmax(Vec16<T>::vmax(v00, v01), Vec16<T>::vmax(v10, v11));
        out[i] = m;
        if (also) also[i] = m;
    }
}

template <typename T>
__global__ void k_maxpool(const T* in, int Hi, int Wi, int C, int S, dc_layer_desc L, T* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    const size_t total = (size_t)S * L.out_h * L.out_w * C;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        int c = (int)(i % C); size_t t = i / C;
        int ox = (int)(t % L.out_w); t /= L.out_w;
        int oy = (int)(t % L.out_h); int s = (int)(t / L.out_h);
        float m = -INFINITY;
        for (int ky = 0; ky < L.kh; ++ky) {
            int iy = oy * L.sh - L.ph + ky;
            if (iy < 0 || iy >= Hi) continue;
            for (int kx = 0; kx < L.kw; ++kx) {
                int ix = ox * L.sw - L.pw + kx;
                if (ix < 0 || ix >= Wi) continue;
                m = fmaxf(m, to_f(in[(((size_t)s * Hi + iy) * Wi + ix) * C + c]));
            }
        }
        out[i] = from_f<T>(m);
    }
}

template <typename T>
__global__ void k_add(const T* a, const T* b, size_t n, int relu, T* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        float v = to_f(a[i]) + to_f(b[i]);
        if (relu) v = fmaxf(v, 0.f);
        out[i] = from_f<T>(v);
    }
}

template <typename T>
__global__ void k_relu(const T* a, size_t n, T* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        out[i] = from_f<T>(fmaxf(to_f(a[i]), 0.f));
}

// 16-byte vectors: element-wise add (+ ReLU) and ReLU are pure HBM traffic, one vector per thread and pass
template <typename T> struct VecOps;
template <> struct VecOps<float> {
    static __device__ __forceinline__ uint4 add(uint4 a, uint4 b, int relu)
    {
        float r[4] = {__uint_as_float(a.x) + __uint_as_float(b.x), __uint_as_float(a.y) + __uint_as_float(b.y),
                      __uint_as_float(a.z) + __uint_as_float(b.z), __uint_as_float(a.w) + __uint_as_float(b.w)};
        if (relu) { for (int i = 0; i < 4; ++i) r[i] = fmaxf(r[i], 0.f); }
        return make_uint4(__float_as_uint(r[0]), __float_as_uint(r[1]), __float_as_uint(r[2]), __float_as_uint(r[3]));
    }
};
template <> struct VecOps<__nv_bfloat16> {
    static __device__ __forceinline__ uint32_t add2(uint32_t a, uint32_t b, int relu)
    {
        const float2 fa = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&a));
        const float2 fb = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&b));
        float x = fa.x + fb.x, y = fa.y + fb.y;                   // fp32 sum, one rounding to bf16 (as the scalar kernel)
        if (relu) { x = fmaxf(x, 0.f); y = fmaxf(y, 0.f); }
        __nv_bfloat162 r = __floats2bfloat162_rn(x, y);
        return *reinterpret_cast<uint32_t*>(&r);
    }
    static __device__ __forceinline__ uint4 add(uint4 a, uint4 b, int relu)
    {
        return make_uint4(add2(a.x, b.x, relu), add2(a.y, b.y, relu), add2(a.z, b.z, relu), add2(a.w, b.w, relu));
    }
};

// out = a + b (+ ReLU); with b == nullptr: out = ReLU(a) (a + 0 is exact)
// Bound by memory.  It walks from the end: what the convolution before it wrote last is still in L2, and the convolution
// after it starts on what this kernel wrote last.  Its operands are not read again in this frame (streaming loads), so
// they do not push those lines out.  ResNet-50 trunk, 128 streams: 3230 -> 3130 us for the whole pass.
template <typename T>
__global__ void k_add_vec(const uint4* a, const uint4* b, size_t nvec, int relu, uint4* out, uint4* also)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nvec; i += (size_t)gridDim.x * blockDim.x) {
        const size_t k = nvec - 1 - i;
        const uint4 va = __ldcs(a + k), vb = b ? __ldcs(b + k) : make_uint4(0, 0, 0, 0);
        const uint4 v = VecOps<T>::add(va, vb, relu);
        out[k] = v;
        if (also) also[k] = v;
    }
}

// Local response normalisation inside each channel over a (2 r + 1)^2 window; pixels outside the map count as zero
// and the divisor stays n^2 at the borders.  One thread per output element; sums in float.
template <typename T>
__global__ void k_lrn(const T* in, int H, int W, int C, int S, int r, float alpha_n2, float beta, float kappa, T* out,
                      const uint32_t* masks, int tiles_x, int tiles_y)
{
    dc_pdl_wait();
    dc_pdl_release();
    const size_t total = (size_t)S * H * W * C;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C); size_t t = i / C;
        const int x = (int)(t % W); t /= W;
        const int y = (int)(t % H); const int s = (int)(t / H);
        if (masks) {                                             // pixel filled from the cache
            const size_t tile = ((size_t)s * tiles_y + y / DC_TILE_H) * tiles_x + x / DC_TILE_W;
            const int bit = DC_TILE_BIT(y % DC_TILE_H, x % DC_TILE_W);
            if ((masks[tile * 4 + (bit >> 5)] >> (bit & 31)) & 1u) continue;
        }
        float sum = 0.f;
        for (int dy = -r; dy <= r; ++dy) {
            const int yy = y + dy;
            if (yy < 0 || yy >= H) continue;
            for (int dx = -r; dx <= r; ++dx) {
                const int xx = x + dx;
                if (xx < 0 || xx >= W) continue;
                const float v = to_f(in[(((size_t)s * H + yy) * W + xx) * C + c]);
                sum += v * v;
            }
        }
        out[i] = from_f<T>(to_f(in[i]) * powf(kappa + alpha_n2 * sum, -beta));
    }
}

// The same for 16-byte vectors of channels, R known.  A thread takes Y rows of one column, so that the squares of a row are
// summed along x once for all the outputs above and below it, and beta = 3/4 (the default) takes two reciprocal square
// roots (inverse_3_4); sums and Newton steps two floats to an instruction.  What bounds it: the loads of a strip, all in flight at once, then
// some 150 instructions per vector; four CTAs per SM hide the one behind the other (R = 2: two, whose registers hold its loads).
// us with a thread per output, two rounded square roots and a division; one float to an instruction; and so (16 streams):
//   32 channels at 128 x 160, R = 1           43, 23, 20.6
//   64 channels at 32 x 40, R = 2 (Y = 1)     14, 9.5, 8.6
template <typename T> struct Unpack;
template <> struct Unpack<float> {
    static __device__ __forceinline__ void get(uint4 v, float* f) { f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w); }
    static __device__ __forceinline__ uint4 put(const float* f) { return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3])); }
};
template <> struct Unpack<__nv_bfloat16> {
    static __device__ __forceinline__ void get(uint4 v, float* f)
    {
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) { f[2 * k] = __uint_as_float(w[k] << 16); f[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u); }
    }
    static __device__ __forceinline__ uint4 put(const float* f)
    {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { const __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * k], f[2 * k + 1]); w[k] = *(const uint32_t*)&p; }
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// Two floats at a time (one instruction, each rounded as on its own).
#define DC_PAIR_OP(name, op)                                                                                                              \
    __device__ __forceinline__ float2 name(float2 a, float2 b)                                                                            \
    {                                                                                                                                     \
        float2 r;                                                                                                                         \
        asm("{\n\t.reg .b64 x, y, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t" op ".rn.f32x2 w, x, y;\n\tmov.b64 {%0, %1}, w;\n\t}" \
            : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                                              \
        return r;                                                                                                                         \
    }
DC_PAIR_OP(add2, "add")
DC_PAIR_OP(mul2, "mul")
#undef DC_PAIR_OP
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 r;
    asm("{\n\t.reg .b64 x, y, z, w;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\tfma.rn.f32x2 w, x, y, z;\n\tmov.b64 {%0, %1}, w;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return r;
}
__device__ __forceinline__ float2 pair_of(float v) { return make_float2(v, v); }
__device__ __forceinline__ float min3_nan(float a, float b, float c) { float r; asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }
__device__ __forceinline__ float max3_nan(float a, float b, float c) { float r; asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }

// d^(-3/4): d^(-1/2) and then (d^(1/2))^(-1/2), each with one Newton step (relative error up to 1.5 * 2^-23 together; up to
// 1.9 with the two rounded square roots and the division that they replace).
__device__ __forceinline__ float2 rsqrt_step(float2 d)
{
    const float2 y = make_float2(rsqrtf(d.x), rsqrtf(d.y)), e = fma2(mul2(make_float2(-d.x, -d.y), y), y, pair_of(1.f));
    return fma2(mul2(pair_of(0.5f), y), e, y);
}
__device__ __forceinline__ float2 inverse_3_4(float2 d)
{
    const float2 y = rsqrt_step(d);
    return mul2(y, rsqrt_step(mul2(d, y)));
}

template <typename T, int R, int Y>
__global__ void __launch_bounds__(256, R == 1 ? 4 : 2) k_lrn_vec(const uint4* in, int H, int W, unsigned cv, float alpha_n2, float beta, float kappa, unsigned strips, unsigned total, uint4* out,
                                                 const uint32_t* masks, int tiles_x, int tiles_y)
{
    constexpr int N = Vec16<T>::N;
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned t = i / cv, c = i - t * cv, u = t / (unsigned)W, s = u / strips;
        const int x = (int)(t - u * (unsigned)W), y0 = (int)(u - s * strips) * Y;
        uint32_t todo = 0;                                       // rows to write: inside the map and not filled from the cache
#pragma unroll
        for (int k = 0; k < Y; ++k)
            if (y0 + k < H) todo |= 1u << k;
        if (masks) {
            const size_t col = (size_t)s * tiles_y * tiles_x + x / DC_TILE_W;
#pragma unroll
            for (int k = 0; k < Y; ++k) {
                const int y = min(y0 + k, H - 1), bit = DC_TILE_BIT(y % DC_TILE_H, x % DC_TILE_W);
                if ((masks[(col + (size_t)(y / DC_TILE_H) * tiles_x) * 4 + (bit >> 5)] >> (bit & 31)) & 1u) todo &= ~(1u << k);
            }
        }
        if (todo == 0) continue;
        const size_t at = ((size_t)s * H + y0) * W + x;
        const uint4* base = in + at * cv + c;
        float2 sum[Y][N / 2];
#pragma unroll
        for (int k = 0; k < Y; ++k)
#pragma unroll
            for (int j = 0; j < N / 2; ++j) sum[k][j] = pair_of(0.f);
        uint4 v[Y + 2 * R][2 * R + 1], mid[Y];                   // the strip's input: all loads at once
#pragma unroll
        for (int r = 0; r < Y + 2 * R; ++r)
#pragma unroll
            for (int dx = 0; dx <= 2 * R; ++dx) {
                const bool in_map = y0 + r - R >= 0 && y0 + r - R < H && x + dx - R >= 0 && x + dx - R < W;
                v[r][dx] = in_map ? dc_ld(base + ((ptrdiff_t)(r - R) * W + (dx - R)) * cv) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
        for (int r = 0; r < Y + 2 * R; ++r) {
            float2 row[N / 2];
#pragma unroll
            for (int j = 0; j < N / 2; ++j) row[j] = pair_of(0.f);
#pragma unroll
            for (int dx = 0; dx <= 2 * R; ++dx) {
                float f[N];
                Unpack<T>::get(v[r][dx], f);
#pragma unroll
                for (int j = 0; j < N / 2; ++j) { const float2 g = make_float2(f[2 * j], f[2 * j + 1]); row[j] = fma2(g, g, row[j]); }
            }
            if (r >= R && r < Y + R) mid[r - R] = v[r][R];
#pragma unroll
            for (int k = 0; k < Y; ++k)
                if (r - R - k >= -R && r - R - k <= R) {
#pragma unroll
                    for (int j = 0; j < N / 2; ++j) sum[k][j] = add2(sum[k][j], row[j]);
                }
        }
#pragma unroll
        for (int k = 0; k < Y; ++k) {
            if (!((todo >> k) & 1u)) continue;
            float f[N];
            Unpack<T>::get(mid[k], f);
            float least = INFINITY, most = -INFINITY;                // NaN if one is
#pragma unroll
            for (int j = 0; j < N / 2; ++j) {
                sum[k][j] = fma2(pair_of(alpha_n2), sum[k][j], pair_of(kappa));
                least = min3_nan(least, sum[k][j].x, sum[k][j].y); most = max3_nan(most, sum[k][j].x, sum[k][j].y);
            }
            if (beta == 0.75f && least > 1e-30f && most < 1e30f) {
#pragma unroll
                for (int j = 0; j < N / 2; ++j) {
                    const float2 o = mul2(make_float2(f[2 * j], f[2 * j + 1]), inverse_3_4(sum[k][j]));
                    f[2 * j] = o.x; f[2 * j + 1] = o.y;
                }
            } else {
#pragma unroll
                for (int j = 0; j < N / 2; ++j) { f[2 * j] *= powf(sum[k][j].x, -beta); f[2 * j + 1] *= powf(sum[k][j].y, -beta); }
            }
            out[(at + (size_t)k * W) * cv + c] = Unpack<T>::put(f);
        }
    }
}

// Channel concatenation of two NHWC maps
template <typename T>
__global__ void k_concat(const T* a, int Ca, const T* b, int Cb, size_t pixels, T* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int C = Ca + Cb;
    const size_t total = pixels * C;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const int c = (int)(i % C); const size_t px = i / C;
        out[i] = c < Ca ? a[px * Ca + c] : b[px * Cb + (c - Ca)];
    }
}
// The same where both inputs' pixels are whole 16-byte vectors.
__global__ void __launch_bounds__(256) k_concat_vec(const uint4* a, unsigned va, const uint4* b, unsigned vb, unsigned total, uint4* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
        const unsigned px = i / (va + vb), c = i - px * (va + vb);
        out[i] = c < va ? dc_ld(a + (size_t)px * va + c) : dc_ld(b + (size_t)px * vb + (c - va));
    }
}

// Plain copy of a map
__global__ void __launch_bounds__(256) k_copy_vec(const uint4* a, unsigned total, uint4* out)
{
    dc_pdl_wait();
    dc_pdl_release();
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) out[i] = dc_ld(a + i);
}

inline int grid_for(const dc_cache* c, size_t n, int block)
{
    const size_t g = (n + block - 1) / block, cap = (size_t)c->num_sms * 16;
    return (int)(g > cap ? cap : (g ? g : 1));
}

}  // namespace

#define DISPATCH(c, expr_f32, expr_bf16) do { if ((c)->cfg.dtype == DC_BF16) { expr_bf16; } else { expr_f32; } } while (0)

// The vector kernels index with 32 bits: a launch takes at most c->piece items (2^31 - 1), and a larger map several launches, cut
// between `units` (rows or streams) of `each` items.  units_per_piece: 0 when a single unit is too large.
static size_t units_per_piece(const dc_cache* c, size_t each) { return c->piece / (each ? each : 1); }

int dc_launch_input_map(dc_cache* c, const uint8_t* frame, size_t pitch)
{
    const int row = c->cfg.width * 3, words = (row + 3) / 4;
    const size_t rows = (size_t)c->S * c->cfg.height, per = units_per_piece(c, words);
    if (per == 0) return DC_ERR_CONFIG;                          // one row of 8 GB
    dc_prof_scope ps(c, DC_ST_INPUT);
    for (size_t r = 0; r < rows; r += per) {
        const size_t n = (rows - r < per ? rows - r : per) * words;
        const dim3 grid((unsigned)grid_for(c, n, 256));
        DISPATCH(c,
            DC_CUDA(dc_launch_pdl(k_input_map<float>, grid, 256, 0, c->stream, frame + r * pitch, pitch, row, words, (unsigned)n, (float*)c->input_map + r * row)),
            DC_CUDA(dc_launch_pdl(k_input_map<__nv_bfloat16>, grid, 256, 0, c->stream, frame + r * pitch, pitch, row, words, (unsigned)n, (__nv_bfloat16*)c->input_map + r * row)));
        c->launches += 1;
    }
    return DC_OK;
}

// The frame straight into the operand copy of convolution `layer` (dc_conv_takes_frame).
int dc_launch_frame_operand(dc_cache* c, int layer, const uint8_t* frame, size_t pitch)
{
    dc_layer_rt& L = c->L[layer];
    dc_prof_scope ps(c, DC_ST_INPUT);
    if (L.s2d_s) {
        const int chunks = L.s2d_cs / 8;
        const int rows = c->S * L.in_h, parts = dc_div_up(L.s2d_ws * chunks, 128), most = dc_div_up(c->num_sms * 16, parts);
        DC_CUDA(dc_launch_pdl(k_frame_s2d, dim3((unsigned)(rows < most ? rows : most), (unsigned)parts), 128, 0, c->stream, frame, pitch, L.s2d_wi, L.s2d_hi, L.s2d_s, L.s2d_py, L.s2d_px, L.in_h, L.s2d_ws,
                              chunks, rows, (uint4*)L.in_s2d));
        c->launches += 1;
    } else {
        const size_t rows = (size_t)c->S * L.in_h, per = units_per_piece(c, L.in_w);
        if (per == 0) return DC_ERR_CONFIG;
        for (size_t r = 0; r < rows; r += per) {
            const size_t n = (rows - r < per ? rows - r : per) * L.in_w;
            DC_CUDA(dc_launch_pdl(k_frame_pad8, dim3((unsigned)grid_for(c, n, 256)), 256, 0, c->stream, frame + r * pitch, pitch, L.in_w, (unsigned)n,
                                  (uint4*)L.in_padded + r * L.in_w));
            c->launches += 1;
        }
    }
    return DC_OK;
}

int dc_launch_resize(dc_cache* c, int layer, const uint8_t* frame, size_t pitch)
{
    dc_layer_rt& L = c->L[layer];
    const dim3 grid((unsigned)(c->S * L.d.out_h));
    const size_t smem = (size_t)((c->cfg.width * 3 + 15) / 16) * 16 * sizeof(uint16_t);
    if (smem > 48 * 1024 || (size_t)c->cfg.height > 255u * (size_t)L.d.out_h) return DC_ERR_CONFIG;   // 16-bit column sums
    // the operand copy of the convolution that reads this resized frame (a table may hold resizes to other sizes too)
    uint4* pad8 = c->resize_feeds >= 0 && c->L[c->resize_feeds].d.in0 == layer ? (uint4*)c->L[c->resize_feeds].in_padded : nullptr;
    dc_prof_scope ps(c, DC_ST_INPUT);
    DISPATCH(c,
        DC_CUDA(dc_launch_pdl(k_resize_area<float>, grid, 256, smem, c->stream, frame, pitch, c->cfg.width, c->cfg.height, c->S, L.d.out_w, L.d.out_h, (float*)L.map[0], (uint4*)nullptr)),
        DC_CUDA(dc_launch_pdl(k_resize_area<__nv_bfloat16>, grid, 256, smem, c->stream, frame, pitch, c->cfg.width, c->cfg.height, c->S, L.d.out_w, L.d.out_h, (__nv_bfloat16*)L.map[0], pad8)));
    c->launches += 1;
    return DC_OK;
}

int dc_launch_maxpool(dc_cache* c, int layer, const void* in, void* out, const uint32_t* masks, void* also)
{
    dc_layer_rt& L = c->L[layer];
    const size_t n = (size_t)c->S * L.d.out_h * L.d.out_w * L.d.cout;
    const bool vec = (L.d.cout * c->elt) % 16 == 0;
    const int cv = L.d.cout * c->elt / 16;
    const size_t out1 = (size_t)L.d.out_h * L.d.out_w * cv, in1 = (size_t)L.in_h * L.in_w * cv, per = vec ? units_per_piece(c, out1) : 0;   // of one stream
    dc_prof_scope ps(c, DC_ST_POINTWISE);
    for (size_t s0 = 0; per > 0; s0 += per) {
        const size_t nv = ((size_t)c->S - s0 < per ? (size_t)c->S - s0 : per) * out1;
        const uint4* from = (const uint4*)in + s0 * in1;
        uint4 *to = (uint4*)out + s0 * out1, *to2 = also ? (uint4*)also + s0 * out1 : nullptr;
        const uint32_t* bits = masks ? masks + s0 * L.tiles_x * L.tiles_y * 4 : nullptr;
        const dim3 grid((unsigned)grid_for(c, nv, 256));
        if (!masks && L.d.kh == 2 && L.d.kw == 2 && L.d.sh == 2 && L.d.sw == 2 && L.d.ph == 0 && L.d.pw == 0 && 2 * L.d.out_h <= L.in_h && 2 * L.d.out_w <= L.in_w) {
            DISPATCH(c,
                DC_CUDA(dc_launch_pdl(k_maxpool2x2_vec<float>, grid, 256, 0, c->stream, from, L.in_h, L.in_w, cv, L.d.out_h, L.d.out_w, (unsigned)nv, to, to2)),
                DC_CUDA(dc_launch_pdl(k_maxpool2x2_vec<__nv_bfloat16>, grid, 256, 0, c->stream, from, L.in_h, L.in_w, cv, L.d.out_h, L.d.out_w, (unsigned)nv, to, to2)));
        } else {
#define DC_POOL(T, K) DC_CUDA(dc_launch_pdl(k_maxpool_vec<T, K>, grid, 256, 0, c->stream, from, L.in_h, L.in_w, (unsigned)cv, L.d, (unsigned)nv, to, to2, bits, L.tiles_x, L.tiles_y))
            if (L.d.kh == 3 && L.d.kw == 3) DISPATCH(c, DC_POOL(float, 3), DC_POOL(__nv_bfloat16, 3));
            else if (L.d.kh == 2 && L.d.kw == 2) DISPATCH(c, DC_POOL(float, 2), DC_POOL(__nv_bfloat16, 2));
            else DISPATCH(c, DC_POOL(float, 0), DC_POOL(__nv_bfloat16, 0));
#undef DC_POOL
        }
        c->launches += 1;
        if (s0 + per >= (size_t)c->S) return DC_OK;
    }
    c->launches += 1;
    if (masks) return DC_ERR_STATE;                             // cached pooling needs 16-byte pixels (checked at creation)
    const dim3 grid((unsigned)grid_for(c, n, 256));
    DISPATCH(c,
        DC_CUDA(dc_launch_pdl(k_maxpool<float>, grid, 256, 0, c->stream, (const float*)in, L.in_h, L.in_w, L.d.cout, c->S, L.d, (float*)out)),
        DC_CUDA(dc_launch_pdl(k_maxpool<__nv_bfloat16>, grid, 256, 0, c->stream, (const __nv_bfloat16*)in, L.in_h, L.in_w, L.d.cout, c->S, L.d, (__nv_bfloat16*)out)));
    return DC_OK;
}

int dc_launch_add(dc_cache* c, int layer, const void* a, const void* b, void* also)
{
    dc_layer_rt& L = c->L[layer];
    const size_t n = (size_t)c->S * L.d.out_h * L.d.out_w * L.d.cout;
    dc_prof_scope ps(c, DC_ST_POINTWISE);
    c->launches += 1;
    if ((n * c->elt) % 16 == 0) {                                 // maps come from cudaMalloc: 256-byte aligned
        const size_t nv = n * c->elt / 16;
        const dim3 grid((unsigned)grid_for(c, nv, 256));
        DISPATCH(c,
            DC_CUDA(dc_launch_pdl(k_add_vec<float>, grid, 256, 0, c->stream, (const uint4*)a, (const uint4*)b, nv, L.d.relu, (uint4*)L.map[0], (uint4*)also)),
            DC_CUDA(dc_launch_pdl(k_add_vec<__nv_bfloat16>, grid, 256, 0, c->stream, (const uint4*)a, (const uint4*)b, nv, L.d.relu, (uint4*)L.map[0], (uint4*)also)));
    } else {
        const dim3 grid((unsigned)grid_for(c, n, 256));
        DISPATCH(c,
            DC_CUDA(dc_launch_pdl(k_add<float>, grid, 256, 0, c->stream, (const float*)a, (const float*)b, n, L.d.relu, (float*)L.map[0])),
            DC_CUDA(dc_launch_pdl(k_add<__nv_bfloat16>, grid, 256, 0, c->stream, (const __nv_bfloat16*)a, (const __nv_bfloat16*)b, n, L.d.relu, (__nv_bfloat16*)L.map[0])));
    }
    return DC_OK;
}

int dc_launch_relu(dc_cache* c, int layer, const void* a)
{
    dc_layer_rt& L = c->L[layer];
    const size_t n = (size_t)c->S * L.d.out_h * L.d.out_w * L.d.cout;
    dc_prof_scope ps(c, DC_ST_POINTWISE);
    c->launches += 1;
    if ((n * c->elt) % 16 == 0) {
        const size_t nv = n * c->elt / 16;
        const dim3 grid((unsigned)grid_for(c, nv, 256));
        DISPATCH(c,
            DC_CUDA(dc_launch_pdl(k_add_vec<float>, grid, 256, 0, c->stream, (const uint4*)a, (const uint4*)nullptr, nv, 1, (uint4*)L.map[0], (uint4*)nullptr)),
            DC_CUDA(dc_launch_pdl(k_add_vec<__nv_bfloat16>, grid, 256, 0, c->stream, (const uint4*)a, (const uint4*)nullptr, nv, 1, (uint4*)L.map[0], (uint4*)nullptr)));
    } else {
        const dim3 grid((unsigned)grid_for(c, n, 256));
        DISPATCH(c,
            DC_CUDA(dc_launch_pdl(k_relu<float>, grid, 256, 0, c->stream, (const float*)a, n, (float*)L.map[0])),
            DC_CUDA(dc_launch_pdl(k_relu<__nv_bfloat16>, grid, 256, 0, c->stream, (const __nv_bfloat16*)a, n, (__nv_bfloat16*)L.map[0])));
    }
    return DC_OK;
}

int dc_launch_lrn(dc_cache* c, int layer, const void* in, void* out, const uint32_t* masks)
{
    dc_layer_rt& L = c->L[layer];
    const size_t n = (size_t)c->S * L.d.out_h * L.d.out_w * L.d.cout;
    const int r = L.d.ph, win = 2 * r + 1;
    const bool defaults = c->cfg.lrn_alpha == 0.0 && c->cfg.lrn_beta == 0.0 && c->cfg.lrn_k == 0.0;
    const float alpha = (float)(defaults ? 1e-4 : c->cfg.lrn_alpha), beta = (float)(defaults ? 0.75 : c->cfg.lrn_beta);
    const float kappa = (float)(defaults ? 1.0 : c->cfg.lrn_k), an = alpha / (win * win);
    dc_prof_scope ps(c, DC_ST_POINTWISE);
    const unsigned cv = (unsigned)(L.d.cout * c->elt / 16);
    const size_t each = (size_t)L.d.out_h * L.d.out_w * cv;                  // of one stream
    const size_t per = (L.d.cout * c->elt) % 16 == 0 && (r == 1 || r == 2) ? units_per_piece(c, each) : 0;
    for (size_t s0 = 0; per > 0; s0 += per) {
        const size_t streams = (size_t)c->S - s0 < per ? (size_t)c->S - s0 : per;
        // strips of two rows where they leave a wave of threads
        const int Y = streams * each >= (size_t)c->num_sms * 2048 * 2 ? 2 : 1;
        const unsigned strips = (unsigned)dc_div_up(L.d.out_h, Y);
        const size_t nv = streams * strips * L.d.out_w * cv;
        const dim3 grid((unsigned)grid_for(c, nv, 256));
        const uint32_t* bits = masks ? masks + s0 * L.tiles_x * L.tiles_y * 4 : nullptr;
#define DC_LRN_VEC(T, R, Y) DC_CUDA(dc_launch_pdl(k_lrn_vec<T, R, Y>, grid, 256, 0, c->stream, (const uint4*)in + s0 * each, L.d.out_h, L.d.out_w, cv, an, beta, kappa, strips, (unsigned)nv, (uint4*)out + s0 * each, bits, L.tiles_x, L.tiles_y))
        if (r == 1 && Y == 2) DISPATCH(c, DC_LRN_VEC(float, 1, 2), DC_LRN_VEC(__nv_bfloat16, 1, 2));
        else if (r == 1) DISPATCH(c, DC_LRN_VEC(float, 1, 1), DC_LRN_VEC(__nv_bfloat16, 1, 1));
        else if (Y == 2) DISPATCH(c, DC_LRN_VEC(float, 2, 2), DC_LRN_VEC(__nv_bfloat16, 2, 2));
        else DISPATCH(c, DC_LRN_VEC(float, 2, 1), DC_LRN_VEC(__nv_bfloat16, 2, 1));
#undef DC_LRN_VEC
        c->launches += 1;
        if (s0 + per >= (size_t)c->S) return DC_OK;
    }
    c->launches += 1;
    const dim3 grid((unsigned)grid_for(c, n, 256));
    DISPATCH(c,
        DC_CUDA(dc_launch_pdl(k_lrn<float>, grid, 256, 0, c->stream, (const float*)in, L.d.out_h, L.d.out_w, L.d.cout, c->S, r, an, beta, kappa, (float*)out, masks, L.tiles_x, L.tiles_y)),
        DC_CUDA(dc_launch_pdl(k_lrn<__nv_bfloat16>, grid, 256, 0, c->stream, (const __nv_bfloat16*)in, L.d.out_h, L.d.out_w, L.d.cout, c->S, r, an, beta, kappa, (__nv_bfloat16*)out, masks, L.tiles_x, L.tiles_y)));
    return DC_OK;
}

int dc_launch_concat(dc_cache* c, int layer, const void* a, int ca, const void* b, int cb)
{
    dc_layer_rt& L = c->L[layer];
    const size_t pixels = (size_t)c->S * L.d.out_h * L.d.out_w, nv = pixels * L.d.cout * c->elt / 16;
    dc_prof_scope ps(c, DC_ST_POINTWISE);
    c->launches += 1;
    if ((ca * c->elt) % 16 == 0 && (cb * c->elt) % 16 == 0 && nv <= c->piece) {
        DC_CUDA(dc_launch_pdl(k_concat_vec, dim3((unsigned)grid_for(c, nv, 256)), 256, 0, c->stream, (const uint4*)a, (unsigned)(ca * c->elt / 16), (const uint4*)b,
                              (unsigned)(cb * c->elt / 16), (unsigned)nv, (uint4*)L.map[0]));
        return DC_OK;
    }
    const dim3 grid((unsigned)grid_for(c, pixels * L.d.cout, 256));
    DISPATCH(c,
        DC_CUDA(dc_launch_pdl(k_concat<float>, grid, 256, 0, c->stream, (const float*)a, ca, (const float*)b, cb, pixels, (float*)L.map[0])),
        DC_CUDA(dc_launch_pdl(k_concat<__nv_bfloat16>, grid, 256, 0, c->stream, (const __nv_bfloat16*)a, ca, (const __nv_bfloat16*)b, cb, pixels, (__nv_bfloat16*)L.map[0])));
    return DC_OK;
}

// May the layer's own kernel write its map a second time, into a caller's buffer?  (Whole maps of 16-byte vectors.)
bool dc_writes_twice(const dc_cache* c, int layer, const void* dst)
{
    const dc_layer_desc& d = c->L[layer].d;
    if ((uintptr_t)dst % 16 != 0) return false;
    if (d.kind == DC_MAXPOOL) return !dc_layer_cached(c, layer) && (d.cout * c->elt) % 16 == 0 && units_per_piece(c, (size_t)d.out_h * d.out_w * (d.cout * c->elt / 16)) > 0;
    return d.kind == DC_ADD && c->L[layer].map_bytes % 16 == 0;
}

// A map into a caller's buffer: by a kernel where both are 16-byte aligned, so that it joins the chain of kernels before it
// without the gap of a copy node.
int dc_launch_copy_map(dc_cache* c, const void* src, void* dst, size_t bytes)
{
    if (bytes % 16 == 0 && (uintptr_t)dst % 16 == 0 && bytes / 16 <= c->piece) {
        const size_t nv = bytes / 16;
        DC_CUDA(dc_launch_pdl(k_copy_vec, dim3((unsigned)grid_for(c, nv, 256)), 256, 0, c->stream, (const uint4*)src, (unsigned)nv, (uint4*)dst));
        c->launches += 1;
        return DC_OK;
    }
    DC_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, c->stream));
    return DC_OK;
}
