// dc_search_blocks_noalloc: block search (Section 4, Steps 2 and 3) for callers that cannot
// allocate device memory.
//
// The regular matcher keeps its Step 3 accumulators (sum of motion vectors and count of blocks
// that pass the PSNR test, per stream) in memory that dc_cache_create allocates.  Some callers
// have no chance to create a cache: code that runs where cudaMalloc is off limits (for instance
// a latency-critical loop whose memory was fixed at start-up), or a plug-in whose host forbids
// allocation after initialisation.  This entry point does the same
// search with the accumulators in a fixed array that lives in the library image itself.
//
// The array holds DC_NOALLOC_MAX_STREAMS x 4 32-bit words (1 KiB).  Every GPU that loads the
// library holds its own copy until the process exits.  All calls on a device share it: each
// call clears the words it uses before its kernels run, and two calls that overlap on the GPU
// (different streams, no ordering between them) race on it and give wrong motion sums.
#include <math.h>

#include "dc_common.cuh"
#include "dc_search_win.cuh"

namespace {

constexpr int kMaxDevices = 64;

// Step 3 accumulators: per stream sum dx, sum dy, K, unused
static __device__ __align__(256) int32_t g_noalloc_acc[4 * DC_NOALLOC_MAX_STREAMS];

// Step 3: mean vector, rounded to nearest with halves away from zero
__global__ void k_mean_noalloc(const int32_t* acc, int S, int32_t* gmv)
{
    dc_pdl_wait();
    dc_pdl_release();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= S) return;
    const int sx = acc[4 * s], sy = acc[4 * s + 1], K = acc[4 * s + 2];
    int mx = 0, my = 0;
    if (K > 0) {
        mx = (2 * abs(sx) + K) / (2 * K); if (sx < 0) mx = -mx;
        my = (2 * abs(sy) + K) / (2 * K); if (sy < 0) my = -my;
    }
    gmv[3 * s] = mx; gmv[3 * s + 1] = my; gmv[3 * s + 2] = K;
}

// Device address of the scratch array, looked up once per device (the symbol's name is only a
// host-side handle; kernels need the address cudaGetSymbolAddress returns for the current device).
int32_t* g_scratch_ptr[kMaxDevices];
int g_sms[kMaxDevices];

}  // namespace

extern "C" int dc_search_blocks_noalloc(const uint8_t* frame_dev, const uint8_t* prev_dev, size_t pitch_bytes,
                                        int32_t width, int32_t height, int32_t n_streams, int32_t block, int32_t range,
                                        int32_t search, double psnr_db, int16_t* block_mv_dev, uint32_t* block_sse_dev,
                                        int32_t* global_mv_dev, void* cuda_stream)
{
    if (!frame_dev || !prev_dev || !block_mv_dev || !block_sse_dev || !global_mv_dev) return DC_ERR_ARG;
    if (width < 1 || height < 1 || n_streams < 1 || pitch_bytes < (size_t)width * 3) return DC_ERR_ARG;
    if (block < 4 || block > 32 || range < 0 || range > 64) return DC_ERR_CONFIG;
    if (search != DC_SEARCH_EXHAUSTIVE && search != DC_SEARCH_DIAMOND) return DC_ERR_CONFIG;
    if (!(psnr_db > 0.0) || !(psnr_db < 200.0)) return DC_ERR_CONFIG;
    if (n_streams > DC_NOALLOC_MAX_STREAMS) return DC_ERR_LIMIT;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    int dev = 0;
    DC_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) return DC_ERR_LIMIT;
    if (!g_scratch_ptr[dev]) {               // first call on this device: resolve the symbol
        int32_t* p = nullptr;
        DC_CUDA(cudaGetSymbolAddress((void**)&p, g_noalloc_acc));
        DC_CUDA(cudaDeviceGetAttribute(&g_sms[dev], cudaDevAttrMultiProcessorCount, dev));
        g_scratch_ptr[dev] = p;
    }
    dc_win_args a;
    const size_t stream_bytes = pitch_bytes * (size_t)height;
    const size_t bytes = stream_bytes * (size_t)(n_streams - 1) + pitch_bytes * (size_t)(height - 1) + (size_t)width * 3;
    a.cur = frame_dev; a.cur_end = frame_dev + bytes; a.cur_pitch = pitch_bytes; a.cur_stream = stream_bytes;
    a.prev = prev_dev; a.prev_end = prev_dev + bytes; a.prev_pitch = pitch_bytes; a.prev_stream = stream_bytes;
    a.W = width; a.H = height; a.B = block; a.R = range; a.S = n_streams; a.search = search; a.skip_k = 1; a.only_clipped = 0;
    a.Gx = dc_div_up(width, block); a.Gy = dc_div_up(height, block);
    for (int i = 0; i < 4; ++i) {
        const int bw = (i & 1) ? width - (a.Gx - 1) * block : block, bh = (i & 2) ? height - (a.Gy - 1) * block : block;
        const double lim = ceil(65025.0 * (double)(bw * bh * 3) / pow(10.0, psnr_db / 10.0)) - 1.0;
        a.limit[i] = lim >= 4294967295.0 ? 4294967295u : (uint32_t)lim;
    }
    a.mv = block_mv_dev; a.sse = block_sse_dev; a.acc = g_scratch_ptr[dev]; a.status = nullptr;
    // the array keeps the previous call's sums: clear this call's part first
    int rc = dc_launch_clear(a.acc, 4 * (int)n_streams, stream);
    if (rc != DC_OK) return rc;
    rc = dc_launch_search_win(a, g_sms[dev], dev, stream);
    if (rc != DC_OK) return rc;
    DC_CUDA(dc_launch_pdl(k_mean_noalloc, dim3((unsigned)dc_div_up(n_streams, 64)), 64, 0, stream, (const int32_t*)a.acc, (int)n_streams, global_mv_dev));
    return DC_OK;
}
