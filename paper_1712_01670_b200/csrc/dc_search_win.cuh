// Interface of dc_search_win.cu: block search over a staged window, for any block size and frame layout.
#pragma once
#include "dc_common.cuh"

struct dc_win_args {
    // frames and the ends of their buffers (reads stay inside [cur, cur_end) and [prev, prev_end))
    const uint8_t* cur; const uint8_t* cur_end; size_t cur_pitch, cur_stream;
    const uint8_t* prev; const uint8_t* prev_end; size_t prev_pitch, prev_stream;
    int W, H, B, R, Gx, Gy, S, search, skip_k;
    int only_clipped;                    // 0: every block; 1: blocks clipped by the frame's edge
    uint32_t limit[4];                   // PSNR test as an SSE bound, index = 2 * (clipped in height) + (clipped in width)
    int16_t* mv; uint32_t* sse; int32_t* acc;   // acc: [S][4], zeroed: sums of Step 3
    int32_t* status;                     // device status word, or NULL
    // set by dc_launch_search_win
    int Rw, margin;                      // pixels around the tile that the window has room for, and how many of them are not staged
    int TX, TY, inv_TX, tiles_x, tiles_y, win_rows, win_cols, win_pitch;   // n / TX = n * inv_TX >> 16 for n < 32
};

// Enqueues the search; fails only with DC_ERR_CUDA.
int dc_launch_search_win(dc_win_args a, int num_sms, int device, cudaStream_t stream);
