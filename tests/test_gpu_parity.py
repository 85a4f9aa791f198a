"""GPU parity: every C-ABI call against the CPU oracle on the same seeded inputs.

Integer results (motion vectors, SSE, matched maps, rectangles at every layer) must be
bit-exact; feature maps within 1e-4 max-abs (float32) or 2e-2 relative (bfloat16).
"""
import ctypes

import numpy as np
import pytest
import torch

from oracle import deepcache_oracle as orc
from paper_1712_01670_b200 import binding as B
from paper_1712_01670_b200.engine import DeepCache, device_view
from paper_1712_01670_b200.synth import configs, nets

import parity_util as U

pytestmark = pytest.mark.gpu


def rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def matcher_only(width, height, n_streams, block, R, search, psnr_db=20.0, skip_k=1, region_mode=0):
    layers = nets.single_conv(height, width)
    ws, bs = nets.random_weights(layers, 1)
    return DeepCache(width, height, layers, ws, bs, n_streams=n_streams, block=block, search_range=R,
                     search=search, psnr_db=psnr_db, skip_k=skip_k, region_mode=region_mode)


def check_pairs(pairs, block, R, search, psnr_db=20.0, skip_k=1, region_mode=0):
    """pairs: list of (prev, cur) frames of equal size, run as one batch of streams."""
    H, W = pairs[0][0].shape[:2]
    dc = matcher_only(W, H, len(pairs), block, R, search, psnr_db, skip_k, region_mode)
    try:
        dc.set_key(np.stack([p for p, _ in pairs]))
        got = dc.match_blocks(np.stack([c for _, c in pairs]))
        for s, (prev, cur) in enumerate(pairs):
            U.assert_match_equal(got, s, orc.match_blocks(cur, prev, block, R, search, psnr_db, skip_k, region_mode),
                                 f"stream {s}")
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


# ------------------------------------------------------------------ dc_match_blocks
def test_match_workload_1_exhaustive():
    w = configs.WORKLOADS[1]()
    sp = w.streams()
    check_pairs([(sp.frame(0)[0], sp.frame(1)[0])], 8, 8, B.DC_SEARCH_EXHAUSTIVE)


@pytest.mark.parametrize("widx,frames", [(2, (1, 2, 5, 9)), (3, (1, 4, 7)), (4, (1, 2, 3))])
def test_match_diamond_streams(widx, frames):
    w = configs.WORKLOADS[widx]()
    sb = w.streams(1, max(frames) + 1)
    check_pairs([(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in frames], w.block, w.range, B.DC_SEARCH_DIAMOND)


@pytest.mark.parametrize("search", [B.DC_SEARCH_EXHAUSTIVE, B.DC_SEARCH_DIAMOND, B.DC_SEARCH_THREE_STEP])
@pytest.mark.parametrize("block,shape", [(8, (40, 56)), (10, (61, 47)), (16, (16, 16)), (16, (90, 131)), (32, (70, 100)), (5, (23, 29))])
def test_match_edge_geometry(search, block, shape):
    g = rng(block * 7 + shape[0])
    H, W = shape
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    moved = np.roll(prev, (2, -3), axis=(0, 1))
    moved[H // 3:H // 3 + 9, W // 4:W // 4 + 11] = g.integers(0, 256, size=(min(9, H - H // 3), min(11, W - W // 4), 3))
    smooth = np.clip(prev.astype(np.int32) + g.integers(-6, 7, size=prev.shape), 0, 255).astype(np.uint8)
    const = np.full_like(prev, 93)
    pairs = [(prev, moved), (prev, prev), (prev, smooth), (const, const), (const, prev)]
    check_pairs(pairs, block, 4, search)


def test_match_ties_and_thresholds():
    # periodic pattern: several displacements tie at SSE 0; the smallest motion must win on both sides
    x = np.arange(64)
    row = ((x % 4) * 60).astype(np.uint8)
    prev = np.repeat(np.repeat(row[None, :, None], 48, 0), 3, 2)
    cur = np.roll(prev, -1, axis=1)
    for search in (B.DC_SEARCH_EXHAUSTIVE, B.DC_SEARCH_DIAMOND, B.DC_SEARCH_THREE_STEP):
        check_pairs([(prev, cur), (cur, prev)], 8, 6, search)
    # other thresholds move the integer SSE bound
    g = rng(3)
    a = g.integers(0, 256, size=(48, 64, 3), dtype=np.uint8)
    b = np.clip(a.astype(np.int32) + g.integers(-40, 41, size=a.shape), 0, 255).astype(np.uint8)
    for T in (12.0, 18.5, 25.0, 33.3):
        check_pairs([(a, b)], 8, 3, B.DC_SEARCH_DIAMOND, psnr_db=T)


def test_match_full_hd_batch():
    """Workload 5's matcher geometry (1920x1080, block 16, range 32, last block row 8 px) on 2 streams."""
    w = configs.WORKLOADS[5]()
    sb = w.streams(2, 3)
    pairs = [(sb.frame(1, s), sb.frame(2, s)) for s in range(2)]
    check_pairs(pairs, 16, 32, B.DC_SEARCH_DIAMOND)
    # k-skip at this size: every searched block is walked with a private window from its start
    check_pairs(pairs, 16, 32, B.DC_SEARCH_DIAMOND, skip_k=2)


@pytest.mark.parametrize("widx,frames,R", [(2, (1, 2, 5), 16), (3, (1, 4), 7), (4, (2, 3), 24), (2, (3,), 1)])
def test_match_three_step_streams(widx, frames, R):
    """Three step search (Section 7.5) as the Step 2 unit: first steps 8, 4, 8 and 1 for these ranges."""
    w = configs.WORKLOADS[widx]()
    sb = w.streams(1, max(frames) + 1)
    check_pairs([(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in frames], w.block, R, B.DC_SEARCH_THREE_STEP)
    check_pairs([(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in frames], 10, R, B.DC_SEARCH_THREE_STEP, skip_k=2)


def test_match_three_step_full_hd():
    w = configs.WORKLOADS[5]()
    sb = w.streams(2, 3)
    check_pairs([(sb.frame(1, s), sb.frame(2, s)) for s in range(2)], 16, 32, B.DC_SEARCH_THREE_STEP)


def test_infer_with_three_step():
    w = configs.WORKLOADS[3]()
    w.search = configs.SEARCH_TSS
    U.run_stream_parity(w, 1, list(range(4)))


@pytest.mark.parametrize("R,shape", [(32, (97, 150)), (16, (64, 64)), (8, (50, 300)), (5, (33, 47)), (13, (80, 131)), (0, (32, 32))])
def test_match_exhaustive_16_fast_path(R, shape):
    """16-pixel blocks with exhaustive search run on the register-blocked kernel (full groups of 32 dx values,
    the remaining columns one candidate per lane) and clipped edge blocks on the generic one."""
    g = rng(R * 31 + shape[0])
    H, W = shape
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    moved = np.roll(prev, (min(R, 3), -min(R, 7)), axis=(0, 1))
    far = np.roll(prev, (-R, R), axis=(0, 1))                  # best vectors at the corner of the range
    smooth = np.clip(prev.astype(np.int32) + g.integers(-6, 7, size=prev.shape), 0, 255).astype(np.uint8)
    const = np.full_like(prev, 200)
    check_pairs([(prev, moved), (prev, far), (prev, smooth), (const, const), (far, prev)], 16, R, B.DC_SEARCH_EXHAUSTIVE)
    check_pairs([(prev, moved)], 16, R, B.DC_SEARCH_EXHAUSTIVE, skip_k=2)


def test_match_exhaustive_video_streams():
    w = configs.WORKLOADS[2]()
    sb = w.streams(1, 4)
    check_pairs([(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in (1, 2, 3)], 16, 16, B.DC_SEARCH_EXHAUSTIVE)
    w = configs.WORKLOADS[5]()                                 # 1920x1080: 120 full columns, last block row 8 px
    sb = w.streams(1, 3)
    f1, f2 = sb.frame(1, 0), sb.frame(2, 0)
    check_pairs([(f1[:200, :1000], f2[:200, :1000])], 16, 32, B.DC_SEARCH_EXHAUSTIVE)


def two_motion_pair(g, H, W):
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    cur = prev.copy()
    cur[:, W // 2:] = np.roll(prev, (-2, 3), axis=(0, 1))[:, W // 2:]
    cur[H // 3:H // 3 + 7, 2:13] = g.integers(0, 256, size=(7, 11, 3))
    return prev, cur


@pytest.mark.parametrize("search", [B.DC_SEARCH_EXHAUSTIVE, B.DC_SEARCH_DIAMOND, B.DC_SEARCH_THREE_STEP])
@pytest.mark.parametrize("block,shape", [(8, (40, 56)), (16, (90, 131)), (16, (64, 64)), (10, (61, 47))])
def test_match_per_block_regions(search, block, shape):
    """The per-block extension of Steps 4-5: own vectors, merge of equal vectors only (fast and generic kernels)."""
    g = rng(block + shape[1])
    H, W = shape
    prev, cur = two_motion_pair(g, H, W)
    smooth = np.clip(prev.astype(np.int32) + g.integers(-6, 7, size=prev.shape), 0, 255).astype(np.uint8)
    check_pairs([(prev, cur), (prev, prev), (prev, smooth), (cur, prev)], block, 4, search,
                region_mode=B.DC_REGIONS_PER_BLOCK)
    check_pairs([(prev, cur)], block, 4, search, skip_k=2, region_mode=B.DC_REGIONS_PER_BLOCK)


def test_match_per_block_streams_and_full_hd():
    w = configs.WORKLOADS[4]()
    sb = w.streams(1, 4)
    check_pairs([(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in (1, 2, 3)], 16, 24, B.DC_SEARCH_DIAMOND,
                region_mode=B.DC_REGIONS_PER_BLOCK)
    w = configs.WORKLOADS[5]()
    sb = w.streams(2, 3)
    check_pairs([(sb.frame(1, s), sb.frame(2, s)) for s in range(2)], 16, 32, B.DC_SEARCH_DIAMOND,
                region_mode=B.DC_REGIONS_PER_BLOCK)


@pytest.mark.parametrize("gx,gy", [(31, 33), (32, 32), (33, 31), (64, 65), (1, 40), (40, 1), (96, 3), (256, 256), (257, 256)])
def test_match_merge_grid_words(gx, gy):
    """Step 5's runs and rectangles across the 32-block words of its bit strings, the largest grid in shared memory with one vector
    per frame (256 x 256; with vectors per block it is beyond) and one beyond in both modes."""
    g = rng(gx * 131 + gy)
    W, H = gx * 4, gy * 4
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    prev[: H // 2] = 77                                        # whole columns and rows that match
    pairs = [(prev, prev)]
    for n in (3, 12):
        cur = prev.copy()
        for _ in range(n):                                     # unmatched rectangles of blocks
            x, y = int(g.integers(0, gx)), int(g.integers(0, gy))
            part = cur[4 * y:4 * (y + int(g.integers(1, 9))), 4 * x:4 * (x + int(g.integers(1, 9)))]
            part[:] = g.integers(0, 256, size=part.shape, dtype=np.uint8)
        pairs.append((prev, cur))
    for mode in (B.DC_REGIONS_GLOBAL, B.DC_REGIONS_PER_BLOCK):
        check_pairs(pairs, 4, 1, B.DC_SEARCH_DIAMOND, region_mode=mode)


@pytest.mark.parametrize("R", [0, 1, 2, 3, 7, 15, 63, 64])
@pytest.mark.parametrize("shape", [(16, 16), (33, 129), (47, 143), (100, 260)])
def test_match_three_step_16_windows(R, shape):
    """The staged three step search: every first step, strips and blocks clipped on either side, ties."""
    g = rng(R * 37 + shape[1])
    H, W = shape
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    far = np.roll(prev, (-min(R, H // 3), min(R, W // 3)), axis=(0, 1))
    const = np.full_like(prev, 50)
    smooth = np.repeat((np.arange(W) // 4 % 3 * 40).astype(np.uint8)[None, :, None], H, 0).repeat(3, 2)
    check_pairs([(prev, far), (const, const), (smooth, np.roll(smooth, 2, axis=1)), (prev, smooth)], 16, R, B.DC_SEARCH_THREE_STEP)


@pytest.mark.parametrize("search,R,block", [(B.DC_SEARCH_DIAMOND, 1, 16), (B.DC_SEARCH_DIAMOND, 5, 16), (B.DC_SEARCH_DIAMOND, 40, 16),
                                            (B.DC_SEARCH_THREE_STEP, 3, 16), (B.DC_SEARCH_THREE_STEP, 31, 16), (B.DC_SEARCH_DIAMOND, 1, 10),
                                            (B.DC_SEARCH_DIAMOND, 12, 10), (B.DC_SEARCH_DIAMOND, 18, 4), (B.DC_SEARCH_DIAMOND, 30, 10),
                                            (B.DC_SEARCH_DIAMOND, 16, 11), (B.DC_SEARCH_DIAMOND, 7, 13), (B.DC_SEARCH_THREE_STEP, 9, 10)])
def test_match_many_tiles(search, R, block):
    """Enough tiles for the searches' instances of many warps per SM, with what their rounds meet at the edges: strips and blocks cut on
    either side, range limits next to the start, equal scores, walks that leave the staged window, ranges beyond a fixed pitch."""
    g = rng(R)
    H, W = 70, 147
    x, y = np.meshgrid(np.arange(W), np.arange(H))
    pairs = []
    for i in range(60):
        kind = i % 4
        if kind == 0:                                              # smooth: long walks along a slope
            base = np.stack([np.hypot(x - W * g.random(), y - H * g.random()) * g.uniform(0.5, 1.5) for _ in range(3)], -1)
            prev = base.astype(np.int64).astype(np.uint8)
            cur = np.roll(prev, (int(g.integers(-9, 10)), int(g.integers(-20, 21))), axis=(0, 1))
        elif kind == 1:                                            # few levels: many equal scores
            prev = (g.integers(0, 2, (H, W, 3)) * 90).astype(np.uint8)
            cur = np.roll(prev, (1, -2), axis=(0, 1))
        elif kind == 2:
            prev = np.repeat(np.repeat(((x // 4) % 3 * 40).astype(np.uint8)[..., None], 3, 2), 1, 0)
            cur = np.roll(prev, 2, axis=1)
        else:
            prev = g.integers(0, 256, (H, W, 3), dtype=np.uint8)
            cur = np.roll(prev, (-2, 2), axis=(0, 1))
        pairs.append((prev, cur))
    check_pairs(pairs, block, R, search)


@pytest.mark.parametrize("S", [2, 40])
@pytest.mark.parametrize("block,W,H", [(17, 100, 87), (20, 81, 100), (21, 150, 64), (24, 97, 98), (31, 94, 125), (32, 67, 100)])
def test_match_verify_large_blocks(block, W, H, S):
    """Step 4 of blocks of more than 16 pixels, a warp per block: rows of 13 to 25 words, two and one to a load, cut on either side, at every place of a
    row in its words, most blocks with a vector that is not the mean."""
    g = rng(block + S)
    pairs = []
    for s in range(S):
        prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
        cur = np.roll(prev, (s % 5 - 2, s % 7 - 3), axis=(0, 1))
        cur = np.clip(cur.astype(int) + g.normal(0, 14, size=cur.shape) * (g.random((H, 1, 1)) < 0.7), 0, 255).astype(np.uint8)
        pairs.append((prev, cur))
    check_pairs(pairs, block, 5, B.DC_SEARCH_DIAMOND)


@pytest.mark.parametrize("h,w,k,st,p", [(33, 41, 3, 2, 1), (32, 32, 7, 2, 3), (47, 35, 5, 3, 2), (30, 31, 7, 3, 0), (39, 227, 11, 4, 0), (41, 43, 11, 4, 5)])
def test_frame_into_block_map(h, w, k, st, p):
    """A frame goes straight into a strided first layer's block map: blocks of 2, 3 and 4, padding on every side, rows that
    end inside a word.  The same values as the block map of the frame's own input map, so the same output."""
    S = 3
    g = rng(h * w)
    nb = nets.NetBuilder(h, w)
    nb.conv(-1, 32, k, st, p, 1)
    ws, bs = nets.random_weights(nb.layers, 5)
    frame = torch.from_numpy(g.integers(0, 256, size=(S, h, w, 3), dtype=np.uint8)).cuda()
    dc = DeepCache(w, h, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_BF16)
    out = dc.infer_frame(frame)
    want = dc.conv_partial(0, (frame.float() * (1.0 / 255.0)).to(torch.bfloat16))
    assert torch.equal(out.view(want.shape), want)
    dc.close()


@pytest.mark.parametrize("hw,S", [((64, 64), 1), ((160, 128), 16)])
def test_infer_back_to_back_frames(hw, S):
    """Frames without a pause: tile lists and first weights are read before a kernel's turn (narrow layers whose weight
    tiles fit the ring whole).  No wait may run out, and the maps are those of frames run one by one."""
    g = rng(S)
    net = nets.inception_lrn_net(*hw)
    ws, bs = nets.random_weights(net, 3)
    # three frames of noise of which two share their left half: much, little and nothing to reuse in turn
    frames = [torch.from_numpy(g.integers(0, 256, size=(S, hw[0], hw[1], 3), dtype=np.uint8)).cuda() for _ in range(3)]
    frames[1][:, :, : hw[1] // 2] = frames[0][:, :, : hw[1] // 2]
    maps = []
    for pause in (False, True):
        dc = DeepCache(hw[1], hw[0], net, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_BF16, cache_pool=True)
        rec = []
        for i in range(300):
            dc.infer_frame(frames[i % 3], want_out=False)
            if pause:
                torch.cuda.synchronize()
            if i in (41, 150, 298, 299):
                rec += [dc.layer_map(k) for k in range(len(net))]
        assert dc.status() == B.DC_OK
        maps.append(rec)
        dc.close()
    assert all(torch.equal(a, b) for a, b in zip(*maps))


@pytest.mark.parametrize("widx", [2, 3, 4])
def test_infer_per_block_regions(widx):
    U.run_stream_parity(configs.WORKLOADS[widx](), 1, list(range(4)), region_mode=B.DC_REGIONS_PER_BLOCK)


@pytest.mark.parametrize("widx,frames", [(2, 6), (3, 5), (5, 3)])
def test_infer_with_cached_pooling(widx, frames):
    """Reuse in max-pooling layers (the extension Section 5 mentions): maps, rectangles and per-layer reuse ratios
    of the pooling layers against the oracle with the same switch."""
    w = configs.WORKLOADS[widx]()
    U.run_stream_parity(w, 2 if widx == 5 else 1, list(range(frames)), cache_pool=True)


def test_cached_pooling_reuses_pixels():
    w = configs.WORKLOADS[2]()
    sb = w.streams(1, 3)
    dc = DeepCache.from_workload(w, cache_pool=True)
    try:
        for i in range(3):
            out, stats = dc.infer_frame(sb.frame(i), want_stats=True)
        pools = [i for i, l in enumerate(w.layers) if l["kind"] == orc.KIND_MAXPOOL]
        assert pools and all(stats[0].reuse_ratio[i] > 0.2 for i in pools)
    finally:
        dc.close()


@pytest.mark.parametrize("dtype", [configs.DTYPE_FP32, configs.DTYPE_BF16])
def test_infer_graph_with_every_layer_kind(dtype):
    """Convolution, LRN, pooling, two branches joined by a concat and a fully-connected head (all rows of Table 2),
    every layer's map and rectangles against the oracle over a refresh, cached frames and the next refresh."""
    w = configs.WORKLOADS[2]()
    w.layers = nets.inception_lrn_net(80, 96)
    w.width, w.height, w.dtype, w.expire_n = 96, 80, dtype, 3
    crop = w.make_streams
    w.make_streams = lambda s, f, first=0: _cropped(crop(s, f, first), 80, 96)
    U.run_stream_parity(w, 2, list(range(5)))
    U.run_stream_parity(w, 1, list(range(3)), cache_pool=True, region_mode=B.DC_REGIONS_PER_BLOCK)


@pytest.mark.parametrize("dtype", [B.DC_FP32, B.DC_BF16])
def test_large_maps_are_launched_in_pieces(dtype):
    """Launches whose kernels index with 32 bits are cut between rows or streams.  With the limit lowered to a few thousand
    items the maps of every layer are the same, for the frame's own map, the padded operand copy, pooling of every window
    and LRN, cached or not, and for a limit below one stream (the general kernels; cached layers stay whole)."""
    S, hi, wi = 5, 45, 53
    b = nets.NetBuilder(hi, wi)
    x = b.conv(-1, 32, 3, 1, 1)
    p2, p3, p5 = b.maxpool(x, 2, 2), b.maxpool(x, 3, 2, 1), b.maxpool(x, 5, 3, 2)
    b.conv(p2, 32, 3, 1, 1)
    b.lrn(p3, 2)
    b.lrn(x, 1)
    b.conv(p5, 32, 1, 1, 0)
    if dtype == B.DC_FP32:
        b.maxpool(-1, 2, 2)                                        # reads the frame's map
    ws, bs = nets.random_weights(b.layers, 2)
    g = rng(6)
    frames = [torch.from_numpy(g.integers(0, 256, size=(S, hi, wi, 3), dtype=np.uint8)).cuda() for _ in range(2)]
    frames[1][:, :, : wi // 2] = frames[0][:, :, : wi // 2]
    limit = B.load().dc_debug_piece
    limit.restype, limit.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
    for pool in (False, True):
        want = None
        for items in ((0, 25000, 9600) if pool else (0, 25000, 9600, 700)):
            dc = DeepCache(wi, hi, b.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, cache_pool=pool)
            assert items == 0 or limit(dc.handle, items) == B.DC_OK
            for f in frames:
                dc.infer_frame(f)
            got = [dc.layer_map(i).float() for i in range(len(b.layers))]
            want = want or got
            for i, (m, w_) in enumerate(zip(got, want)):
                if b.layers[i]["kind"] == B.DC_LRN and 0 < items < 20000:
                    torch.testing.assert_close(m, w_, rtol=0.01, atol=1e-5)       # the general kernel's own power function
                else:
                    assert torch.equal(m, w_), (items, i)
            assert dc.status() == B.DC_OK
            dc.close()


class _cropped:
    """A stream batch cut to the top-left h x w pixels of every frame."""

    def __init__(self, batch, h, w):
        self.batch, self.h, self.w = batch, h, w

    def frame(self, i, s=None):
        f = self.batch.frame(i) if s is None else self.batch.frame(i, s)
        return np.ascontiguousarray(f[..., :self.h, :self.w, :])


@pytest.mark.parametrize("dtype", [B.DC_FP32, B.DC_BF16])
def test_lrn_in_strips_of_two_rows(dtype):
    """Maps large enough that a thread takes two rows: the bits of the launches stream by stream, where it takes one, over full frames and
    reused pixels (odd heights; rectangles that begin and end inside a strip, rows 1 to 28 and 3 to 28), and the formula in 64 bits: the
    window's sum is rounded up to ten times by 2^-24, the power by 1.5 * 2^-23, alpha and the product by 2^-24; bfloat16 by 2^-9."""
    S, hi, wi, ch = 72, 45, 53, 32
    least, most = (h * w * ch * (4 if dtype == B.DC_FP32 else 2) // 16 for h, w in ((hi - 2, wi - 2), (hi, wi)))
    assert S * least >= torch.cuda.get_device_properties(0).multi_processor_count * 4096 > most
    b = nets.NetBuilder(hi, wi)
    b.lrn(b.conv(-1, ch, 3, 1, 0), 1)
    b.lrn(b.conv(-1, ch, 3, 1, 1), 2)
    ws, bs = nets.random_weights(b.layers, 2)
    g = rng(6)
    frames = [torch.from_numpy(g.integers(0, 256, size=(S, hi, wi, 3), dtype=np.uint8)).cuda() for _ in range(2)]
    frames[1][:, :35, : wi // 2] = frames[0][:, :35, : wi // 2]
    limit = B.load().dc_debug_piece
    limit.restype, limit.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
    for pool in (False, True):
        want = None
        for items in (0, most + 100):
            dc = DeepCache(wi, hi, b.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, cache_pool=pool, lrn=(2.0, 0.75, 1.0))
            assert items == 0 or limit(dc.handle, items) == B.DC_OK
            got = []
            for f in frames:
                _, stats = dc.infer_frame(f, want_stats=True)
                for r in (1, 2):
                    layer, n = 2 * r - 1, 2 * r + 1
                    got.append(dc.layer_map(layer))
                    if pool and f is frames[1]:
                        assert min(st.reuse_ratio[layer] for st in stats) > 0.05
                        continue
                    a = dc.layer_map(layer - 1).double()
                    sums = torch.nn.functional.avg_pool2d((a * a).permute(0, 3, 1, 2), n, 1, r, divisor_override=1).permute(0, 2, 3, 1)
                    exact = a * (1.0 + 2.0 / (n * n) * sums) ** -0.75
                    assert ((got[-1].double() - exact).abs() <= (7 * 2.0 ** -23 if dtype == B.DC_FP32 else 2.0 ** -8) * exact.abs()).all()
            want = want or got
            assert all(torch.equal(u, v) for u, v in zip(got, want)), items
            assert dc.status() == B.DC_OK
            dc.close()


@pytest.mark.parametrize("dtype", [B.DC_FP32, B.DC_BF16])
@pytest.mark.parametrize("last", ["maxpool", "maxpool2", "add"])
def test_last_map_into_any_buffer(dtype, last):
    """A last pooling or add layer that writes the caller's buffer itself: at any element, and in launches of pieces."""
    S, hi, wi = 5, 45, 54
    b = nets.NetBuilder(hi, wi)
    x = b.conv(-1, 32, 3, 1, 1)
    if last == "add":
        b.add(x, b.conv(x, 32, 1, 1, 0))
    else:
        b.maxpool(x, 2, 2) if last == "maxpool2" else b.maxpool(x, 3, 2, 1)
    ws, bs = nets.random_weights(b.layers, 2)
    frames = torch.from_numpy(rng(8).integers(0, 256, size=(2, S, hi, wi, 3), dtype=np.uint8)).cuda()
    limit = B.load().dc_debug_piece
    limit.restype, limit.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
    want = None
    for items in (0, 9600, 700):
        for off in (0, 1, 8):
            dc = DeepCache(wi, hi, b.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype)
            assert items == 0 or limit(dc.handle, items) == B.DC_OK
            n = int(np.prod(dc.out_shape(-1)))
            got = []
            for f in frames:
                room = torch.full((n + 24,), 7.0, dtype=dc.tdtype, device="cuda")
                B.dc_infer_frame(dc.handle, f, wi * 3, room[off:off + n])
                assert (room[:off] == 7).all() and (room[off + n:] == 7).all()
                got.append(room[off:off + n].view(dc.out_shape(-1)))
                assert torch.equal(got[-1], dc.layer_map(len(b.layers) - 1))
            want = want or got
            assert all(torch.equal(u, v) for u, v in zip(got, want)), (items, off)
            dc.close()


@pytest.mark.parametrize("k", [2, 3])
def test_match_k_skip(k):
    """Section 4's k-skip: Step 2 on every k-th block row and column only (16-px fast path and generic path)."""
    w = configs.WORKLOADS[2]()
    sb = w.streams(1, 4)
    pairs = [(sb.frame(i - 1)[0], sb.frame(i)[0]) for i in (1, 2, 3)]
    check_pairs(pairs, 16, 16, B.DC_SEARCH_DIAMOND, skip_k=k)
    check_pairs(pairs, 10, 6, B.DC_SEARCH_DIAMOND, skip_k=k)
    check_pairs([(p[:96, :96], c[:96, :96]) for p, c in pairs], 8, 3, B.DC_SEARCH_EXHAUSTIVE, skip_k=k)


def test_infer_with_k_skip():
    U.run_stream_parity(configs.WORKLOADS[3](), 1, list(range(5)), skip_k=2)


def test_match_needs_a_key():
    dc = matcher_only(32, 32, 1, 8, 4, B.DC_SEARCH_DIAMOND)
    try:
        with pytest.raises(B.DeepCacheError) as e:
            dc.match_blocks(np.zeros((32, 32, 3), np.uint8))
        assert e.value.status == B.DC_ERR_STATE
    finally:
        dc.close()


# ------------------------------------------------------------------ dc_propagate_regions
def random_regions(g, n, W, H, max_shift=9):
    out = np.zeros(n, orc.REGION_DTYPE)
    for i in range(n):
        w, h = int(g.integers(1, W // 2)), int(g.integers(1, H // 2))
        x, y = int(g.integers(0, W - w + 1)), int(g.integers(0, H - h + 1))
        sx = int(np.clip(x + g.integers(-max_shift, max_shift + 1), 0, W - w))
        sy = int(np.clip(y + g.integers(-max_shift, max_shift + 1), 0, H - h))
        out[i] = (x, y, w, h, sx, sy)
    return out


def check_propagation(layers, W, H, n_streams, executable=True):
    g = rng(len(layers))
    if executable:
        ws, bs = nets.random_weights(layers, 2)
    else:
        ws, bs = [None] * len(layers), [None] * len(layers)
    dc = DeepCache(W, H, layers, ws, bs, n_streams=n_streams, block=16, search_range=8, dtype=B.DC_BF16)
    try:
        regs = torch.zeros((n_streams, dc.max_regions, 6), dtype=torch.int32)
        counts, per_stream = [], []
        for s in range(n_streams):
            n = int(g.integers(0, min(dc.max_regions, 40) + 1)) if s else min(dc.max_regions, 37)
            r = random_regions(g, n, W, H)
            per_stream.append(r)
            counts.append(n)
            if n:
                regs[s, :n] = torch.from_numpy(np.ascontiguousarray(r).view(np.int32).reshape(n, 6))
        out, n_out = dc.propagate_regions(regs.cuda(), torch.tensor(counts, dtype=torch.int32).cuda())
        for s in range(n_streams):
            want = orc.propagate(layers, (H, W), per_stream[s])
            for li in range(len(layers)):
                U.assert_regions_equal(U.regions_np(out[li, s, :counts[s]]), want[li], f"layer {li} stream {s}")
                assert int(n_out[li, s]) == counts[s]
                assert not out[li, s, counts[s]:].any()
    finally:
        dc.close()


@pytest.mark.parametrize("net,W,H", [("small", 227, 227), ("alexnet", 227, 227), ("resnet", 224, 224), ("vgg", 1920, 1080)])
def test_propagate_networks(net, W, H):
    layers = {"small": lambda: nets.small_cnn(H, W), "alexnet": lambda: nets.alexnet_trunk(H, W),
              "resnet": lambda: nets.resnet50_trunk(H, W), "vgg": lambda: nets.vgg16_trunk(224, 224, H, W)}[net]()
    check_propagation(layers, W, H, 3)


@pytest.mark.parametrize("S,slots,odd", [(4, 37 * 32, 0), (5, 37 * 32 - 1, 1), (1, 1, 0), (1, 33, 1), (3, 65, 0)])
def test_propagate_lists_of_any_length(S, slots, odd):
    """A caller's lists in CTAs of 32 and of 64 rectangles, with last ones that are not full, written to arrays that start at any word."""
    layers = nets.inception_lrn_net(96, 128)
    ws, bs = nets.random_weights(layers, 3)
    dc = DeepCache(128, 96, layers, ws, bs, n_streams=S, block=16, search_range=2, dtype=B.DC_BF16, max_regions=slots)
    try:
        g = rng(slots)
        n = [slots - min(s, slots - 1) for s in range(S)]
        regs = np.zeros((S, slots, 6), np.int32)
        for s in range(S):
            w, h = g.integers(1, 90, n[s]), g.integers(1, 70, n[s])
            x, y = g.integers(0, 128 - w + 1), g.integers(0, 96 - h + 1)
            regs[s, :n[s]] = np.stack([x, y, w, h, g.integers(0, 128 - w + 1), g.integers(0, 96 - h + 1)], 1)
        buf = torch.full((odd + len(layers) * S * slots * 6,), -7, dtype=torch.int32, device="cuda")
        out = buf[odd:].view(len(layers), S, slots, 6)
        n_out = torch.zeros((len(layers), S), dtype=torch.int32, device="cuda")
        B.dc_propagate_regions(dc.handle, torch.from_numpy(regs).cuda(), torch.tensor(n, dtype=torch.int32, device="cuda"), 0, len(layers), out, n_out)
        torch.cuda.synchronize()
        assert not odd or int(buf[0]) == -7
        for s in range(S):
            want = orc.propagate(layers, (96, 128), U.regions_np(torch.from_numpy(regs[s, :n[s]])))
            for l in range(len(layers)):
                U.assert_regions_equal(U.regions_np(out[l, s, :n[s]]), want[l], f"stream {s} layer {l}")
                assert not out[l, s, n[s]:].any() and int(n_out[l, s]) == n[s]
    finally:
        dc.close()


def test_propagate_table2_rows():
    """Layer kinds that only region propagation knows (LRN, concat, fully connected)."""
    b = nets.NetBuilder(96, 96)
    c1 = b.conv(-1, 16, 11, 2, 5)
    b.layers.append(dict(kind=B.DC_RELU, kh=1, kw=1, sh=1, sw=1, ph=0, pw=0, cin=16, cout=16, relu=0, in0=c1, in1=-1, out_h=48, out_w=48))
    b.layers.append(dict(kind=B.DC_LRN, kh=5, kw=5, sh=1, sw=1, ph=2, pw=2, cin=16, cout=16, relu=0, in0=1, in1=-1, out_h=48, out_w=48))
    p = b.maxpool(2, 3, 2, 1)
    q = b.conv(2, 16, 3, 2, 1)
    b.layers.append(dict(kind=B.DC_CONCAT, kh=1, kw=1, sh=1, sw=1, ph=0, pw=0, cin=16, cout=32, relu=0, in0=p, in1=q, out_h=24, out_w=24))
    b.layers.append(dict(kind=B.DC_FC, kh=1, kw=1, sh=1, sw=1, ph=0, pw=0, cin=32, cout=10, relu=0, in0=5, in1=-1, out_h=1, out_w=1))
    check_propagation(b.layers, 96, 96, 2, executable=False)


def test_propagate_many_branches_and_late_readers():
    """More open branches than a thread keeps places for (the rest is read back from the table), rectangles that vanish on the way, and late
    readers of the frame: no warp may end before them."""
    b = nets.NetBuilder(96, 80)
    xs = [b.conv(-1, 16, 3, 1, 1)]
    for k in (1, 3, 1, 7, 1, 9, 1, 1):
        xs.append(b.conv(xs[-1], 16, k, 1, k // 2))
    y = b.conv(xs[-1], 16, 11, 1, 5)
    for x in xs:                                                    # nine branches, closed in the order they were opened
        y = b.add(x, y)
    late = b.conv(-1, 16, 1, 1, 0)
    y = b.add(y, late)
    z = b.conv(-1, 16, 5, 1, 2)
    b.concat(z, late)
    check_propagation(b.layers, 80, 96, 3)


def test_propagate_strides_that_are_no_power_of_two():
    b = nets.NetBuilder(120, 140)
    x = b.conv(-1, 16, 3, 1, 1)
    p = b.conv(x, 16, 5, 3, 2)
    q = b.maxpool(x, 3, 3, 1)
    y = b.add(p, q)
    y = b.conv(y, 16, 3, 2, 1)
    b.maxpool(y, 2, 5, 0)
    b.conv(x, 16, 7, 6, 3)
    b.conv(x, 16, 1, 4, 0)
    check_propagation(b.layers, 140, 120, 3)


def winding_pair(R):
    """A frame and its predecessor in which the walk of one block winds through its whole search range, and the walk's centres.  The block is grey
    but for its first pixel, so that a candidate's SSE falls with the previous frame's pixel there along one direction of colour space; all
    pixels of the previous frame lie on one sphere around grey, so that nothing else changes it.  Their colours get better along the path, whose
    centres' diamonds hold no later centre but the next."""
    path = [(0, 0)]

    def go(dx, dy):
        path.append((path[-1][0] + dx, path[-1][1] + dy))

    E = R - 2
    while path[-1][0] > -E and path[-1][1] < E - 4:                  # to a corner, then row by row through the rest
        go(-1, 1)
    go(0, 2), go(1, 1)
    sx = 1
    while True:
        left = -E if path[-1][1] <= -8 else max(-E, 9 - path[-1][1])
        while path[-1][0] + 2 <= E if sx > 0 else path[-1][0] - 2 >= left:
            go(2 * sx, 0)
        if path[-1][1] - 3 < -E:
            break
        go(0, -2), go(-sx, -1)
        sx = -sx
    v = np.arange(-127, 128)
    sphere = np.stack([c.ravel() for c in np.meshgrid(v, v, v, indexing="ij")], 1)
    sphere = sphere[(sphere ** 2).sum(1) == 15461]
    towards = np.array([127, 101, 83])
    _, first = np.unique(sphere @ towards, return_index=True)        # by how far they lie in that direction
    colours = sphere[first]
    assert len(colours) > len(path)
    size = 16 + 2 * R
    cur = np.full((size, size, 3), 128, np.uint8)
    cur[R, R] += towards.astype(np.uint8)
    prev = np.broadcast_to(128 + colours[0], (size, size, 3)).astype(np.uint8)
    for i, (x, y) in enumerate(path):
        prev[R + y, R + x] = 128 + colours[len(colours) - len(path) + i]
    return prev, cur, path


def test_match_winding_walk():
    """A walk of two thousand moves through several hundred windows: every one of them is made, to the last."""
    R = 64
    prev, cur, path = winding_pair(R)
    m = orc.match_blocks(cur, prev, 16, R, B.DC_SEARCH_DIAMOND, 20.0)
    assert tuple(np.asarray(m["mv"])[4, 4]) == path[-1] and len(path) > 2000
    check_pairs([(prev, cur)], 16, R, B.DC_SEARCH_DIAMOND)


def test_propagate_more_rectangles_than_a_batch_holds():
    """A frame's rectangles in several batches (a deep network leaves room for few of them at once): table, lists and counts of every layer."""
    b = nets.NetBuilder(128, 128)
    x = b.conv(-1, 16, 3, 1, 1)
    for _ in range(59):
        x = b.conv(x, 16, 1, 1, 0)
    ws, bs = nets.random_weights(b.layers, 2)
    dc = DeepCache(128, 128, b.layers, ws, bs, n_streams=2, block=4, search_range=0, dtype=B.DC_BF16)
    try:
        f0 = rng(5).integers(0, 256, (2, 128, 128, 3), dtype=np.uint8)
        f1 = f0.copy()
        for s in range(2):
            for y in range(32):
                for bx in range((y + s) % 3, 32, 3):
                    f1[s, 4 * y:4 * y + 4, 4 * bx:4 * bx + 4] ^= 0x80
        dc.infer_frame(f0)
        _, stats = dc.infer_frame(f1, want_stats=True)
        regs0, n = dc.layer_regions(-1)
        for s in range(2):
            count = int(n[s])
            assert count > 300
            want = orc.propagate(b.layers, (128, 128), U.regions_np(regs0[s, :count]))
            for li in range(len(b.layers)):
                regs, _ = dc.layer_regions(li)
                U.assert_regions_equal(U.regions_np(regs[s, :count]), want[li], f"layer {li} stream {s}")
                assert abs(stats[s].reuse_ratio[li] - float((want[li]["w"] * want[li]["h"]).sum()) / 128 ** 2) < 1e-6
    finally:
        dc.close()


# ------------------------------------------------------------------ dc_conv_partial
@pytest.mark.parametrize("dtype", [B.DC_FP32, B.DC_BF16])
@pytest.mark.parametrize("hi,wi,cin,cout,k,s,p,relu", [
    (37, 45, 3, 16, 3, 1, 1, 1), (64, 64, 32, 64, 3, 1, 1, 1), (227, 227, 3, 96, 11, 4, 0, 1),
    (27, 27, 96, 256, 5, 1, 2, 1), (56, 56, 64, 128, 1, 2, 0, 0), (30, 33, 16, 24, 3, 2, 1, 0),
    (14, 14, 256, 512, 3, 1, 1, 1), (224, 224, 3, 64, 7, 2, 3, 1), (40, 52, 3, 64, 3, 1, 1, 1),
    (33, 35, 3, 32, 5, 1, 2, 0), (28, 28, 32, 96, 3, 1, 1, 1), (20, 24, 16, 64, 1, 1, 0, 1),
    (28, 28, 64, 64, 3, 2, 1, 1), (31, 29, 128, 64, 3, 2, 1, 0), (40, 40, 32, 32, 5, 3, 2, 1)])
def test_conv_partial(dtype, hi, wi, cin, cout, k, s, p, relu):
    g = rng(hi + cin + k)
    bf16 = dtype == B.DC_BF16
    quant = orc.QUANT_BF16 if bf16 else orc.QUANT_NONE
    S = 2
    b = nets.NetBuilder(hi, wi, cin)
    b.conv(-1, cout, k, s, p, relu)
    L = b.layers[0]
    wts = g.normal(0, np.sqrt(2.0 / (k * k * cin)), size=(cout, k, k, cin)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    layers = [dict(L)]
    x = g.normal(size=(S, hi, wi, cin))
    prev = g.normal(size=(S, L["out_h"], L["out_w"], cout))
    # inputs exactly representable in the map's element type, so copies can be compared bit for bit
    x, prev = x.astype(np.float32).astype(np.float64), prev.astype(np.float32).astype(np.float64)
    xq = np.stack([orc.quant_array(v, quant) for v in x])
    pq = np.stack([orc.quant_array(v, quant) for v in prev])
    tdt = torch.bfloat16 if bf16 else torch.float32
    # the library validates cin against the frame's 3 channels for in0 = -1, so give the conv a
    # producer with the right shape when cin != 3: a 1x1 conv from the frame stands in
    if cin == 3:
        net, li, fh, fw = layers, 0, hi, wi
        ws, bs = [wts], [bias]
    else:
        nb = nets.NetBuilder(hi, wi)
        a = nb.conv(-1, cin, 1, 1, 0)
        nb.conv(a, cout, k, s, p, relu)
        net, li, fh, fw = nb.layers, 1, hi, wi
        ws = [np.zeros((cin, 1, 1, 3), np.float32), wts]
        bs = [np.zeros(cin, np.float32), bias]
    dc = DeepCache(fw, fh, net, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, max_regions=8)
    try:
        regs = torch.zeros((S, dc.max_regions, 6), dtype=torch.int32)
        per_stream, counts = [], []
        for s_ in range(S):
            n = min(dc.max_regions, 6)
            # disjoint rectangles: split the output into a grid of cells, one rectangle inside each
            r = np.zeros(n, orc.REGION_DTYPE)
            cw, ch = L["out_w"] // 3, L["out_h"] // 2
            for i in range(n):
                cx, cy = (i % 3) * cw, (i // 3) * ch
                w_ = int(g.integers(1, cw + 1)); h_ = int(g.integers(1, ch + 1))
                x0 = cx + int(g.integers(0, cw - w_ + 1)); y0 = cy + int(g.integers(0, ch - h_ + 1))
                sx = int(g.integers(0, L["out_w"] - w_ + 1)); sy = int(g.integers(0, L["out_h"] - h_ + 1))
                r[i] = (x0, y0, w_, h_, sx, sy)
            if s_ == 1:
                r[2] = (0, 0, 0, 0, 0, 0)          # a vanished slot
            per_stream.append(r); counts.append(n)
            regs[s_, :n] = torch.from_numpy(np.ascontiguousarray(r).view(np.int32).reshape(n, 6))
        xin = torch.from_numpy(xq).to(tdt).cuda()
        pin = torch.from_numpy(pq).to(tdt).cuda()
        full = dc.conv_partial(li, xin)
        part = dc.conv_partial(li, xin, pin, regs.cuda(), torch.tensor(counts, dtype=torch.int32).cuda())
        wq = orc.quant_array(wts, quant)
        for s_ in range(S):
            want_full, _ = orc.conv_reuse(xq[s_], L, wq, bias, quant)
            want, reused = orc.conv_reuse(xq[s_], L, wq, bias, quant, pq[s_], per_stream[s_])
            U.assert_map_close(full[s_], want_full, bf16, "full")
            U.assert_map_close(part[s_], want, bf16, "partial")
            if bf16:
                U.assert_map_close_per_element(full[s_], want_full, "full, per element")
            m = reused.astype(bool)
            got = part[s_].float().cpu().numpy().astype(np.float64)
            assert m.any() and np.array_equal(got[m], want[m]), "reused pixels must be bit-equal copies of the cached map"
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


def test_conv_partial_ignores_rectangles_outside_the_map():
    """A caller's rectangle that leaves the map on either side, or a count beyond max_regions, must not become an
    out-of-bounds access: such rectangles are not reused (their pixels are convolved) and the status word says so."""
    g = rng(77)
    hi, wi, cout = 37, 45, 16
    b = nets.NetBuilder(hi, wi, 3)
    b.conv(-1, cout, 3, 1, 1, 1)
    L = b.layers[0]
    wts = g.normal(0, 0.2, size=(cout, 3, 3, 3)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    x = g.normal(size=(1, hi, wi, 3)).astype(np.float32).astype(np.float64)
    prev = g.normal(size=(1, hi, wi, cout)).astype(np.float32).astype(np.float64)
    dc = DeepCache(wi, hi, [dict(L)], [wts], [bias], n_streams=1, block=16, search_range=4, dtype=B.DC_FP32, max_regions=8)
    try:
        good = (4, 5, 10, 9, 7, 2)
        bad = [(30, 3, 10, 6, 40, 3),            # cached side leaves the map on the right
               (2, 30, 5, 6, 2, -1),             # cached side starts above the map
               (-3, 20, 8, 4, 0, 20),            # current side starts left of the map
               (20, 20, 100, 4, 0, 0),           # wider than the map
               (10, 25, 2 ** 30, 2 ** 30, 5, 5),  # sizes that would overflow a sum
               (12, 12, -4, 3, 1, 1)]            # negative width: an empty slot, not an error
        regs = torch.zeros((1, dc.max_regions, 6), dtype=torch.int32)
        for i, r in enumerate([good] + bad):
            regs[0, i] = torch.tensor(r, dtype=torch.int32)
        xin, pin = torch.from_numpy(x).float().cuda(), torch.from_numpy(prev).float().cuda()
        # a count far beyond the table: cut to max_regions (the eighth slot is all zeros)
        part = dc.conv_partial(0, xin, pin, regs.cuda(), torch.tensor([1000], dtype=torch.int32).cuda())
        only_good = np.zeros(1, orc.REGION_DTYPE); only_good[0] = good
        want, reused = orc.conv_reuse(x[0], L, wts, bias, orc.QUANT_NONE, prev[0], only_good)
        U.assert_map_close(part[0], want, False, "bad rectangles ignored")
        m = reused.astype(bool)
        assert np.array_equal(part[0].cpu().numpy().astype(np.float64)[m], want[m])
        assert dc.status() == B.DC_ERR_ARG
        dc.reset()
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("dtype,cin,cout,k", [(B.DC_FP32, 16, 32, 3), (B.DC_FP32, 8, 12, 1), (B.DC_FP32, 8, 20, 0), (B.DC_BF16, 24, 16, 3), (B.DC_BF16, 64, 64, 3)])
def test_conv_partial_takes_maps_at_any_element(dtype, cin, cout, k):
    """A caller's maps that start one element past an aligned address: the kernels that move vectors leave them to the one
    that does not; where only those exist, and for the reuse copy, the call is refused before any launch."""
    S, hi, wi = 2, 9, 11
    nb = nets.NetBuilder(hi, wi)
    a = nb.conv(-1, cin, 1, 1, 0)
    nb.conv(a, cout, k, 1, k // 2, 1) if k else nb.fc(a, cout, relu=1)
    ws, bs = nets.random_weights(nb.layers, 5)
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, max_regions=4)
    try:
        shape = dc.out_shape(1)
        x = torch.from_numpy(rng(cin).normal(size=(S, hi, wi, cin)).astype(np.float32)).to(dc.tdtype).cuda()
        want = dc.conv_partial(1, x)
        xs = torch.zeros(x.numel() + 8, dtype=dc.tdtype, device="cuda")[1:1 + x.numel()].view(x.shape)
        xs.copy_(x)
        out = torch.zeros(want.numel() + 8, dtype=dc.tdtype, device="cuda")[1:1 + want.numel()].view(shape)
        regs, n = torch.zeros((S, 4, 6), dtype=torch.int32, device="cuda"), torch.zeros(S, dtype=torch.int32, device="cuda")
        ok = torch.zeros_like(want)
        if B.dc_cache_layer_conv_scheme(dc.handle, 1) > 0:
            for i, o in ((x, out), (xs, ok)):
                with pytest.raises(B.DeepCacheError) as e:
                    B.dc_conv_partial(dc.handle, 1, i, None, None, None, o)
                assert e.value.status == B.DC_ERR_ARG
        else:
            for i, o in ((xs, ok), (x, out), (xs, out)):
                o.zero_()
                B.dc_conv_partial(dc.handle, 1, i, None, None, None, o)
                U.assert_map_close(o, want.float().cpu().numpy().astype(np.float64), dtype == B.DC_BF16, "unaligned")
        for p_, o in ((want, out), (out, ok)):
            with pytest.raises(B.DeepCacheError) as e:
                B.dc_conv_partial(dc.handle, 1, x, p_, regs, n, o)
            assert e.value.status == B.DC_ERR_ARG
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


def test_conv_partial_with_rectangles_where_propagation_left_them():
    """dc_propagate_regions leaves a caller's rectangles in the cache's table (dc_cache_layer_regions): a convolution given
    that table reuses them, although no rectangle of the last frame was left at the layer."""
    S, hi, wi = 2, 48, 64
    nb = nets.NetBuilder(hi, wi)
    nb.conv(nb.conv(-1, 32, 3, 1, 1), 64, 3, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 9)
    g = rng(41)
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
    try:
        for _ in range(2):                                          # two frames of noise: nothing matches
            _, st = dc.infer_frame(g.integers(0, 256, size=(S, hi, wi, 3), dtype=np.uint8), want_stats=True)
        assert not st[0].refreshed and st[0].n_regions == 0
        regs = torch.tensor([[[4, 4, 40, 33, 5, 6]] + [[0] * 6] * 3, [[0, 0, 64, 48, 0, 0]] + [[0] * 6] * 3], dtype=torch.int32).cuda()
        n = torch.tensor([1, 1], dtype=torch.int32).cuda()
        out, _ = dc.propagate_regions(regs, n)
        x = torch.from_numpy(g.normal(size=(S, hi, wi, 32)).astype(np.float32)).cuda()
        prev = torch.from_numpy(g.normal(size=(S, hi, wi, 64)).astype(np.float32)).cuda()
        ptr, _ = B.dc_cache_layer_regions(dc.handle, 1)
        table = device_view(ptr, (S, dc.max_regions, 6), torch.int32, dc.device)
        assert torch.equal(table, out[1])
        assert torch.equal(dc.conv_partial(1, x, prev, table, n), dc.conv_partial(1, x, prev, out[1].contiguous(), n))
    finally:
        dc.close()


@pytest.mark.parametrize("dtype", [B.DC_FP32, B.DC_BF16])
def test_conv_partial_in_a_graph_launched_again(dtype):
    """One dc_conv_partial captured and launched several times, other calls between: every launch counts its tiles from zero."""
    S, hi, wi = 2, 50, 70
    nb = nets.NetBuilder(hi, wi)
    nb.conv(nb.conv(-1, 64, 1, 1, 0), 64, 3, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 9)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, max_regions=4)
        g = rng(31)
        x, prev = (torch.from_numpy(g.normal(size=(S, hi, wi, 64)).astype(np.float32)).to(dc.tdtype).cuda() for _ in range(2))
        regs = torch.tensor([[[3, 4, 40, 33, 5, 6]] + [[0] * 6] * 3, [[0, 0, 70, 50, 0, 0]] + [[0] * 6] * 3], dtype=torch.int32).cuda()
        n = torch.tensor([1, 1], dtype=torch.int32).cuda()
        want, other = dc.conv_partial(1, x, prev, regs, n), dc.conv_partial(1, prev, x, regs, n)
        out = torch.zeros_like(want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        B.dc_conv_partial(dc.handle, 1, x, prev, regs, n, out)
    with torch.cuda.stream(stream):
        for k in range(5):
            out.zero_()
            graph.replay()
            stream.synchronize()
            assert torch.equal(out, want), f"launch {k}"
            if k == 2:
                assert torch.equal(dc.conv_partial(1, prev, x, regs, n), other)
        assert dc.status() == B.DC_OK
        dc.close()


@pytest.mark.parametrize("scheme", [1, 2, 3, 4, 5, 6, 7, 8, 9])
def test_conv_schemes_forced(scheme, monkeypatch):
    """Every operand scheme of the tensor-core convolution (tap by tap, patch, column slabs; one or two tiles per
    item; column slabs on CTA pairs; tap by tap on flat tiles) on layers it can take: VGG-shaped 3x3 layers, a 5x5 layer and odd map sizes,
    through cached frames."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    b = nets.NetBuilder(45, 53)
    x = b.conv(-1, 64, 3, 1, 1)
    x = b.conv(x, 64, 3, 1, 1)
    x = b.conv(x, 128, 5, 1, 2)
    x = b.maxpool(x, 2, 2)
    x = b.conv(x, 256, 3, 1, 1)
    b.conv(x, 256, 3, 1, 1, relu=0)
    w = configs.small_cnn_stream()
    w.layers, w.dtype, w.width, w.height = b.layers, configs.DTYPE_BF16, 53, 45
    inner = w.make_streams
    w.make_streams = lambda s, f, first=0: _cropped(inner(s, f), 45, 53)
    U.run_stream_parity(w, 2, [0, 1, 2])


# ------------------------------------------------------------------ dc_infer_frame
@pytest.mark.parametrize("first,second", [((60, 70), (24, 30)), ((24, 30), (60, 70))])
def test_infer_with_two_resized_inputs(first, second):
    """Two area resizes to different sizes, each read by a convolution over three channels: a resize fills the operand
    copy of its own reader only."""
    b = nets.NetBuilder(80, 96)
    for h, w in (first, second):
        b.conv(b.resize_area(-1, h, w), 64, 3, 1, 1)
    w = configs.small_cnn_stream()
    w.layers, w.dtype, w.width, w.height = b.layers, configs.DTYPE_BF16, 96, 80
    inner = w.make_streams
    w.make_streams = lambda s, f, first=0: _cropped(inner(s, f), 80, 96)
    U.run_stream_parity(w, 2, [0, 1, 2])


def test_infer_workload_1():
    U.run_stream_parity(configs.WORKLOADS[1](), 1, [0, 1])


def test_infer_workload_2_through_an_expiry():
    U.run_stream_parity(configs.WORKLOADS[2](), 1, list(range(12)))


def test_infer_workload_3_alexnet_bf16():
    U.run_stream_parity(configs.WORKLOADS[3](), 1, list(range(12)))


@pytest.mark.parametrize("dtype", [configs.DTYPE_FP32, configs.DTYPE_BF16])
def test_infer_alexnet_with_grouped_convolutions(dtype):
    """The AlexNet trunk with two channel groups in its second, fourth and fifth convolutions: every layer's
    rectangles, reuse ratios and maps against the oracle, cached frames included."""
    w = configs.alexnet_stream(grouped=True, dtype=dtype)
    U.run_stream_parity(w, 1, list(range(4)))
    # in bfloat16 every convolution, the grouped ones included, runs on the tensor-core kernels (one launch per group)
    dc = DeepCache.from_workload(w, n_streams=1)
    try:
        schemes = [B.dc_cache_layer_conv_scheme(dc.handle, i) for i, l in enumerate(w.layers) if l["kind"] == 0]
        assert len(schemes) == 5 and any(l.get("groups", 1) > 1 for l in w.layers)
        assert all(v >= 1 for v in schemes) if dtype == configs.DTYPE_BF16 else all(v == 0 for v in schemes)
    finally:
        dc.close()


def test_infer_workload_4_resnet50_bf16():
    U.run_stream_parity(configs.WORKLOADS[4](), 1, list(range(4)))


@pytest.mark.parametrize("wid,frames", [(3, [0, 1, 2]), (4, [0, 1])])
def test_infer_small_map_trunks_three_streams(wid, frames):
    """The AlexNet and ResNet-50 trunks with three streams in one cache: tiles of their small maps may hold pixels of
    two streams (flat tiles), and their strided first layers run on the space-to-depth copy; every layer's map of
    every stream against the oracle."""
    U.run_stream_parity(configs.WORKLOADS[wid](), 3, frames)


def test_infer_workload_5_two_streams():
    """Full-HD matching, area resize to 224x224, VGG-16 trunk; 2 of the 32 streams, frames 0-2."""
    U.run_stream_parity(configs.WORKLOADS[5](), 2, [0, 1, 2])


def test_infer_workload_5_full_batch_sampled_streams():
    """The benchmark's own configuration: all 32 full-HD streams in one cache, the loop bench.py times
    (dc_infer_frame(t), then dc_lookahead_frame(t + 1)), frames 0-3.  The oracle follows three of the streams
    (first, one in the middle, last): motion vector, counts, frame rectangles and the final map of every frame."""
    w = configs.WORKLOADS[5]()
    S, n_frames, sample = w.n_streams, 4, (0, 13, w.n_streams - 1)
    bf16 = w.dtype == configs.DTYPE_BF16
    sb = w.streams(S, n_frames)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).cuda() for i in range(n_frames)]
    oracles = dict(zip(sample, U.make_oracles(w, len(sample))))
    dc = DeepCache.from_workload(w, n_streams=S)
    try:
        pitch = w.width * 3
        for i in range(n_frames):
            out, st = dc.infer_frame(frames[i], want_stats=True)
            out = out.clone()
            regs0, _ = dc.layer_regions(-1)
            regs0 = regs0.clone()
            if i + 1 < n_frames:
                B.dc_lookahead_frame(dc.handle, frames[i + 1], pitch)
            for s in sample:
                o = oracles[s].infer_frame(sb.frame(i, s))
                what = f"frame {i} stream {s} of {S}"
                assert bool(st[s].refreshed) == o["refreshed"], what
                if not o["refreshed"]:
                    m = o["match"]
                    assert (st[s].mvx, st[s].mvy, st[s].k_passed) == (m["M"][0], m["M"][1], m["K"]), what
                    assert st[s].n_matched == int(m["matched"].sum()) and st[s].n_regions == len(m["regions"]), what
                    U.assert_regions_equal(U.regions_np(regs0[s, :len(m["regions"])]), m["regions"], what + " frame rectangles")
                U.assert_map_close(out[s], o["out"], bf16, what + " output")
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


def test_infer_identical_frames_and_reset():
    w = configs.WORKLOADS[2]()
    f = w.streams(1, 1).frame(0)
    dc = DeepCache.from_workload(w)
    try:
        a = dc.infer_frame(f).clone()
        b, st = dc.infer_frame(f, want_stats=True)
        assert not st[0].refreshed and (st[0].mvx, st[0].mvy) == (0, 0) and st[0].n_regions == 1
        assert torch.equal(a, b)                     # everything reusable was copied, the rest recomputed identically
        dc.reset()
        c, st = dc.infer_frame(f, want_stats=True)
        assert st[0].refreshed and torch.equal(a, c)
    finally:
        dc.close()


def test_infer_host_buffers_with_and_without_prefetch():
    """dc_infer_frame_host (host frames in, last map out) with the next frame prefetched, without, and with a
    prefetch that is then not used: all equal dc_infer_frame on device buffers, bit for bit."""
    w = configs.WORKLOADS[2]()
    sb = w.streams(1, 6)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).pin_memory() for i in range(6)]
    ref = DeepCache.from_workload(w)
    dc = DeepCache.from_workload(w)
    try:
        pitch = w.width * 3
        out_host = torch.empty(ref.out_shape(-1), dtype=torch.float32).pin_memory()
        B.dc_prefetch_frame_host(dc.handle, frames[0].data_ptr(), pitch)
        for i in range(6):
            want = ref.infer_frame(frames[i].cuda())
            if i in (0, 1, 3):                        # the usual loop: prefetch the next frame, then compute this one
                B.dc_prefetch_frame_host(dc.handle, frames[i + 1].data_ptr(), pitch)
            B.dc_infer_frame_host(dc.handle, frames[i].data_ptr(), pitch, out_host.data_ptr())
            assert torch.equal(out_host, want.cpu()), f"frame {i}"
        # a third pending prefetch is refused
        B.dc_prefetch_frame_host(dc.handle, frames[0].data_ptr(), pitch)
        B.dc_prefetch_frame_host(dc.handle, frames[1].data_ptr(), pitch)
        with pytest.raises(B.DeepCacheError) as e:
            B.dc_prefetch_frame_host(dc.handle, frames[2].data_ptr(), pitch)
        assert e.value.status == B.DC_ERR_STATE
        assert dc.status() == B.DC_OK
    finally:
        ref.close(); dc.close()


def test_infer_host_drops_a_prefetch_that_is_announced():
    """A frame that was not prefetched while both buffers hold prefetches, the first of them announced already: the dropped one's copy and match are
    not taken for it, and the frames behind it, prefetched and not, come out as from device buffers."""
    w = configs.WORKLOADS[2]()
    sb = w.streams(1, 6)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).pin_memory() for i in range(6)]
    ref, dc = DeepCache.from_workload(w), DeepCache.from_workload(w)
    try:
        out = torch.empty(ref.out_shape(-1), dtype=torch.float32).pin_memory()

        def prefetch(i):
            B.dc_prefetch_frame_host(dc.handle, frames[i].data_ptr(), w.width * 3)

        def infer(i):
            want = ref.infer_frame(frames[i].cuda())
            B.dc_infer_frame_host(dc.handle, frames[i].data_ptr(), w.width * 3, out.data_ptr())
            assert torch.equal(out, want.cpu()), f"frame {i}"

        infer(5)
        prefetch(0)
        infer(1)                                      # announces frame 0
        prefetch(2)
        infer(3)                                      # takes frame 0's buffer, announces frame 2
        infer(2)
        infer(4)
        assert dc.status() == B.DC_OK
    finally:
        ref.close(); dc.close()


def test_region_overflow_sets_the_status_word():
    """More rectangles than max_regions: the extra ones are dropped and the device status word says so."""
    prev = rng(2).integers(0, 256, size=(64, 64, 3), dtype=np.uint8)
    cur = prev.copy()
    cur[::16, :] = 255 - cur[::16, :]                 # ruin every other 8-px block row: matched rows alternate
    cur[:, 24:32] = 255 - cur[:, 24:32]               # and one block column: two runs per matched row
    layers = nets.single_conv(64, 64)
    ws, bs = nets.random_weights(layers, 1)
    want = orc.match_blocks(cur, prev, 8, 2, orc.SEARCH_DS, 20.0)
    assert len(want["regions"]) > 2
    dc = DeepCache(64, 64, layers, ws, bs, block=8, search_range=2, max_regions=2)
    try:
        dc.set_key(prev)
        got = dc.match_blocks(cur)
        assert int(got["n_regions"][0]) == 2
        U.assert_regions_equal(U.regions_np(got["regions"][0, :2]), want["regions"][:2], "kept rectangles")
        assert dc.status() == B.DC_ERR_OVERFLOW
        dc.reset()
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("scheme", [5, 7])
@pytest.mark.parametrize("hi,wi,cin,cout,k,p", [(14, 14, 256, 512, 3, 1), (28, 28, 128, 256, 3, 1), (17, 23, 64, 128, 5, 2), (9, 40, 128, 256, 1, 0)])
def test_conv_wide_layers_on_cta_pairs(scheme, hi, wi, cin, cout, k, p, monkeypatch):
    """The wide layers (128 - 512 output channels) forced onto the CTA-pair kernel (7), and onto the single-CTA column-slab
    kernel (5) for comparison: full convolution and partial convolution with an odd number of dirty tiles."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    _one_layer_full_and_partial(hi, wi, cin, cout, k, 1, p, 3, scheme)


@pytest.mark.parametrize("hi,wi,cin,cout,k,st,p,S", [
    (7, 7, 512, 64, 3, 1, 1, 1),         # one tile, more steps per CTA than ring slots
    (7, 7, 128, 256, 1, 1, 0, 5),        # two steps in all: clusters of two
    (14, 14, 64, 96, 3, 2, 1, 3),        # strided, 32-channel blocks, 7 x 7 output
    (13, 21, 48, 64, 3, 1, 1, 2),        # 16-channel steps, 32-byte operand rows
    (17, 9, 32, 32, 5, 1, 2, 2),         # 64-byte operand rows, partial tiles
])
def test_conv_on_clusters(hi, wi, cin, cout, k, st, p, S, monkeypatch):
    """Few tiles: the reduction split over a cluster of CTAs, full and partial convolution (scheme 10)."""
    monkeypatch.setenv("DC_CONV_SCHEME", "10")
    _one_layer_full_and_partial(hi, wi, cin, cout, k, st, p, S, 10)


@pytest.mark.parametrize("what", ["add", "groups", "last block filled up", "strided"])
def test_conv_narrow_blocks(what, monkeypatch, capfd):
    """Tap-by-tap layers in blocks of 32 and of 64 output channels: the bits of the widest blocks, full and partial."""
    nb = nets.NetBuilder(28, 30)
    x = nb.conv(-1, 256, 3, 1, 1)
    if what == "add":                                                # taken along by the convolution before it
        nb.add(nb.conv(nb.conv(x, 64, 1, 1, 0), 256, 1, 1, 0, relu=0), x)
    elif what == "groups":
        nb.conv(x, 512, 3, 1, 1, groups=2)
    elif what == "strided":
        nb.conv(x, 256, 3, 2, 1)
    else:
        nb.conv(x, 248, 3, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 7)
    g = rng(3)
    f0 = g.integers(0, 256, (1, 28, 30, 3), dtype=np.uint8)
    f1 = f0.copy()
    f1[:, 9:17, 4:12] ^= 0x5A
    monkeypatch.setenv("DC_VERBOSE", "1")
    monkeypatch.setenv("DC_CONV_SCHEME", "1")
    outs = {}
    for width in (0, 32, 64):
        monkeypatch.setenv("DC_CONV_BLOCK", str(width))
        capfd.readouterr()
        dc = DeepCache(30, 28, nb.layers, ws, bs, block=4, search_range=2, dtype=B.DC_BF16)
        try:
            chosen = [l for l in capfd.readouterr().err.splitlines() if ": chose code 1, " in l]
            assert width == 0 or any(f" {width} channels per block" in l for l in chosen), chosen
            outs[width] = [dc.infer_frame(f).clone() for f in (f0, f1)] + [dc.layer_map(l) for l in range(len(nb.layers))]
            assert dc.status() == B.DC_OK
        finally:
            dc.close()
    for width in (32, 64):
        for a, b in zip(outs[0], outs[width]):
            assert torch.equal(a, b), f"{width} channels per block"


@pytest.mark.parametrize("scheme", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("hi,wi,cin,cout,k,st,p,S", [
    (33, 18, 32, 16, 3, 1, 1, 3),        # half of the only block
    (16, 9, 64, 40, 5, 1, 2, 2),         # one 16-byte piece of the second
    (20, 24, 48, 120, 3, 1, 1, 1),       # blocks of 128, the last 8 channels absent
    (30, 33, 16, 24, 3, 2, 1, 2),        # strided: tap by tap alone
])
def test_conv_channels_filled_up_to_blocks(scheme, hi, wi, cin, cout, k, st, p, S, monkeypatch):
    """Output channels that are no multiple of 32 on the tensor-core kernels."""
    if st > 1 and scheme > 2:
        pytest.skip("patches and slabs take stride 1 alone")
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    _one_layer_full_and_partial(hi, wi, cin, cout, k, st, p, S, scheme, forced=True)


@pytest.mark.parametrize("st", [1, 2])
def test_conv_channels_filled_up_take_maps_at_any_element(st):
    nb = nets.NetBuilder(21, 18)
    nb.conv(nb.conv(-1, 32, 1, 1, 0), 24, 3, st, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 5)
    dc = DeepCache(18, 21, nb.layers, ws, bs, n_streams=2, block=16, search_range=4, dtype=B.DC_BF16, max_regions=4)
    try:
        assert B.dc_cache_layer_conv_scheme(dc.handle, 1) > 0
        x = torch.from_numpy(rng(3).normal(size=(2, 21, 18, 32)).astype(np.float32)).to(dc.tdtype).cuda()
        want = dc.conv_partial(1, x)
        off = lambda t: torch.zeros(t.numel() + 8, dtype=dc.tdtype, device="cuda")[1:1 + t.numel()].view(t.shape)
        xs = off(x)
        xs.copy_(x)
        for i, o in ((xs, torch.zeros_like(want)), (x, off(want)), (xs, off(want))):
            B.dc_conv_partial(dc.handle, 1, i, None, None, None, o)
            U.assert_map_close(o, want.float().cpu().numpy().astype(np.float64), True, "unaligned")
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("scheme", [8, 9])
@pytest.mark.parametrize("hi,wi,cin,cout,k,st,p,S", [
    (7, 7, 128, 256, 3, 1, 1, 5),        # 7 pieces per stream: every tile holds pieces of two or three streams
    (14, 14, 256, 512, 3, 1, 1, 3),      # two pieces per row
    (13, 13, 64, 96, 3, 1, 1, 4),        # a cut last piece in every row; 32-channel blocks
    (27, 27, 32, 64, 5, 2, 2, 3),        # a strided layer (14 x 14 output), 64-byte operand rows
    (9, 40, 128, 256, 1, 1, 0, 3),       # 1 x 1
    (3, 5, 64, 64, 3, 1, 1, 1),          # one tile, mostly absent
])
def test_conv_flat_tiles_across_rows_and_streams(scheme, hi, wi, cin, cout, k, st, p, S, monkeypatch):
    """Small maps on tiles made of 16 row pieces of 8 pixels that run on across rows and streams (scheme 8; 9 with two
    tiles per item): the reuse bitmap, the dirty list and the copies then follow that numbering too."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    _one_layer_full_and_partial(hi, wi, cin, cout, k, st, p, S, scheme)


@pytest.mark.parametrize("scheme", [8, 9])
@pytest.mark.parametrize("hi,wi,cin,cout,st,S", [
    (7, 7, 128, 96, 1, 5),               # rows of one group, the last tile not full
    (14, 13, 64, 128, 1, 3),             # two groups, the second cut
    (28, 56, 32, 64, 2, 2),              # every other row and column of the stack, four groups
    (9, 120, 16, 32, 1, 2),              # a row is a tile
])
def test_conv_flat_tiles_as_whole_rows(scheme, hi, wi, cin, cout, st, S, monkeypatch):
    """1 x 1 layers whose flat tiles are whole rows of the stacked streams."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    _one_layer_full_and_partial(hi, wi, cin, cout, 1, st, 0, S, scheme)


@pytest.mark.parametrize("scheme", [8, 9])
@pytest.mark.parametrize("hi,wi,cin,cout,k,st,p,S", [
    (7, 7, 64, 128, 3, 1, 1, 5),         # two images a tile, 14 of 16 groups, the last tile half full
    (4, 6, 32, 64, 3, 1, 1, 9),          # four images
    (3, 13, 64, 32, 5, 1, 2, 5),         # rows of two groups, two images
    (14, 14, 128, 64, 3, 2, 1, 4),       # strided
    (16, 8, 64, 64, 3, 1, 1, 2),         # an image is a tile
    (9, 8, 64, 64, 3, 1, 1, 3),          # an image is no whole part of a tile: groups one by one
    (1, 5, 16, 32, 2, 1, 1, 7),          # a last row that reads padding alone
])
def test_conv_flat_tiles_as_whole_images(scheme, hi, wi, cin, cout, k, st, p, S, monkeypatch):
    """Small maps under kernels of more than one tap: flat tiles of whole images."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    _one_layer_full_and_partial(hi, wi, cin, cout, k, st, p, S, scheme)


@pytest.mark.parametrize("hi,wi,cin,cout,k,S,groups", [
    (28, 28, 128, 256, 3, 2, 1),         # two chunks of 64 channels, CTA pairs too
    (13, 13, 96, 64, 5, 3, 1),           # 32-channel steps, a half-empty last chunk
    (17, 23, 96, 128, 5, 1, 2),          # 48 channels per group: 16-channel steps
    (9, 40, 192, 32, 3, 1, 1),           # the narrowest channel block
])
def test_conv_schemes_agree_bit_for_bit(hi, wi, cin, cout, k, S, groups, monkeypatch):
    """What a layer was timed with must not show in its output: all operand schemes but the clusters sum in one order."""
    g = rng(hi + cin + k)
    nb = nets.NetBuilder(hi, wi)
    nb.conv(nb.conv(-1, cin, 1, 1, 0), cout, k, 1, k // 2, 1, groups=groups)
    ws, bs = nets.random_weights(nb.layers, 7)
    x = torch.from_numpy(g.normal(size=(S, hi, wi, cin)).astype(np.float32)).to(torch.bfloat16).cuda()
    want, taken = None, set()
    for scheme in range(1, 10):
        monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
        dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_BF16)
        out = dc.conv_partial(1, x)
        taken.add(B.dc_cache_layer_conv_scheme(dc.handle, 1))
        want = out if want is None else want
        assert torch.equal(out, want), f"scheme {scheme}"
        dc.close()
    assert len(taken) >= 6


@pytest.mark.parametrize("net,S", [("resnet50", 1), ("resnet50", 4), ("alexnet", 1), ("alexnet_grouped", 3)])
def test_caches_of_one_configuration_repeat_themselves(net, S):
    """Three caches, each timing its kernels anew: the same maps at every layer, bit for bit."""
    layers = nets.resnet50_trunk(224, 224) if net == "resnet50" else nets.alexnet_trunk(227, 227, grouped=net == "alexnet_grouped")
    W = layers[0]["out_w"] * 2 if net == "resnet50" else 227
    ws, bs = nets.random_weights(layers, 4)
    g = rng(S)
    frames = [torch.from_numpy(g.integers(0, 256, size=(S, W, W, 3), dtype=np.uint8)).cuda() for _ in range(2)]
    frames[1][:, : W // 2] = frames[0][:, : W // 2]
    maps = None
    for _ in range(3):
        dc = DeepCache(W, W, layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_BF16)
        for f in frames:
            dc.infer_frame(f)
        got = [dc.layer_map(i) for i in range(len(layers))]
        maps = maps or got
        assert all(torch.equal(a, b) for a, b in zip(got, maps))
        dc.close()


@pytest.mark.parametrize("S", [1, 3])
def test_residual_add_in_the_cluster_kernel(S, monkeypatch):
    """Residual blocks whose last convolution runs on clusters and does the add as well: full frames, cached frames (reused
    pixels are added too), the add with and without ReLU, its other operand a convolution or an earlier add."""
    monkeypatch.setenv("DC_CONV_SCHEME", "10")
    b = nets.NetBuilder(45, 53)
    x = b.conv(-1, 64, 3, 2, 1)
    last = []
    for relu, proj in ((1, False), (0, True), (1, False)):
        y = b.conv(b.conv(x, 32, 1, 1, 0), 64, 3, 1, 1, 0)
        other = b.conv(x, 64, 3, 1, 1, 0) if proj else x           # a projection comes later than the branch and takes the add
        last.append(max(y, other))
        x = b.add(y, other, relu)
    w = configs.small_cnn_stream()
    w.layers, w.dtype, w.width, w.height, w.expire_n = b.layers, configs.DTYPE_BF16, 53, 45, 3
    inner = w.make_streams
    w.make_streams = lambda s, f, first=0: _cropped(inner(s, f), 45, 53)
    dc = DeepCache.from_workload(w, n_streams=S)
    assert all(B.dc_cache_layer_conv_scheme(dc.handle, i) == 10 for i in last)
    dc.close()
    U.run_stream_parity(w, S, [0, 1, 2, 3, 4])


@pytest.mark.parametrize("scheme,S", [(1, 1), (1, 9), (8, 4)])
def test_residual_add_in_the_tap_by_tap_kernel(scheme, S, monkeypatch):
    """The same with few tiles tap by tap: whole tiles and flat ones, the add with and without ReLU, after a projection too; as many
    streams as leave every tile an SM (9: 72 or 144 items) take the add along, twice as many do not."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    b = nets.NetBuilder(45, 53)
    x = b.conv(-1, 64, 3, 2, 1)
    for relu, proj in ((1, False), (0, True), (1, False)):
        y = b.conv(b.conv(x, 32, 1, 1, 0), 64, 1, 1, 0, 0)
        x = b.add(y, b.conv(x, 64, 1, 1, 0, 0) if proj else x, relu)
    w = configs.small_cnn_stream()
    w.layers, w.dtype, w.width, w.height, w.expire_n = b.layers, configs.DTYPE_BF16, 53, 45, 3
    inner = w.make_streams
    w.make_streams = lambda s, f, first=0: _cropped(inner(s, f), 45, 53)
    U.run_stream_parity(w, S, [0, 1, 2, 3])
    if S == 9:
        U.run_stream_parity(w, S + 10, [0, 1])


def test_first_frame_of_a_cache_reads_the_weights_of_its_choice():
    """The tuner packs weights for the widths it tries; the first frame, launched at once, must find the final packing: the
    same maps as the same frame given to the warm cache."""
    b = nets.NetBuilder(57, 57)
    x = b.conv(-1, 64, 3, 1, 1)
    for cout in (128, 128, 256, 256):
        x = b.conv(x, cout, 3, 1, 1)
    ws, bs = nets.random_weights(b.layers, 12)
    f = torch.from_numpy(rng(8).integers(0, 256, size=(16, 57, 57, 3), dtype=np.uint8)).cuda()
    for _ in range(8):
        dc = DeepCache(57, 57, b.layers, ws, bs, n_streams=16, block=16, search_range=4, dtype=B.DC_BF16)
        dc.infer_frame(f, want_out=False)
        first = [dc.layer_map(i) for i in range(len(b.layers))]
        dc.reset()
        dc.infer_frame(f, want_out=False)
        assert all(torch.equal(a, dc.layer_map(i)) for i, a in enumerate(first))
        dc.close()


def _one_layer_full_and_partial(hi, wi, cin, cout, k, st, p, S, scheme, forced=False):
    g = rng(hi * 7 + cout)
    nb = nets.NetBuilder(hi, wi)
    a = nb.conv(-1, cin, 1, 1, 0)
    nb.conv(a, cout, k, st, p, 1)
    L = nb.layers[1]
    wts = g.normal(0, np.sqrt(2.0 / (k * k * cin)), size=(cout, k, k, cin)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    ws = [np.zeros((cin, 1, 1, 3), np.float32), wts]
    bs = [np.zeros(cin, np.float32), bias]
    xq = np.stack([orc.quant_array(g.normal(size=(hi, wi, cin)), orc.QUANT_BF16) for _ in range(S)])
    pq = np.stack([orc.quant_array(g.normal(size=(L["out_h"], L["out_w"], cout)), orc.QUANT_BF16) for _ in range(S)])
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_BF16, max_regions=4)
    try:
        if forced or scheme >= 8:
            assert B.dc_cache_layer_conv_scheme(dc.handle, 1) == scheme
        xin = torch.from_numpy(xq).to(torch.bfloat16).cuda()
        pin = torch.from_numpy(pq).to(torch.bfloat16).cuda()
        full = dc.conv_partial(1, xin)
        # one rectangle that covers the whole map of stream 1 (its tiles are clean: the dirty count becomes odd for
        # most shapes) and a small one in stream 0
        regs = torch.zeros((S, dc.max_regions, 6), dtype=torch.int32)
        counts = torch.zeros(S, dtype=torch.int32)
        ow, oh = L["out_w"], L["out_h"]
        regs[0, 0] = torch.tensor([1, 2, min(5, ow - 2), min(4, oh - 2), 2, 1] if oh >= 4 else [1, 1, ow - 1, oh - 1, 0, 0], dtype=torch.int32)
        counts[0] = 1
        if S > 1:
            regs[1, 0] = torch.tensor([0, 0, ow, oh, 0, 0], dtype=torch.int32)
            counts[1] = 1
        part = dc.conv_partial(1, xin, pin, regs.cuda(), counts.cuda())
        wq = orc.quant_array(wts, orc.QUANT_BF16)
        for s_ in range(S):
            r = np.zeros(1, orc.REGION_DTYPE)
            r[0] = tuple(int(v) for v in regs[s_, 0])
            want_full, _ = orc.conv_reuse(xq[s_], L, wq, bias, orc.QUANT_BF16)
            want, reused = orc.conv_reuse(xq[s_], L, wq, bias, orc.QUANT_BF16, pq[s_], r[:int(counts[s_])])
            U.assert_map_close(full[s_], want_full, True, f"full, stream {s_}")
            U.assert_map_close_per_element(full[s_], want_full, f"full, per element, stream {s_}")
            U.assert_map_close(part[s_], want, True, f"partial, stream {s_}")
            m = reused.astype(bool)
            got = part[s_].float().cpu().numpy().astype(np.float64)
            assert np.array_equal(got[m], want[m])
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("hi,wi,cout,k,st,p,S", [
    (59, 63, 96, 11, 4, 0, 3),       # AlexNet's first layer: 4 x 4 blocks of 3 channels = 48 -> 64 channels, 3 x 3 taps
    (45, 53, 64, 7, 2, 3, 2),        # ResNet's stem: 2 x 2 blocks = 12 -> 16 channels, 4 x 4 taps, three zero rows in front
    (37, 41, 32, 5, 2, 2, 2),
    (30, 34, 64, 3, 2, 1, 1),
    (40, 43, 32, 7, 3, 2, 2),        # 3 x 3 blocks = 27 -> 32 channels
    (33, 35, 64, 11, 4, 2, 2),       # padding that is not a multiple of the stride
])
def test_conv_strided_first_layers_as_space_to_depth(hi, wi, cout, k, st, p, S):
    """Strided convolutions on RGB run as stride-1 convolutions over a space-to-depth copy of their input: full and
    partial convolution against the oracle's strided one."""
    g = rng(hi * 3 + k)
    nb = nets.NetBuilder(hi, wi)
    nb.conv(-1, cout, k, st, p, 1)
    L = nb.layers[0]
    oh, ow = L["out_h"], L["out_w"]
    wts = g.normal(0, np.sqrt(2.0 / (k * k * 3)), size=(cout, k, k, 3)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    xq = np.stack([orc.quant_array(g.uniform(0, 1, size=(hi, wi, 3)), orc.QUANT_BF16) for _ in range(S)])
    pq = np.stack([orc.quant_array(g.normal(size=(oh, ow, cout)), orc.QUANT_BF16) for _ in range(S)])
    dc = DeepCache(wi, hi, nb.layers, [wts], [bias], n_streams=S, block=16, search_range=4, dtype=B.DC_BF16, max_regions=4)
    try:
        assert B.dc_cache_layer_conv_scheme(dc.handle, 0) >= 1          # a tensor-core scheme
        xin = torch.from_numpy(xq).to(torch.bfloat16).cuda()
        pin = torch.from_numpy(pq).to(torch.bfloat16).cuda()
        full = dc.conv_partial(0, xin)
        regs = torch.zeros((S, dc.max_regions, 6), dtype=torch.int32)
        counts = torch.zeros(S, dtype=torch.int32)
        regs[0, 0] = torch.tensor([1, 2, min(5, ow - 2), min(4, oh - 3), 2, 1], dtype=torch.int32)
        counts[0] = 1
        part = dc.conv_partial(0, xin, pin, regs.cuda(), counts.cuda())
        wq = orc.quant_array(wts, orc.QUANT_BF16)
        for s_ in range(S):
            r = np.zeros(1, orc.REGION_DTYPE)
            r[0] = tuple(int(v) for v in regs[s_, 0])
            want_full, _ = orc.conv_reuse(xq[s_], L, wq, bias, orc.QUANT_BF16)
            want, reused = orc.conv_reuse(xq[s_], L, wq, bias, orc.QUANT_BF16, pq[s_], r[:int(counts[s_])])
            U.assert_map_close(full[s_], want_full, True, f"full, stream {s_}")
            U.assert_map_close_per_element(full[s_], want_full, f"full, per element, stream {s_}")
            U.assert_map_close(part[s_], want, True, f"partial, stream {s_}")
            m = reused.astype(bool)
            got = part[s_].float().cpu().numpy().astype(np.float64)
            assert np.array_equal(got[m], want[m])
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("cin,k", [(64, 3), (32, 1), (3, 3), (128, 7)])      # column-slab / patch kernels, tap-by-tap kernel, few-channel kernel, CTA pairs
def test_bounded_device_waits_run_out_and_the_cache_stays_usable(cin, k, monkeypatch):
    """Failure detection without a fault: one convolution launch is armed so that its producer issues no copy.  The
    other roles' waits then run out after a few milliseconds instead of spinning for ever: the kernel returns, the
    status word reads DC_ERR_TIMEOUT, tensor memory is free again, and the next launch on the same cache is correct."""
    g = rng(90 + cin)
    hi = wi = 40
    cout = 64
    if k == 7:                                                     # stands for: a 3x3 layer of 128 -> 256 channels forced onto CTA pairs
        k, cout = 3, 256
        monkeypatch.setenv("DC_CONV_SCHEME", "7")
    nb = nets.NetBuilder(hi, wi)
    if cin == 3:
        nb.conv(-1, cout, k, 1, k // 2, 1)
        li = 0
        ws = [g.normal(0, 0.2, size=(cout, k, k, 3)).astype(np.float32)]
        bs = [g.normal(0, 0.1, size=cout).astype(np.float32)]
    else:
        a = nb.conv(-1, cin, 1, 1, 0)
        nb.conv(a, cout, k, 1, k // 2, 1)
        li = 1
        ws = [np.zeros((cin, 1, 1, 3), np.float32), g.normal(0, 0.1, size=(cout, k, k, cin)).astype(np.float32)]
        bs = [np.zeros(cin, np.float32), g.normal(0, 0.1, size=cout).astype(np.float32)]
    L = nb.layers[li]
    x = orc.quant_array(g.normal(size=(hi, wi, cin)), orc.QUANT_BF16)
    want, _ = orc.conv_reuse(x, L, orc.quant_array(ws[li], orc.QUANT_BF16), bs[li], orc.QUANT_BF16)
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=1, block=16, search_range=4, dtype=B.DC_BF16)
    try:
        stall = B.load().dc_debug_stall_next_conv
        stall.restype = ctypes.c_int
        stall.argtypes = [ctypes.c_void_p, ctypes.c_int]
        xin = torch.from_numpy(x[None]).to(torch.bfloat16).cuda()
        U.assert_map_close(dc.conv_partial(li, xin)[0], want, True, "before")
        assert dc.status() == B.DC_OK
        assert stall(dc.handle, 5) == B.DC_OK
        dc.conv_partial(li, xin)                                   # returns normally; its output is not valid
        assert dc.status() == B.DC_ERR_TIMEOUT
        dc.reset()                                                 # clears the status word
        assert dc.status() == B.DC_OK
        U.assert_map_close(dc.conv_partial(li, xin)[0], want, True, "after")
        assert dc.status() == B.DC_OK
        assert stall(dc.handle, 0) == B.DC_ERR_ARG and stall(None, 5) == B.DC_ERR_ARG
    finally:
        dc.close()


@pytest.mark.parametrize("scheme", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10])
def test_bounded_waits_run_out_in_every_scheme(scheme, monkeypatch):
    """The forced timeout of the test above on each operand scheme of the tensor-core convolution, asked for by number."""
    monkeypatch.setenv("DC_CONV_SCHEME", str(scheme))
    hw = 14 if scheme >= 8 else 32                                 # flat tiles: maps that blocks fill poorly
    nb = nets.NetBuilder(hw, hw)
    nb.conv(nb.conv(-1, 128, 1, 1, 0), 256, 3, 1, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 3)
    x = torch.from_numpy(rng(4).normal(size=(2, hw, hw, 128)).astype(np.float32)).to(torch.bfloat16).cuda()
    dc = DeepCache(hw, hw, nb.layers, ws, bs, n_streams=2, block=16, search_range=4, dtype=B.DC_BF16)
    try:
        assert B.dc_cache_layer_conv_scheme(dc.handle, 1) == scheme
        stall = B.load().dc_debug_stall_next_conv
        stall.restype, stall.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
        want = dc.conv_partial(1, x)
        assert stall(dc.handle, 5) == B.DC_OK
        dc.conv_partial(1, x)                                      # returns normally; its output is not valid
        assert dc.status() == B.DC_ERR_TIMEOUT
        dc.reset()
        assert torch.equal(dc.conv_partial(1, x), want) and dc.status() == B.DC_OK
    finally:
        dc.close()


def test_a_cluster_with_one_stalled_cta_stores_nothing(monkeypatch):
    """One CTA of every cluster gets no operands and gives up: the others have only a part of the sums and must not store
    it.  The next launch is correct."""
    monkeypatch.setenv("DC_CONV_SCHEME", "10")
    g = rng(17)
    nb = nets.NetBuilder(13, 13)
    nb.conv(nb.conv(-1, 256, 1, 1, 0), 128, 3, 1, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 3)
    x = torch.from_numpy(g.normal(size=(2, 13, 13, 256)).astype(np.float32)).to(torch.bfloat16).cuda()
    dc = DeepCache(13, 13, nb.layers, ws, bs, n_streams=2, block=16, search_range=4, dtype=B.DC_BF16)
    try:
        assert B.dc_cache_layer_conv_scheme(dc.handle, 1) == 10
        stall = B.load().dc_debug_stall_next_conv
        stall.restype, stall.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
        want = dc.conv_partial(1, x)
        assert want.any()
        assert stall(dc.handle, 5) == B.DC_OK
        out = dc.conv_partial(1, x)                                # into a map of zeros
        assert dc.status() == B.DC_ERR_TIMEOUT and not out.any()
        dc.reset()
        assert torch.equal(dc.conv_partial(1, x), want) and dc.status() == B.DC_OK
    finally:
        dc.close()


def test_lookahead_gives_identical_results():
    """dc_lookahead_frame moves the matching of frame t+1 beside the inference of frame t; outputs, motion
    vectors and rectangles must not change.  Also: a lookahead for a frame that is then not used.
    One cache runs the sequence twice (plain, then with lookahead) so that both passes use the same kernels."""
    w = configs.WORKLOADS[3]()
    sb = w.streams(1, 13)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).cuda() for i in range(13)]
    dc = DeepCache.from_workload(w)
    try:
        pitch = w.width * 3

        def run(lookahead):
            rec = []
            dc.reset()
            for i in range(12):
                out, st = dc.infer_frame(frames[i], want_stats=True)
                out = out.clone()
                if lookahead:
                    if i == 5:
                        B.dc_lookahead_frame(dc.handle, frames[0], pitch)        # announced, but frame 6 comes next
                    elif i != 7:
                        B.dc_lookahead_frame(dc.handle, frames[i + 1], pitch)    # crosses the expiry at frame 10
                regs, _ = dc.layer_regions(-1)
                key = (st[0].refreshed, st[0].mvx, st[0].mvy, st[0].k_passed, st[0].n_matched, st[0].n_regions)
                rec.append((out, key, regs[0, :st[0].n_regions].clone()))
            return rec

        plain, ahead = run(False), run(True)
        assert any(not k[0] and k[4] > 0 for _, k, _ in plain)
        for i, ((o0, k0, r0), (o1, k1, r1)) in enumerate(zip(plain, ahead)):
            assert k0 == k1, f"frame {i}: {k0} vs {k1}"
            if not k0[0]:
                assert torch.equal(r0, r1), f"frame {i} rectangles"
            assert torch.equal(o0, o1), f"frame {i} output"
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("S,W,H", [(1, 400, 240), (60, 400, 240), (80, 160, 96)])
def test_propagate_frames_of_many_rectangles(S, W, H):
    """A frame's rectangles shared by four CTAs, by two, and by none, in batches that the frame fills and does not: table, counts and reuse, frame
    after frame, announced and not."""
    nb = nets.NetBuilder(H, W)
    x = nb.conv(-1, 16, 3, 1, 1)
    for k in (1, 1, 3, 1, 1):
        x = nb.conv(x, 16, k, 1, k // 2)
    ws, bs = nets.random_weights(nb.layers, 2)
    g = rng(S)
    base = g.integers(0, 256, (S, H, W, 3), dtype=np.uint8)
    frames = []
    for t in range(5):
        f = base.copy()
        for s in range(S):
            share = (0.0, 0.45, 0.1, 0.02, 0.5)[(t + s) % 5]
            for y, x0 in np.argwhere(g.random((H // 8, W // 8)) < share):
                f[s, 8 * y:8 * y + 8, 8 * x0:8 * x0 + 8] = g.integers(0, 256, (8, 8, 3))
        frames.append(torch.from_numpy(f).cuda())
    kw = dict(n_streams=S, block=8, search_range=0, dtype=B.DC_BF16, max_regions=W // 8 * (H // 8))
    dc, ahead = DeepCache(W, H, nb.layers, ws, bs, **kw), DeepCache(W, H, nb.layers, ws, bs, **kw)
    try:
        for t, f in enumerate(frames):
            _, st = dc.infer_frame(f, want_stats=True)
            _, st2 = ahead.infer_frame(f, want_stats=True)
            if t + 1 < len(frames):
                B.dc_lookahead_frame(ahead.handle, frames[t + 1], W * 3)
            if st[0].refreshed:
                continue
            regs0 = dc.layer_regions(-1)[0].cpu()
            tables = [dc.layer_regions(l)[0].cpu() for l in range(len(nb.layers))]
            for s in range(S):
                n = st[s].n_regions
                assert list(st[s].reuse_ratio[:len(nb.layers)]) == list(st2[s].reuse_ratio[:len(nb.layers)])
                want = orc.propagate(nb.layers, (H, W), U.regions_np(regs0[s, :n]))
                for l in range(len(nb.layers)):
                    U.assert_regions_equal(U.regions_np(tables[l][s, :n]), want[l], f"frame {t} stream {s} layer {l}")
                    assert abs(st[s].reuse_ratio[l] - float((want[l]["w"] * want[l]["h"]).sum()) / (W * H)) < 1e-6
        assert max(x.n_regions for x in st) > (256 if W == 400 else 40) and dc.status() == B.DC_OK and ahead.status() == B.DC_OK
    finally:
        dc.close(); ahead.close()


@pytest.mark.parametrize("recorded", [1, 2])
def test_first_lookahead_in_a_graph(recorded):
    """The first announced frames of a cache recorded in a capture, where nothing may be allocated, and launched from there; then announced by
    plain calls, with the match sets standing either way round.  Outputs are those of frames that were not announced."""
    w = configs.WORKLOADS[3]()
    sb = w.streams(1, 7)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).cuda() for i in range(7)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dc = DeepCache.from_workload(w)
        pitch = w.width * 3
        want = [dc.infer_frame(f).clone() for f in frames]
        dc.reset()
        got = [dc.infer_frame(frames[0]).clone()]
        outs = [torch.empty_like(got[0]) for _ in range(recorded)]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for k in range(recorded):
            B.dc_lookahead_frame(dc.handle, frames[1 + k], pitch)
            B.dc_infer_frame(dc.handle, frames[1 + k], pitch, outs[k], None)
    with torch.cuda.stream(stream):
        graph.replay()
        stream.synchronize()
        got += outs
        for i in range(1 + recorded, 7):
            if i > 1 + recorded:            # behind a capture a frame that is not announced comes first
                B.dc_lookahead_frame(dc.handle, frames[i], pitch)
            got.append(dc.infer_frame(frames[i]).clone())
        stream.synchronize()
        assert dc.status() == B.DC_OK
    for i, (x, y) in enumerate(zip(want, got)):
        assert torch.equal(x, y), f"frame {i}"
    del graph
    dc.close()


@pytest.mark.parametrize("asked", ["first", "late", "behind other calls"])
def test_rectangles_of_announced_frames_stay_where_the_program_found_them(asked):
    """dc_cache_layer_regions names one address of a layer's rectangles for the cache's life.  Asked for once, before or after frames have been
    announced, it holds those of each frame that follows, announced or not; announcing frames takes no memory."""
    w = configs.WORKLOADS[3]()
    sb = w.streams(1, 9)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).cuda() for i in range(9)]
    dc = DeepCache.from_workload(w)
    try:
        n_layers, pitch = len(w.layers), w.width * 3

        def tables(ptrs, n):
            torch.cuda.synchronize()
            return [device_view(p, (dc.max_regions, 6), torch.int32, dc.device)[:n].clone() for p in ptrs]

        def ask():
            return [B.dc_cache_layer_regions(dc.handle, l)[0] for l in range(n_layers)]

        want = []
        for f in frames:                                            # one after the other, in a cache of its own
            if not want:
                plain = DeepCache.from_workload(w)
            _, st = plain.infer_frame(f, want_stats=True)
            want.append([plain.layer_regions(l)[0][0, :st[0].n_regions] for l in range(n_layers)])
        plain.close()
        assert sum(int((r[0][:, 2] > 0).sum()) for r in want[1:]) > 8
        size = dc.bytes()
        ptrs = ask() if asked == "first" else None
        for i, f in enumerate(frames):
            _, st = dc.infer_frame(f, want_stats=True)
            if i not in (5, len(frames) - 1):
                B.dc_lookahead_frame(dc.handle, frames[i + 1], pitch)
            if i < 3 and asked != "first":
                continue
            if ptrs is None and asked == "behind other calls":      # what writes the frame's rectangles, and some layers' tables, anew
                other = dc.match_blocks(frames[0])
                out, _ = dc.propagate_regions(other["regions"], other["n_regions"], 0, 2)
                ptrs = ask()
                got = tables(ptrs, st[0].n_regions)
                for l in range(n_layers):
                    assert torch.equal(got[l], out[l, 0, :st[0].n_regions] if l < 2 else want[i][l]), f"frame {i} layer {l}"
                continue
            ptrs = ptrs or ask()
            assert ask() == ptrs
            if not st[0].refreshed:
                for l, (x, y) in enumerate(zip(tables(ptrs, st[0].n_regions), want[i])):
                    assert torch.equal(x, y), f"frame {i} layer {l}"
        assert dc.bytes() == size and dc.status() == B.DC_OK
    finally:
        dc.close()


def test_rectangles_of_announced_frames_in_a_graph():
    """A graph of an announced frame, recorded before the program asks for the address of a layer's rectangles, leaves them there when it is
    launched again behind that, over the frame its buffer then holds."""
    w = configs.WORKLOADS[3]()
    sb = w.streams(1, 3)
    frames = [torch.from_numpy(np.ascontiguousarray(sb.frame(i))).cuda() for i in range(3)]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        dc = DeepCache.from_workload(w)
        dc.infer_frame(frames[0])
        _, st = dc.infer_frame(frames[2], want_stats=True)          # the frame of the second launch, behind frame 0
        n, want = st[0].n_regions, [dc.layer_regions(l)[0][0, :st[0].n_regions] for l in range(len(w.layers))]
        dc.close()
        dc = DeepCache.from_workload(w)
        dc.infer_frame(frames[0])
        buf = frames[1].clone()
        stream.synchronize()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        B.dc_lookahead_frame(dc.handle, buf, w.width * 3)
        B.dc_infer_frame(dc.handle, buf, w.width * 3, None, None)
    with torch.cuda.stream(stream):
        graph.replay()
        ptrs = [B.dc_cache_layer_regions(dc.handle, l)[0] for l in range(len(w.layers))]
        buf.copy_(frames[2])
        graph.replay()
        stream.synchronize()
        assert n > 0 and dc.status() == B.DC_OK
        for l, p in enumerate(ptrs):
            assert torch.equal(device_view(p, (dc.max_regions, 6), torch.int32, dc.device)[:n], want[l]), f"layer {l}"
    del graph
    dc.close()


@pytest.mark.parametrize("search,R", [(B.DC_SEARCH_DIAMOND, 12), (B.DC_SEARCH_THREE_STEP, 9)])
@pytest.mark.parametrize("W,H,S", [(64, 48, 2), (144, 70, 3), (64, 37, 160)])
def test_frames_matched_where_they_lie(search, R, W, H, S):
    """Frames of whole aligned blocks are read by the search where the caller has them, others through a copy: the same frames at any pitch and
    start give the same matches, outputs and keys, frame by frame, announced or not, also from a buffer that is filled anew behind a call."""
    g = rng(W + R)
    coarse = torch.from_numpy(g.integers(0, 256, (S, 3, H // 8 + 6, W // 8 + 6)).astype(np.float32))
    base = torch.nn.functional.interpolate(coarse, scale_factor=8, mode="bilinear").permute(0, 2, 3, 1).numpy().astype(np.uint8)
    frames = np.stack([base[:, 3 * t:3 * t + H, 20 - 2 * t:20 - 2 * t + W] for t in range(5)])
    frames[3, :, :17, :20] ^= 0x55
    nb = nets.NetBuilder(H, W)
    nb.conv(nb.conv(-1, 16, 3, 1, 1), 16, 3, 1, 1)
    ws, bs = nets.random_weights(nb.layers, 5)
    records = []
    for pitch, start, ahead in ((W * 3, 0, False), (W * 3, 0, True), (W * 3 + 48, 16, False), (W * 3 + 7, 0, False), (W * 3, 5, True), (W * 3 + 16, 8, False)):
        dc = DeepCache(W, H, nb.layers, ws, bs, n_streams=S, block=16, search_range=R, search=search, dtype=B.DC_FP32, expire_n=4)
        bufs = [torch.zeros(start + S * H * pitch, dtype=torch.uint8, device="cuda") for _ in range(2)]

        def put(t):
            v = bufs[t % 2][start:].view(S, H, pitch)[:, :, :W * 3]
            v.copy_(torch.from_numpy(np.ascontiguousarray(frames[t])).cuda().reshape(S, H, W * 3))
            return bufs[t % 2][start:]

        rec, f = [], put(0)
        for t in range(5):
            out = torch.empty(dc.out_shape(-1), device="cuda")
            B.dc_infer_frame(dc.handle, f, pitch, out)
            if t + 1 < 5:
                f = put(t + 1)                                    # behind the call, on the same stream
                if ahead:
                    B.dc_lookahead_frame(dc.handle, f, pitch)
                elif t == 1:
                    mv = torch.zeros((S, dc.Gy, dc.Gx, 2), dtype=torch.int16, device="cuda")
                    matched = torch.zeros((S, dc.Gy, dc.Gx), dtype=torch.uint8, device="cuda")
                    B.dc_match_blocks(dc.handle, f, pitch, mv, None, matched, None, None, None)
                    rec_match = (mv, matched)
            rec.append((out, dc.layer_regions(-1)[1]))
        assert dc.status() == B.DC_OK
        records.append((rec, None if ahead else rec_match))
        torch.cuda.synchronize()
        dc.close()
    assert records[0][1][1].any()
    for rec, match in records[1:]:
        for (o0, n0), (o1, n1) in zip(records[0][0], rec):
            assert torch.equal(o0, o1) and torch.equal(n0, n1)
        if match is not None:
            assert all(torch.equal(x, y) for x, y in zip(records[0][1], match))


def test_lookahead_waits_for_the_calls_between():
    """dc_lookahead_frame right behind dc_match_blocks (whose frame lies where the announced one goes) and behind
    dc_cache_set_key (which changes the key that it is matched against)."""
    W, H, S = 1280, 720, 4
    g = rng(12)
    base = np.repeat(np.repeat(g.integers(0, 256, size=(S, H // 8, W // 8, 3), dtype=np.uint8), 8, 1), 8, 2)
    f = [torch.from_numpy(np.roll(base, (3 * k, -2 * k), axis=(1, 2))).cuda() for k in range(4)]
    layers = nets.vgg16_trunk(224, 224, H, W)[:3]
    ws, bs = nets.random_weights(layers, 2)
    rec = []
    for early in (False, True):
        dc = DeepCache(W, H, layers, ws, bs, n_streams=S, block=16, search_range=16, dtype=B.DC_BF16)
        out = [torch.zeros(s_, dtype=t, device="cuda") for s_, t in (((S, dc.Gy, dc.Gx, 2), torch.int16), ((S, dc.Gy, dc.Gx), torch.int32), ((S, 3), torch.int32))]

        def pause():
            if not early:
                torch.cuda.synchronize()

        dc.infer_frame(f[0])
        B.dc_lookahead_frame(dc.handle, f[1], W * 3)
        dc.infer_frame(f[1])
        pause()
        B.dc_match_blocks(dc.handle, f[3], W * 3, out[0], out[1], None, out[2], None, None)
        pause()
        B.dc_lookahead_frame(dc.handle, f[2], W * 3)
        pause()
        a = dc.infer_frame(f[2])
        pause()
        B.dc_cache_set_key(dc.handle, f[0], W * 3)
        pause()
        B.dc_lookahead_frame(dc.handle, f[3], W * 3)
        pause()
        _, st = dc.infer_frame(f[3], want_stats=True)
        rec.append((*[o.clone() for o in out], a, torch.tensor([[s_.mvx, s_.mvy, s_.k_passed, s_.n_matched] for s_ in st])))
        assert dc.status() == B.DC_OK
        dc.close()
    assert all(torch.equal(x, y) for x, y in zip(*rec))


@pytest.mark.parametrize("dtype,hi,wi,cin,cout,k,S,groups", [
    (B.DC_FP32, 130, 200, 4, 64, 3, 3, 1),       # 8 x 8 sums per thread, 64-channel blocks, one short chunk
    (B.DC_FP32, 140, 210, 7, 32, 3, 5, 1),       # 8 x 8 sums, 32-channel blocks, channels not a multiple of four
    (B.DC_FP32, 90, 140, 24, 128, 1, 6, 1),      # 1 x 1, a last chunk that is half full
    (B.DC_FP32, 19, 21, 10, 20, 5, 2, 1),         # 8 x 4 sums, a last block that is not full, 5 x 5 taps
    (B.DC_FP32, 17, 9, 12, 24, 3, 2, 2),         # two channel groups
    (B.DC_BF16, 33, 18, 24, 16, 3, 3, 1),        # bfloat16 with channel counts the tensor-core kernels do not take
    (B.DC_BF16, 16, 8, 24, 40, 1, 2, 1),         # exactly one tile per stream
    (B.DC_FP32, 7, 9, 7, 12, 0, 5, 1),           # one output pixel (k = 0: the kernel covers the map), odd reduction
    (B.DC_BF16, 8, 10, 64, 48, 0, 9, 1),
])
def test_conv_on_cuda_cores(dtype, hi, wi, cin, cout, k, S, groups):
    """The register-blocked kernel and the one for single output pixels: full and partial convolution against the
    oracle at partial tiles, partial channel blocks and chunks, groups, every shape of a thread's sums."""
    g = rng(hi * 5 + wi + cout)
    bf16 = dtype == B.DC_BF16
    quant = orc.QUANT_BF16 if bf16 else orc.QUANT_NONE
    nb = nets.NetBuilder(hi, wi)
    x0 = nb.conv(-1, 4 if cin % 4 else cin, 1, 1, 0)
    while nb.shape(x0)[2] < cin:                                    # an odd channel count: the frame's three channels joined on
        x0 = nb.concat(x0, -1)
    if k:
        nb.conv(x0, cout, k, 1, k // 2, 1, groups=groups)
    else:
        nb.fc(x0, cout, relu=1)
    L = dict(nb.layers[-1], kind=0, sh=1, sw=1)
    li = len(nb.layers) - 1
    wts = g.normal(0, np.sqrt(2.0 / (L["kh"] * L["kw"] * cin / groups)), size=(cout, L["kh"], L["kw"], cin // groups)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    ws = [np.zeros((l["cout"], 1, 1, 3), np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [wts]
    bs = [np.zeros(l["cout"], np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [bias]
    q = lambda shape: np.stack([orc.quant_array(g.normal(size=shape).astype(np.float32).astype(np.float64), quant) for _ in range(S)])
    xq, pq = q((hi, wi, cin)), q((L["out_h"], L["out_w"], cout))
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=dtype, max_regions=4)
    try:
        assert B.dc_cache_layer_conv_scheme(dc.handle, li) == 0
        xin, pin = torch.from_numpy(xq).to(dc.tdtype).cuda(), torch.from_numpy(pq).to(dc.tdtype).cuda()
        full = dc.conv_partial(li, xin)
        regs = torch.zeros((S, dc.max_regions, 6), dtype=torch.int32)
        counts = torch.zeros(S, dtype=torch.int32)
        ow, oh = L["out_w"], L["out_h"]
        if oh > 4:
            regs[0, 0] = torch.tensor([1, 2, ow // 2, min(11, oh - 3), 2, 1], dtype=torch.int32)
            counts[0] = 1
        regs[1, 0] = torch.tensor([0, 0, ow, oh, 0, 0], dtype=torch.int32)       # a stream with nothing left to compute
        counts[1] = 1
        part = dc.conv_partial(li, xin, pin, regs.cuda(), counts.cuda())
        wq = orc.quant_array(wts, quant)
        for s_ in range(S):
            r = np.zeros(1, orc.REGION_DTYPE)
            r[0] = tuple(int(v) for v in regs[s_, 0])
            want_full, _ = orc.conv_reuse(xq[s_], L, wq, bias, quant)
            want, reused = orc.conv_reuse(xq[s_], L, wq, bias, quant, pq[s_], r[:int(counts[s_])])
            U.assert_map_close(full[s_], want_full, bf16, f"full, stream {s_}")
            U.assert_map_close(part[s_], want, bf16, f"partial, stream {s_}")
            m = reused.astype(bool)
            assert np.array_equal(part[s_].float().cpu().numpy().astype(np.float64)[m], want[m])
        assert dc.status() == B.DC_OK
    finally:
        dc.close()


@pytest.mark.parametrize("search", [B.DC_SEARCH_EXHAUSTIVE, B.DC_SEARCH_DIAMOND, B.DC_SEARCH_THREE_STEP])
@pytest.mark.parametrize("block,R,shape", [(4, 12, (41, 67)), (13, 9, (70, 131)), (24, 64, (150, 170)), (32, 33, (64, 96)), (9, 7, (200, 181))])
def test_match_staged_window_shapes(search, block, R, shape):
    """Block sizes whose lanes own 1 to 32 pixels with a last one that is full or not, windows that shrink the tile (large
    ranges), clipped right columns and bottom rows, k-skip."""
    g = rng(block * 3 + R)
    H, W = shape
    prev = g.integers(0, 256, size=(H, W, 3), dtype=np.uint8)
    smooth = np.repeat(np.repeat(g.integers(0, 256, size=(H // 8 + 1, W // 8 + 1, 3), dtype=np.uint8), 8, 0), 8, 1)[:H, :W]
    pairs = [(prev, np.roll(prev, (min(R, 5), -min(R, 6)), axis=(0, 1))), (smooth, np.roll(smooth, (-3, 4), axis=(0, 1))), (prev, smooth)]
    check_pairs(pairs, block, R, search)
    check_pairs(pairs[1:2], block, R, search, skip_k=2)


@pytest.mark.parametrize("search", [B.DC_SEARCH_DIAMOND, B.DC_SEARCH_THREE_STEP])
@pytest.mark.parametrize("block,R", [(4, 64), (6, 33), (8, 64), (10, 40), (14, 64), (20, 64), (32, 64)])
def test_match_walks_leave_the_staged_window(search, block, R):
    """Ranges beyond what the walks stage: a smooth texture moved by up to 60 pixels leads the walks out of the window, at its
    edge, across the frame's edges and past the range."""
    g = rng(block * 5 + R)
    H, W = 190, 230
    lat = g.uniform(0, 255, size=(H // 24 + 4, W // 24 + 4, 3))
    y, x = np.arange(H + 80) / 30.0, np.arange(W + 80) / 30.0
    iy, ix = y.astype(int) % lat.shape[0], x.astype(int) % lat.shape[1]
    fy, fx = (y - y.astype(int))[:, None, None], (x - x.astype(int))[None, :, None]
    rows = lat[iy] * (1 - fy) + lat[(iy + 1) % lat.shape[0]] * fy
    tex = (rows[:, ix] * (1 - fx) + rows[:, (ix + 1) % lat.shape[1]] * fx).astype(np.uint8)
    cut = lambda dy, dx: np.ascontiguousarray(tex[40 + dy:40 + dy + H, 40 + dx:40 + dx + W])
    pairs = [(cut(0, 0), cut(dy, dx)) for dy, dx in ((33, -31), (-38, 36), (2, 39), (0, 1))]
    far = [orc.match_blocks(c, p, block, R, search, 20.0, 1, 0)["mv"] for p, c in pairs]
    assert max(np.abs(m).max() for m in far) > (32 if search == B.DC_SEARCH_DIAMOND or R >= 63 else 28)     # three steps reach 31 or 63
    check_pairs(pairs, block, R, search)
    check_pairs(pairs[:1], block, R, search, skip_k=2)


@pytest.mark.parametrize("hi,wi,cin,cout,k,S,groups", [
    (17, 9, 16, 32, 3, 2, 1),           # one step of 16 channels, tiles cut on both sides
    (64, 72, 32, 64, 3, 4, 1),          # one whole patch of 32 channels, 64 output channels
    (113, 113, 64, 64, 3, 6, 1),        # wide blocks, several items per CTA
    (30, 22, 80, 128, 3, 3, 1),         # a last patch of one step
    (33, 21, 20, 36, 3, 2, 1),          # channels beyond the last of a step and of a block
    (40, 30, 48, 64, 5, 3, 1),          # 5 x 5: the largest patch
    (90, 140, 24, 128, 1, 6, 1),        # 1 x 1
    (16, 8, 200, 96, 1, 2, 1),          # several 1 x 1 patches to a drain, the last drain not full
    (24, 20, 40, 72, 3, 2, 2),          # two channel groups
    (19, 25, 19, 40, 3, 2, 1),          # pixels that no vector load takes
])
def test_conv_fp32_on_tensor_cores(hi, wi, cin, cout, k, S, groups):
    """float32 layers whose operands are split into bf16 pieces: full and partial, against 64-bit sums.  Every product is within
    2^-24 of the float one; a sum in the tensor core (steps = 2 k of 16 channels and three products, at most 12 for 1 x 1) may
    be cut by 2^-23 of the terms' magnitudes per step, a sum in registers rounds by 2^-24.  Those are an element's worst cases; the
    2-norm of all errors is 0.5e-7 to 1.5e-7 of the output's, and 20 times that without one of the six products of pieces (2^-17 of a
    term each, 2^-18.5 in the mean square)."""
    g = rng(hi * 7 + wi + cout)
    nb = nets.NetBuilder(hi, wi)
    x0 = nb.conv(-1, cin - 3 if cin % 4 else cin, 1, 1, 0)
    if nb.shape(x0)[2] < cin:
        x0 = nb.concat(x0, -1)                                      # an odd channel count: the frame's three channels joined on
    nb.conv(x0, cout, k, 1, k // 2, 1, groups=groups)
    li, L = len(nb.layers) - 1, nb.layers[-1]
    wts = g.normal(0, np.sqrt(2.0 / (k * k * cin / groups)), size=(cout, k, k, cin // groups)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    ws = [np.zeros((l["cout"], 1, 1, 3), np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [wts]
    bs = [np.zeros(l["cout"], np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [bias]
    dc = DeepCache(wi, hi, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
    try:
        xin = torch.from_numpy(g.normal(size=(S, hi, wi, cin)).astype(np.float32)).cuda()
        prev = torch.from_numpy(g.normal(size=(S, hi, wi, cout)).astype(np.float32)).cuda()
        conv = lambda x, w, b: torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), w, b, padding=k // 2, groups=groups).permute(0, 2, 3, 1)
        w64 = torch.from_numpy(wts).cuda().double().permute(0, 3, 1, 2)
        want = conv(xin, w64, torch.from_numpy(bias).cuda().double()).relu()
        drains = -(-(-(-cin // groups // 32) * k) // (1 if k > 1 else 3))
        bound = (36 * 2.0 ** -23 + (drains + 4) * 2.0 ** -24) * (conv(xin.abs(), w64.abs(), None) + 1.0)
        full = dc.conv_partial(li, xin)
        assert ((full.double() - want).abs() <= bound).all()
        assert (full.double() - want).norm() <= 2.5e-7 * want.norm()
        regs, counts = torch.zeros((S, 4, 6), dtype=torch.int32, device="cuda"), torch.zeros(S, dtype=torch.int32, device="cuda")
        regs[0, 0] = torch.tensor([1, 2, wi // 2, hi - 5, 2, 1], dtype=torch.int32)
        regs[1, 0] = torch.tensor([0, 0, wi, hi, 0, 0], dtype=torch.int32)          # a stream with nothing left to compute
        counts[:2] = 1
        part = dc.conv_partial(li, xin, prev, regs, counts)
        made = full.clone()                                         # what is computed does not depend on what is reused
        made[1] = prev[1]
        made[0, 2:hi - 3, 1:1 + wi // 2] = prev[0, 1:hi - 4, 2:2 + wi // 2]
        assert torch.equal(part, made) and dc.status() == B.DC_OK
        stall = B.load().dc_debug_stall_next_conv
        stall.restype, stall.argtypes = ctypes.c_int, [ctypes.c_void_p, ctypes.c_int]
        assert stall(dc.handle, 5) == B.DC_OK
        dc.conv_partial(li, xin)                                    # returns normally; its output is not valid
        assert dc.status() == B.DC_ERR_TIMEOUT
        dc.reset()
        assert torch.equal(dc.conv_partial(li, xin), full) and dc.status() == B.DC_OK
    finally:
        dc.close()


def test_conv_fp32_on_tensor_cores_with_values_that_do_not_split():
    """Infinities, NaN and the largest floats come out as from a chain of FMAs; tiles without them are not touched."""
    g = rng(77)
    nb = nets.NetBuilder(48, 40)
    nb.conv(nb.conv(-1, 32, 1, 1, 0), 64, 3, 1, 1, 0)
    wts = g.normal(0, 0.1, size=(64, 3, 3, 32)).astype(np.float32)
    wts[5] = 0.5                                                   # exact in one piece: the others are zero
    zero = np.zeros(64, np.float32)
    dc = DeepCache(40, 48, nb.layers, [np.zeros((32, 1, 1, 3), np.float32), wts], [zero[:32], zero], n_streams=1, block=16, search_range=4,
                   dtype=B.DC_FP32, max_regions=4)
    try:
        x = torch.from_numpy(g.normal(size=(1, 48, 40, 32)).astype(np.float32)).cuda()
        clean = dc.conv_partial(1, x)
        x[0, 3, 3, 7], x[0, 20, 12, 1], x[0, 37, 30, 31], x[0, 37, 12, 4] = float("inf"), float("-inf"), float("nan"), 3.402e38
        got = dc.conv_partial(1, x)
        want = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), torch.from_numpy(wts).cuda().double().permute(0, 3, 1, 2), padding=1).permute(0, 2, 3, 1).float()
        odd = ~torch.isfinite(want) | (want.abs() > 1e30)
        assert odd.sum() >= 4 * 9 * 63
        assert torch.equal(torch.isnan(got), torch.isnan(want))
        assert torch.equal(got[torch.isinf(want)], want[torch.isinf(want)])
        big = odd & torch.isfinite(want)
        assert torch.allclose(got[big], want[big], rtol=1e-6)
        assert (got[~odd] - clean[~odd]).abs().max() < 1e-4
        far = torch.ones((48, 40), dtype=torch.bool, device="cuda")
        for y, xx in ((3, 3), (20, 12), (37, 30), (37, 12)):       # whole tiles whose patch holds one of them
            far[max(0, (y - 1) // 16 * 16):(y + 1) // 16 * 16 + 16, max(0, (xx - 1) // 8 * 8):(xx + 1) // 8 * 8 + 8] = False
        assert far.sum() > 500 and torch.equal(got[0][far], clean[0][far])
    finally:
        dc.close()


@pytest.mark.parametrize("cin,k,S", [(32, 3, 24), (32, 3, 10), (96, 3, 24), (16, 5, 24), (32, 1, 24), (200, 1, 11)])
def test_conv_fp32_items_in_turns(cin, k, S):
    """Layers with several items per CTA, finished by two groups of warps in turn, with weights that stay in shared memory (one patch of channels)
    and that do not: stream by stream the bits of one stream alone, where every item has an SM, also where pixels are left to FMAs or reused."""
    g = rng(cin + k)
    H, W = 48, 39
    nb = nets.NetBuilder(H, W)
    nb.conv(nb.conv(-1, cin, 1, 1, 0), 32, k, 1, k // 2, 0)
    wts = g.normal(0, np.sqrt(2.0 / (k * k * cin)), size=(32, k, k, cin)).astype(np.float32)
    bias = g.normal(0, 0.1, size=32).astype(np.float32)
    x = g.normal(size=(S, H, W, cin)).astype(np.float32)
    x[::3, 5, 7, 1], x[1::4, 33, 20, 0] = np.inf, np.float32(2.0 ** -120 * 1.2345678)
    x[::2, 16:32, 8:16] = 0.0
    x, prev = torch.from_numpy(x).cuda(), torch.from_numpy(g.normal(size=(S, H, W, 32)).astype(np.float32)).cuda()
    regs, n = torch.zeros((S, 4, 6), dtype=torch.int32, device="cuda"), torch.ones(S, dtype=torch.int32, device="cuda")
    regs[:, 0] = torch.tensor([3, 2, 30, 21, 1, 4], dtype=torch.int32)

    def run(lo, hi):
        dc = DeepCache(W, H, nb.layers, [np.zeros((cin, 1, 1, 3), np.float32), wts], [np.zeros(cin, np.float32), bias], n_streams=hi - lo, block=16,
                       search_range=4, dtype=B.DC_FP32, max_regions=4)
        try:
            outs = [dc.conv_partial(1, x[lo:hi]), dc.conv_partial(1, x[lo:hi], prev[lo:hi], regs[lo:hi], n[lo:hi])]
            assert dc.status() == B.DC_OK
            return outs
        finally:
            dc.close()

    full, part = run(0, S)
    assert (~torch.isfinite(full)).any()
    for s in range(S):
        one_full, one_part = run(s, s + 1)
        assert torch.allclose(full[s], one_full[0], rtol=0, atol=0, equal_nan=True) and torch.allclose(part[s], one_part[0], rtol=0, atol=0, equal_nan=True)


@pytest.mark.parametrize("cin,S", [(32, 40), (96, 31)])
def test_conv_fp32_many_items_in_turns(cin, S):
    """The same of 3 x 3 layers with more than three items per SM, which alone are finished in turns."""
    test_conv_fp32_items_in_turns(cin, 3, S)


@pytest.mark.parametrize("relu", [0, 1])
@pytest.mark.parametrize("cin,cout,k,H,W,S,groups", [(32, 64, 3, 48, 40, 1, 1), (64, 32, 1, 33, 21, 2, 1), (40, 72, 5, 30, 22, 2, 2), (64, 64, 3, 113, 113, 4, 1)])
def test_conv_fp32_sums_beyond_the_largest_float(cin, cout, k, H, W, S, groups, relu, monkeypatch):
    """Finite operands whose sums leave the float range: infinities as from a chain of FMAs, never NaN, and +infinity after ReLU.  All the
    products of a channel have one sign, so that the order of the sum does not matter; most pixels stay far below."""
    g = rng(cin + cout + k)
    nb = nets.NetBuilder(H, W)
    nb.conv(nb.conv(-1, cin, 1, 1, 0), cout, k, 1, k // 2, relu, groups=groups)
    wts = np.abs(g.normal(0, 0.1, size=(cout, k, k, cin // groups))).astype(np.float32) + np.float32(0.1)
    wts[1::2] *= -1
    wts[:8] = np.ldexp(wts[:8], 70)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    x = g.uniform(0.5, 1.0, size=(S, H, W, cin)).astype(np.float32)
    x[:, 5:9, 3:7] = np.ldexp(x[:, 5:9, 3:7], 60)                   # sums of 2^130 and more
    x[:, 20:24, 14:17] = np.ldexp(x[:, 20:24, 14:17], 70)           # 2^140
    x[:, 20:22, 2:4] = np.ldexp(x[:, 20:22, 2:4], 40)               # 2^110: large and finite
    x = torch.from_numpy(x).cuda()
    out = []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(W, H, nb.layers, [np.zeros((cin, 1, 1, 3), np.float32), wts], [np.zeros(cin, np.float32), bias], n_streams=S, block=16,
                       search_range=4, dtype=B.DC_FP32, max_regions=4)
        out.append(dc.conv_partial(1, x))
        if not cores:                                               # reuse leaves the other pixels' bits as they are
            regs, n = torch.zeros((S, 4, 6), dtype=torch.int32, device="cuda"), torch.ones(S, dtype=torch.int32, device="cuda")
            regs[:, 0] = torch.tensor([2, 4, 6, 2, 2, 4], dtype=torch.int32)
            assert torch.equal(dc.conv_partial(1, x, out[0], regs, n), out[0])
        dc.close()
    got, want = out
    over = torch.isinf(want)
    assert over.sum() >= S * 20 * 4 and not torch.isnan(want).any()
    assert torch.equal(torch.isinf(got), over) and torch.equal(got[over], want[over])
    assert torch.allclose(got[~over], want[~over], rtol=1e-5, atol=1e-4)        # sums of one sign: both within (terms) 2^-24 of the exact one


@pytest.mark.parametrize("cin,cout,k,H,W,S,groups", [(64, 64, 3, 113, 113, 4, 1), (32, 32, 3, 60, 50, 2, 1), (40, 72, 5, 30, 22, 2, 2), (71, 36, 1, 40, 33, 3, 1), (19, 40, 3, 19, 25, 2, 1)])
def test_conv_fp32_every_tile_computed_by_fmas(cin, cout, k, H, W, S, groups, monkeypatch):
    """An infinity in every tile: every bit as the CUDA-core kernel has it, and a pass takes a small multiple of that kernel's time (1.4 to 3.5
    measured; the bound leaves room for a busy host)."""
    g = rng(cin * 3 + cout + k)
    nb = nets.NetBuilder(H, W)
    x0 = nb.conv(-1, cin - 3 if cin % 4 else cin, 1, 1, 0)
    if nb.shape(x0)[2] < cin:
        x0 = nb.concat(x0, -1)
    nb.conv(x0, cout, k, 1, k // 2, 0, groups=groups)
    li = len(nb.layers) - 1
    wts = g.normal(0, np.sqrt(2.0 / (k * k * cin / groups)), size=(cout, k, k, cin // groups)).astype(np.float32)
    bias = g.normal(0, 0.1, size=cout).astype(np.float32)
    ws = [np.zeros((l["cout"], 1, 1, 3), np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [wts]
    bs = [np.zeros(l["cout"], np.float32) if l["kind"] == 0 else None for l in nb.layers[:-1]] + [bias]
    x = torch.from_numpy(g.normal(size=(S, H, W, cin)).astype(np.float32)).cuda()
    want = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), torch.from_numpy(wts).cuda().double().permute(0, 3, 1, 2),
                                      torch.from_numpy(bias).cuda().double(), padding=k // 2, groups=groups).permute(0, 2, 3, 1)
    seen = torch.zeros((S, H, W), dtype=torch.bool, device="cuda")
    for y in range(0, H, 16):
        for xx in range(0, W, 8):
            x[:, y, xx, ::cin // groups] = float("inf")             # in every group's first channel
            seen[:, max(0, y - k // 2):y + k // 2 + 1, max(0, xx - k // 2):xx + k // 2 + 1] = True
    clear, plain = ~seen, torch.where(torch.isinf(x), 1.0, x)
    outs, us, us_plain = [], [], []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(W, H, nb.layers, ws, bs, n_streams=S, block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
        out = dc.conv_partial(li, x)
        assert not torch.isfinite(out[seen]).any() and torch.isfinite(out[clear]).all()
        assert (out.double() - want)[clear].norm() < 6e-7 * want[clear].norm()
        outs.append(out.clone())
        for inp, times in ((x, us), (plain, us_plain)):
            best = 1e9
            for _ in range(5):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                B.dc_conv_partial(dc.handle, li, inp, None, None, None, out)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) * 1e3)
            times.append(best)
        dc.close()
    assert torch.equal(outs[0][clear], outs[1][clear]) and torch.allclose(*outs, rtol=0, atol=0, equal_nan=True)
    assert us[0] <= 5 * us[1] + 50
    assert S * H * W < 40000 or us_plain[0] < us_plain[1]           # without such values no tile goes there: 43 and 118 us


@pytest.mark.parametrize("cin,cout,k,H,W,S,groups", [(32, 64, 3, 48, 40, 1, 1), (64, 32, 1, 33, 21, 2, 1), (40, 72, 5, 30, 22, 2, 2), (64, 64, 3, 113, 113, 4, 1)])
def test_conv_fp32_sums_of_both_signs_beyond_the_largest_float(cin, cout, k, H, W, S, groups, monkeypatch):
    """Terms of either sign whose partial sums overflow: what is not finite is as the CUDA-core kernel has it, bit for bit (its order
    decides between infinity and NaN); what is finite is right."""
    g = rng(cin + 2 * cout + k)
    nb = nets.NetBuilder(H, W)
    nb.conv(nb.conv(-1, cin, 1, 1, 0), cout, k, 1, k // 2, 0, groups=groups)
    wts = np.ldexp(g.normal(size=(cout, k, k, cin // groups)).astype(np.float32), 63)
    x = torch.from_numpy(np.ldexp(g.normal(size=(S, H, W, cin)).astype(np.float32), 61)).cuda()
    out = []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(W, H, nb.layers, [np.zeros((cin, 1, 1, 3), np.float32), wts], [np.zeros(cin, np.float32), np.zeros(cout, np.float32)], n_streams=S,
                       block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
        out.append(dc.conv_partial(1, x))
        dc.close()
    got, want = out
    bad = ~torch.isfinite(got)
    assert bad.sum() > 0.01 * got.numel() and (~bad).sum() > 0.01 * got.numel()
    assert torch.allclose(got[bad], want[bad], rtol=0, atol=0, equal_nan=True)
    conv = lambda a, b: torch.nn.functional.conv2d(a.double().permute(0, 3, 1, 2), torch.from_numpy(b).cuda().double().permute(0, 3, 1, 2), padding=k // 2, groups=groups).permute(0, 2, 3, 1)
    assert ((got.double() - conv(x, wts)).abs() <= 1e-6 * conv(x.abs(), np.abs(wts)))[~bad].all()


@pytest.mark.parametrize("e,f", [(-100, 60), (-108, 60), (-112, 60), (-118, 100), (-122, 100), (-126, 100), (-140, 120), (60, -105), (100, -112), (100, -118), (110, -126)])
def test_conv_fp32_operands_too_small_to_split(e, f, monkeypatch):
    """Inputs of 2^e and weights of 2^f: the third bf16 piece of a float below 2^-110 is cut, or all of them.  Against 64-bit sums and the
    CUDA-core kernel: the error in the 2-norm is no larger than the latter's (0.6 to 0.7 of it)."""
    g = rng(79)
    nb = nets.NetBuilder(48, 40)
    nb.conv(nb.conv(-1, 32, 1, 1, 0), 64, 3, 1, 1, 0)
    wts = np.ldexp(g.normal(size=(64, 3, 3, 32)).astype(np.float32), f)
    x = np.zeros((1, 48, 40, 32), np.float32)
    x[:, :30] = np.ldexp(g.normal(size=(1, 30, 40, 32)).astype(np.float32), e)      # (zeros split)
    x = torch.from_numpy(x).cuda()
    want = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), torch.from_numpy(wts).cuda().double().permute(0, 3, 1, 2), padding=1).permute(0, 2, 3, 1)
    err = []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(40, 48, nb.layers, [np.zeros((32, 1, 1, 3), np.float32), wts], [np.zeros(32, np.float32), np.zeros(64, np.float32)],
                       n_streams=1, block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
        err.append(float((dc.conv_partial(1, x).double() - want).norm() / want.norm()))
        dc.close()
    assert err[0] <= 1.1 * err[1] and err[1] < 3e-7


@pytest.mark.parametrize("e,f", [(-55, -55), (-60, -60), (-63, -63), (-66, -66), (-70, -70), (-73, -70), (-20, -100)])
def test_conv_fp32_products_where_floats_have_fewer_bits(e, f, monkeypatch):
    """Inputs of 2^e and weights of 2^f that split, but whose small products or sums lie under the smallest normal float: no further from 64-bit
    sums than the CUDA-core kernel."""
    g = rng(79)
    nb = nets.NetBuilder(48, 40)
    nb.conv(nb.conv(-1, 32, 1, 1, 0), 64, 3, 1, 1, 0)
    wts = np.ldexp(g.normal(size=(64, 3, 3, 32)).astype(np.float32), f)
    x = np.zeros((1, 48, 40, 32), np.float32)
    x[:, :30] = np.ldexp(g.normal(size=(1, 30, 40, 32)).astype(np.float32), e)      # (zeros split)
    x = torch.from_numpy(x).cuda()
    want = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), torch.from_numpy(wts).cuda().double().permute(0, 3, 1, 2), padding=1).permute(0, 2, 3, 1)
    err = []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(40, 48, nb.layers, [np.zeros((32, 1, 1, 3), np.float32), wts], [np.zeros(32, np.float32), np.zeros(64, np.float32)],
                       n_streams=1, block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
        err.append(float((dc.conv_partial(1, x).double() - want).norm() / want.norm()))
        dc.close()
    assert err[0] <= err[1]


def test_conv_fp32_weights_that_do_not_split(monkeypatch):
    g = rng(78)
    nb = nets.NetBuilder(24, 40)
    nb.conv(nb.conv(-1, 16, 1, 1, 0), 32, 3, 1, 1, 0)
    wts = g.normal(0, 0.1, size=(32, 3, 3, 16)).astype(np.float32)
    wts[3, 1, 1, 2] = 3.402e38
    x = torch.from_numpy(g.uniform(-0.2, 0.2, size=(1, 24, 40, 16)).astype(np.float32)).cuda()
    out = []
    for cores in (False, True):
        if cores:
            monkeypatch.setenv("DC_NO_TENSOR_CORES", "1")
        dc = DeepCache(40, 24, nb.layers, [np.zeros((16, 1, 1, 3), np.float32), wts], [np.zeros(16, np.float32), np.zeros(32, np.float32)], n_streams=1,
                       block=16, search_range=4, dtype=B.DC_FP32, max_regions=4)
        out.append(dc.conv_partial(1, x))
        dc.close()
    assert torch.isfinite(out[0]).all() and torch.equal(*out)
