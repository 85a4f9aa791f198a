"""The work that users of the framework have it do, as cases that can be timed and compared.

A deployment runs video streams through a cache: `infer` is the loop of `DeepCache.infer_frame` (optionally announcing
the next frame), from one stream (latency) to a server's batch; `host` is the same with frames in pinned host memory;
`calls` is a program with an executor of its own, which calls the matcher, region propagation and the partial
convolution one by one; `search` is the block search for programs that may not allocate.  A pass is one new frame of
every stream.  Frames are a textured canvas that pans, with a disturbance that no motion explains, and are visited back
and forth, so that every pass has the motion of a video; every `expire`-th frame is a full one, as in use.
"""
import math

import numpy as np
import torch

from paper_1712_01670_b200 import binding as B
from paper_1712_01670_b200.engine import DeepCache
from paper_1712_01670_b200.synth import nets

FRAMES = 4                                   # distinct frames of a state, visited 0 1 2 3 2 1 0 ...
SEARCH = {"exhaustive": B.DC_SEARCH_EXHAUSTIVE, "diamond": B.DC_SEARCH_DIAMOND, "three_step": B.DC_SEARCH_THREE_STEP}
# share of a trunk's convolution work that its kind of video leaves to compute (the rest comes from the cache)
FRESH = {"small_cnn": 0.35, "convs": 0.5, "inception": 0.6}


def case(name, do, net, width, height, streams, dtype, block=16, range_=16, search="diamond", motion=3, disturb="patches", ahead=False,
         expire=10, skip=1, pool=False, own_vectors=False):
    c = dict(do=do, net=net, width=width, height=height, streams=streams, dtype=dtype, block=block, range=range_, search=search,
             motion=motion, disturb=disturb, ahead=ahead, expire=expire, skip=skip, pool=pool, own_vectors=own_vectors)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest use: one layer on a 64 x 64 image, step by step (the tiny workload)
        case("calls 64x64 one stream", "calls", "convs", 64, 64, 1, "fp32", block=8, range_=8, search="exhaustive"),
        # one camera, float network (the small CNN workload as it stands)
        case("small cnn one stream", "infer", "small_cnn", 227, 227, 1, "fp32", disturb="rects"),
        # one camera, latency, next frame announced (the AlexNet and ResNet-50 workloads as they stand)
        case("alexnet one stream", "infer", "alexnet", 227, 227, 1, "bf16", motion=4, ahead=True),
        case("resnet50 one stream", "infer", "resnet50", 224, 224, 1, "bf16", range_=24, motion=6, disturb="window", ahead=True),
        # a server's batches: the benchmark's full-HD workload, and the other trunks with many streams
        case("vgg full-hd 32 streams", "infer", "vgg16", 1920, 1080, 32, "bf16", range_=32, motion=8, ahead=True),
        case("resnet50 128 streams", "infer", "resnet50", 224, 224, 128, "bf16", range_=24, motion=6, disturb="window"),
        case("alexnet grouped 96 streams", "infer", "alexnet_grouped", 227, 227, 96, "bf16", motion=4),
        # float network for several cameras with the engine's default matcher settings (the paper's block of 10)
        case("small cnn 24 streams", "infer", "small_cnn", 227, 227, 24, "fp32", block=10, range_=8, disturb="rects"),
        # every layer kind, reuse in pooling and LRN layers too, rectangles with their blocks' own vectors
        case("inception pooled reuse", "infer", "inception", 160, 128, 16, "bf16", range_=8, pool=True, own_vectors=True),
        # frames that arrive in host memory
        case("host vgg 720p 6 streams", "host", "vgg16", 1280, 720, 6, "bf16", range_=32, motion=8),
        # a program with its own executor on full-HD streams
        case("calls full-hd 8 streams", "calls", "convs", 1920, 1080, 8, "bf16", range_=16, search="three_step", motion=6),
        # a program that may not allocate
        case("search 720p 4 streams", "search", "none", 1280, 720, 4, "none", block=10, range_=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: any trunk, frame size (ragged ones too), number of streams, matcher setting."""
    largest = max(_weight(c) for c in listed())
    kind = rng.choice(["trunk", "trunk", "trunk", "small_cnn", "small_cnn", "inception", "host", "calls", "calls", "search"])
    disturb, motion, block = rng.choice(["patches", "rects", "window"]), rng.randint(2, 8), rng.choice([16, 16, 16, 10, 8])
    range_ = rng.randint(8, 32) if block == 16 else rng.randint(6, 12)
    if kind == "trunk":
        net = rng.choice(["alexnet", "alexnet_grouped", "resnet50", "vgg16"])
        w, h = (_log_int(rng, 320, 1920), _log_int(rng, 240, 1080)) if net == "vgg16" else (rng.randint(200, 260), rng.randint(200, 260))
        c = case("", "infer", net, w, h, _log_int(rng, 1, 128), "bf16", block, range_, motion=motion, disturb=disturb,
                 ahead=rng.random() < 0.5, skip=rng.choice([1, 1, 1, 2]), expire=rng.choice([10, 10, 20]))
    elif kind == "small_cnn":
        c = case("", "infer", "small_cnn", rng.randint(120, 330), rng.randint(120, 330), _log_int(rng, 1, 32), rng.choice(["fp32", "fp32", "bf16"]),
                 block, range_, motion=motion, disturb=disturb, ahead=rng.random() < 0.3, own_vectors=rng.random() < 0.2)
    elif kind == "inception":
        c = case("", "infer", "inception", rng.randint(64, 190), rng.randint(64, 190), _log_int(rng, 1, 64), rng.choice(["bf16", "fp32"]),
                 block, range_, motion=motion, disturb=disturb, pool=rng.random() < 0.7, own_vectors=rng.random() < 0.5)
    elif kind == "host":
        net = rng.choice(["vgg16", "alexnet", "resnet50"])
        w, h = (_log_int(rng, 320, 1920), _log_int(rng, 240, 1080)) if net == "vgg16" else (rng.randint(200, 260), rng.randint(200, 260))
        c = case("", "host", net, w, h, _log_int(rng, 1, 12), "bf16", block, range_, motion=motion, disturb=disturb)
    elif kind == "calls":
        search = rng.choice(["diamond", "three_step", "exhaustive"])
        top = 640 if search == "exhaustive" else 1920
        c = case("", "calls", "convs", _log_int(rng, 64, top), _log_int(rng, 64, top * 9 // 16), _log_int(rng, 1, 16), rng.choice(["bf16", "fp32"]),
                 block, min(range_, 16), search, motion=motion, disturb=disturb, own_vectors=rng.random() < 0.3)
    else:
        search = rng.choice(["diamond", "diamond", "exhaustive"])
        top = 480 if search == "exhaustive" else 1920
        c = case("", "search", "none", _log_int(rng, 96, top), _log_int(rng, 96, top * 9 // 16), _log_int(rng, 1, 16), "none", block,
                 min(range_, 16 if search == "diamond" else 8), search, motion=motion, disturb=disturb)
    while c["streams"] > 1 and _weight(c) > largest:
        c["streams"] = c["streams"] * 2 // 3
    return c


# ---- networks -------------------------------------------------------------------------------------------------------
def _layers(c):
    w, h = c["width"], c["height"]
    if c["net"] == "small_cnn":
        return nets.small_cnn(h, w)
    if c["net"] in ("alexnet", "alexnet_grouped"):
        return nets.alexnet_trunk(h, w, grouped=c["net"] == "alexnet_grouped")
    if c["net"] == "resnet50":
        return nets.resnet50_trunk(h, w)
    if c["net"] == "vgg16":
        return nets.vgg16_trunk(224, 224, h, w)
    if c["net"] == "inception":
        return nets.inception_lrn_net(h, w)
    b = nets.NetBuilder(h, w)                                # "convs": two convolutions, after an area resize when frames are large
    x = b.resize_area(-1, 224, 224) if w >= 224 and h >= 224 else -1
    x = b.conv(x, 16 if w * h <= 64 * 64 else 64, 3, 1, 1)
    b.conv(x, 64, 3, 1, 1)
    return b.layers


def _weights(layers, gen):
    """He-normal weights and small biases (the last convolution of a residual branch at half scale), as numpy arrays."""
    into_add = {l["in0"] for l in layers if l["kind"] == nets.KIND_ADD}
    ws, bs = [], []
    for i, l in enumerate(layers):
        if l["kind"] not in (nets.KIND_CONV, nets.KIND_FC):
            ws.append(None)
            bs.append(None)
            continue
        shape = (l["cout"], l["kh"], l["kw"], l["cin"] // max(1, l.get("groups", 1)))
        sd = math.sqrt(2.0 / (shape[1] * shape[2] * shape[3])) * (0.5 if i in into_add else 1.0)
        ws.append((torch.randn(shape, generator=gen, device="cuda") * sd).cpu().numpy())
        bs.append((torch.randn(l["cout"], generator=gen, device="cuda") * 0.05).cpu().numpy())
    return ws, bs


# ---- frames ---------------------------------------------------------------------------------------------------------
def _canvas(size, gen):
    """Toroidal value noise, four octaves, uint8."""
    acc = torch.zeros((size, size, 3), device="cuda")
    for period, amp in ((64, 1.0), (32, 0.5), (16, 0.25), (8, 0.125)):
        n = size // period
        lat = torch.rand((n, n, 3), generator=gen, device="cuda")
        pos = torch.arange(size, device="cuda") / period
        i0 = pos.long() % n
        i1, f = (i0 + 1) % n, pos - pos.floor()
        rows = lat[:, i0] * (1 - f)[None, :, None] + lat[:, i1] * f[None, :, None]
        acc += amp * (rows[i0] * (1 - f)[:, None, None] + rows[i1] * f[:, None, None])
    acc -= acc.min()
    return (acc * (255.0 / acc.max())).round().to(torch.uint8)


def _frames(c, gen, rng):
    """FRAMES consecutive frames of every stream, (FRAMES, S, H, W, 3) uint8 on the GPU."""
    S, H, W = c["streams"], c["height"], c["width"]
    size = 512
    while size < max(H, W):
        size *= 2
    canvas = _canvas(size, gen)
    out = torch.empty((FRAMES, S, H, W, 3), dtype=torch.uint8, device="cuda")
    ay, ax = torch.arange(H, device="cuda"), torch.arange(W, device="cuda")
    patch = 64 if H >= 480 else 24
    n_patch = math.ceil((0.2 if H >= 480 else 0.1) * H * W / (patch * patch))
    for s in range(S):
        pos = rng.integers(0, size, 2)
        rect, vel, col = rng.integers(0, max(1, min(H, W) - 32), (3, 2)), rng.integers(-4, 5, (3, 2)), rng.integers(0, 256, (3, 3), dtype=np.uint8)
        wh, ww = int(round(H * math.sqrt(0.15))), int(round(W * math.sqrt(0.15)))
        win = rng.integers(0, (H - wh, W - ww))
        for t in range(FRAMES):
            if t:
                speed, angle = rng.integers(0, c["motion"] + 1), rng.random() * 2 * math.pi
                pos = pos + np.rint([speed * math.sin(angle), speed * math.cos(angle)]).astype(np.int64)
            y, x = ay, ax
            if c["disturb"] == "window":                      # zoom jitter of two per cent about the centre
                z = 1.0 + (rng.random() * 2 - 1) * 0.02
                y, x = (((ay - H / 2) / z + H / 2).round().long(), ((ax - W / 2) / z + W / 2).round().long())
            f = out[t, s]
            f.copy_(canvas[((y + int(pos[0])) % size)[:, None], ((x + int(pos[1])) % size)[None, :]])
            if c["disturb"] == "rects":                       # solid rectangles that move on their own
                for r in range(3):
                    ry, rx = np.clip(rect[r] + t * vel[r], 0, (max(0, H - 32), max(0, W - 32)))
                    f[ry:ry + 32, rx:rx + 32] = torch.from_numpy(col[r]).cuda()
            elif c["disturb"] == "patches":                   # squares of fresh noise
                p = min(patch, H, W)
                at = torch.from_numpy(rng.integers(0, (H - p + 1, W - p + 1), (n_patch, 2))).cuda()
                k = torch.arange(p, device="cuda")
                noise = torch.randint(0, 256, (n_patch * p * p, 3), generator=gen, device="cuda", dtype=torch.uint8)
                order = torch.full((H, W), -1, dtype=torch.long, device="cuda")       # later squares lie over earlier ones
                idx = (at[:, :1] + k)[:, :, None] * W + (at[:, 1:] + k)[:, None, :]
                order.view(-1).scatter_reduce_(0, idx.reshape(-1), torch.arange(n_patch * p * p, device="cuda"), "amax")
                hit = order >= 0
                f[hit] = noise[order[hit]]
            else:                                             # one window of fresh noise
                wy, wx = np.clip(win + t * 3, 0, (H - wh, W - ww))
                f[wy:wy + wh, wx:wx + ww] = torch.randint(0, 256, (wh, ww, 3), generator=gen, device="cuda", dtype=torch.uint8)
    return out


# ---- states and passes ----------------------------------------------------------------------------------------------
_streams = []


def _raised_stream():
    """The program's one stream of raised priority: its caches work on it one after the other."""
    if not _streams:
        _streams.append(torch.cuda.Stream(priority=-1))
    return _streams[0]


def _order(i):
    i %= 2 * FRAMES - 2
    return i if i < FRAMES else 2 * FRAMES - 2 - i


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    frames = _frames(c, gen, rng)
    S, W, H = c["streams"], c["width"], c["height"]
    st = dict(c=c, frames=frames, i=0, pitch=W * 3)
    gx, gy = -(-W // c["block"]), -(-H // c["block"])
    grids = dict(mv=torch.zeros((S, gy, gx, 2), dtype=torch.int16, device="cuda"), sse=torch.zeros((S, gy, gx), dtype=torch.int32, device="cuda"),
                 matched=torch.zeros((S, gy, gx), dtype=torch.uint8, device="cuda"), gmv=torch.zeros((S, 3), dtype=torch.int32, device="cuda"))
    if c["do"] == "search":
        st.update(grids)
        return st
    layers = _layers(c)
    ws, bs = _weights(layers, gen)
    # the cache works on the stream that is current when it is made; a program that announces frames gives it a raised priority
    st["stream"] = _raised_stream() if c["ahead"] else torch.cuda.current_stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st["stream"]):
        dc = DeepCache(W, H, layers, ws, bs, n_streams=S, block=c["block"], search_range=c["range"], search=SEARCH[c["search"]],
                       expire_n=c["expire"], dtype=B.DC_BF16 if c["dtype"] == "bf16" else B.DC_FP32, skip_k=c["skip"],
                       region_mode=B.DC_REGIONS_PER_BLOCK if c["own_vectors"] else B.DC_REGIONS_GLOBAL, cache_pool=c["pool"])
    st["dc"], st["views"] = dc, {}
    st["last"] = max(i for i, l in enumerate(layers) if l["kind"] == nets.KIND_CONV)
    if c["do"] == "host":
        st["frames"] = frames.cpu().pin_memory()
        st["out"] = torch.zeros(dc.out_shape(-1), dtype=dc.tdtype).pin_memory()
        B.dc_prefetch_frame_host(dc.handle, st["frames"][0].data_ptr(), st["pitch"])
        _host(st)
    elif c["do"] == "infer":
        _infer(st)                                            # the stream is running: the next pass is a cached frame
    else:
        st.update(grids)
        st["n"] = torch.zeros((S,), dtype=torch.int32, device="cuda")
        st["regions"] = torch.zeros((S, dc.max_regions, 6), dtype=torch.int32, device="cuda")
        first = len(layers) - 2
        st["first"], st["table"] = first, torch.zeros((2, S, dc.max_regions, 6), dtype=torch.int32, device="cuda")
        maps = frames.reshape(FRAMES * S, H, W, 3).permute(0, 3, 1, 2)
        size = (layers[first]["out_h"], layers[first]["out_w"])
        chunks = [torch.nn.functional.adaptive_avg_pool2d(m.float() / 255, size).permute(0, 2, 3, 1).to(dc.tdtype) for m in maps.split(8)]
        st["in"] = torch.cat(chunks).reshape(FRAMES, S, *size, 3).contiguous()
        st["maps"] = [[torch.zeros(dc.out_shape(first + k), dtype=dc.tdtype, device="cuda") for _ in range(2)] for k in range(2)]
        B.dc_cache_set_key(dc.handle, frames[0], st["pitch"])
        B.dc_conv_partial(dc.handle, first, st["in"][0], None, None, None, st["maps"][0][0])
        B.dc_conv_partial(dc.handle, first + 1, st["maps"][0][0], None, None, None, st["maps"][1][0])
        st["i"] = 1
    torch.cuda.synchronize()
    return st


class _CacheMap:
    """A map inside a cache for torch.as_tensor; the tensor keeps this object, and so the cache that owns the memory, alive."""

    def __init__(self, dc, ptr, layer):
        self.dc = dc
        typestr = "<i2" if dc.tdtype == torch.bfloat16 else "<f4"
        self.__cuda_array_interface__ = dict(shape=dc.out_shape(layer), typestr=typestr, data=(ptr, False), version=2)


def _features(st):
    """The last convolution's map inside the cache (what the next frame may reuse; a head would read it), as a tensor."""
    dc, layer = st["dc"], st["last"]
    ptr, _ = B.dc_cache_layer_map(dc.handle, layer)
    if ptr not in st["views"]:
        st["views"][ptr] = torch.as_tensor(_CacheMap(dc, ptr, layer), device=dc.device).view(dc.tdtype)
    return st["views"][ptr]


def _infer(st):
    dc, frames, i = st["dc"], st["frames"], st["i"]
    out = dc.infer_frame(frames[_order(i)])
    features = _features(st)
    if st["c"]["ahead"]:
        B.dc_lookahead_frame(dc.handle, frames[_order(i + 1)], st["pitch"])
    st["i"] = i + 1
    return out, features


def _host(st):
    dc, frames, i = st["dc"], st["frames"], st["i"]
    B.dc_prefetch_frame_host(dc.handle, frames[_order(i + 1)].data_ptr(), st["pitch"])
    B.dc_infer_frame_host(dc.handle, frames[_order(i)].data_ptr(), st["pitch"], st["out"].data_ptr())
    st["i"] = i + 1
    return st["out"], _features(st)


def _calls(st):
    h, i, first, regs = st["dc"].handle, st["i"], st["first"], st["table"]
    cur, (m0, m1) = _order(i), st["maps"]
    old, new = (i - 1) & 1, i & 1
    B.dc_match_blocks(h, st["frames"][cur], st["pitch"], st["mv"], st["sse"], st["matched"], st["gmv"], st["regions"], st["n"])
    B.dc_propagate_regions(h, st["regions"], st["n"], first, first + 2, regs)
    B.dc_conv_partial(h, first, st["in"][cur], m0[old], regs[0], st["n"], m0[new])
    B.dc_conv_partial(h, first + 1, m0[new], m1[old], regs[1], st["n"], m1[new])
    B.dc_cache_set_key(h, st["frames"][cur], st["pitch"])
    st["i"] = i + 1
    return dict(mv=st["mv"], sse=st["sse"], matched=st["matched"], gmv=st["gmv"], n=st["n"], regions=regs, out0=m0[new], out1=m1[new])


def _search(st):
    c, i, f = st["c"], st["i"], st["frames"]
    B.dc_search_blocks_noalloc(f[_order(i + 1)], f[_order(i)], st["pitch"], c["width"], c["height"], c["streams"], c["block"], c["range"],
                               SEARCH[c["search"]], 20.0, st["mv"], st["sse"], st["gmv"])
    st["i"] = i + 1
    return dict(mv=st["mv"], sse=st["sse"], gmv=st["gmv"])


def run(state):
    do = state["c"]["do"]
    if do == "search":
        return _search(state)
    with torch.cuda.stream(state["stream"]):
        return _infer(state) if do == "infer" else _host(state) if do == "host" else _calls(state)


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    c = case
    S, frame = c["streams"], c["streams"] * c["width"] * c["height"] * 3
    blocks = S * (-(-c["width"] // c["block"])) * (-(-c["height"] // c["block"]))
    if c["do"] == "search":                                   # both frames in, a vector and a score per block out
        return {"bytes": 2 * frame + 8 * blocks, "flops": 0}
    elt = 2 if c["dtype"] == "bf16" else 4
    layers = _layers(c)
    weights = sum(l["cout"] * l["kh"] * l["kw"] * (l["cin"] // max(1, l["groups"])) for l in layers if l["kind"] in (0, 7))
    macs = sum(l["out_h"] * l["out_w"] * l["cout"] * l["kh"] * l["kw"] * (l["cin"] // max(1, l["groups"])) for l in layers if l["kind"] in (0, 7))
    last, conv = layers[-1], [l for l in layers if l["kind"] == 0][-1]
    out = S * last["out_h"] * last["out_w"] * last["cout"] * elt
    kept = S * conv["out_h"] * conv["out_w"] * conv["cout"] * elt
    # the new frame is read and kept as the next key, the previous one is read; weights once; the output and the features once
    bytes_ = 3 * frame + weights * elt + out + (kept if conv is not last else 0)
    if c["do"] == "calls":
        a = layers[-2]
        bytes_ += S * a["out_h"] * a["out_w"] * (3 + 3 * a["cout"]) * elt + 2 * out + 9 * blocks
    return {"bytes": bytes_, "flops": 2.0 * S * macs * FRESH.get(c["net"], 0.95)}


def _weight(c):
    """A pass's cost for keeping drawn cases within the listed ones': bytes, operations, and the exhaustive search's candidates."""
    w = work(c)
    share = (2 * c["range"] + 1) ** 2 if c["search"] == "exhaustive" else 0
    rate = 50 if c["dtype"] == "bf16" else 5
    return max(w["bytes"], w["flops"] / rate, share * c["streams"] * c["width"] * c["height"] / 20)


def tolerance(case):
    # integers (vectors, scores, rectangles) exact; bf16 maps: rounding of every layer's output; fp32 maps: the order of sums
    return "exact" if case["do"] == "search" else {"rel": 1e-2, "max": 0.2} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 1e-3}
