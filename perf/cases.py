"""The workloads by which this library's speed is measured.

Every case is one pass of a program that uses the library through its public
calls: one graph on one frame, a batch of frames, or requests to a server, on
device memory the program owns (torch tensors wrapped as images).  The graphs
are the ones the library's benchmark and tests run: the edge detector, the
corner detectors, the applications of the paper's evaluation, morphology,
camera statistics.  Frames are synthetic: rectangles of random grey on a random
background plus Gaussian noise (sigma 10).

  listed()           the cases
  draw(rng)          one more case of the same ranges
  prepare(case, s)   inputs of seed s, images, verified graphs
  run(state)         one pass and its outputs
  work(case)         bytes and operations no pass can do without
  exact(case, s)     the outputs in 64-bit torch arithmetic
"""
import math

import numpy as np
import torch

from paper_2008_11476_gb300 import apps as A
from paper_2008_11476_gb300 import graphs as PG
from paper_2008_11476_gb300 import hvx as H
from paper_2008_11476_gb300 import synth

BORDERS = {"replicate": H.HVX_BORDER_REPLICATE, "undefined": H.HVX_BORDER_UNDEFINED,
           "constant": H.HVX_BORDER_CONSTANT}
THRESHOLD = 100          # edge masks
CORNER_THRESHOLD = {"harris": 1e6, "tomasi": A.TOMASI_THRESHOLD}
SERVE_SIZES = [(640, 480), (1920, 1080), (3840, 2160)]
MAX_PIXELS = 100e6       # of a drawn case


def _case(name, graph, w, h, n=1, call="frame", border="replicate", response=False, mixed=False):
    return {"name": name, "graph": graph, "w": w, "h": h, "n": n, "call": call, "border": border,
            "response": response, "mixed": mixed}


def listed():
    return [
        # the smallest call: a denoising filter on one VGA frame, launch latency
        _case("gaussian 640x480", "gaussian", 640, 480),
        # a video loop: the edge detector on each full-HD frame as it arrives
        _case("edge 1080p", "edge", 1920, 1080),
        # the headline: the edge detector over a buffered clip, one batch call
        _case("edge 64 x 1080p", "edge", 1920, 1080, 64, "batch"),
        # an image collection: 256 pictures of any size in one batch call
        _case("edge 256 mixed", "edge", 3840, 2160, 256, "batch", mixed=True),
        # corner detection on 4K film frames
        _case("harris 16 x 4096x2160", "harris", 4096, 2160, 16, "batch", "undefined"),
        # corners with the binary32 response kept (for ranking), replicated
        # borders, one frame of the paper's size
        _case("harris response 1020x1020", "harris", 1020, 1020, 1, "frame", "replicate", True),
        # the tracker's corner measure (Shi-Tomasi) over full-HD frames
        _case("tomasi 16 x 1080p", "tomasi", 1920, 1080, 16, "batch", "undefined"),
        # a chain of three convolutions: custom filters that run fused
        _case("fchain 16 x 1080p", "fchain", 1920, 1080, 16, "batch"),
        # sharpening of photographs of an odd size, S16 results
        _case("unsharp 16 x 2043x1361", "unsharp", 2043, 1361, 16, "batch"),
        # morphology (closing, difference, median, mask) on each frame
        _case("morphology 1080p", "morphology", 1920, 1080),
        # camera statistics: luma of a UYVY 4K frame, mean and deviation,
        # extrema, histogram and an equalised copy
        _case("statistics 3840x2160", "statistics", 3840, 2160),
        # serving: 32 requests of all graphs and sizes that arrive together
        _case("serve 32 requests", "serve", 3840, 2160, 32, "server"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same graphs: sizes from thumbnails to 4K, odd ones among
    them, single frames and batches."""
    graph = rng.choice(["gaussian", "edge", "edge", "harris", "tomasi", "fchain", "unsharp",
                        "laplacian", "gauss5", "sobel", "sobel_x", "edgfig2", "morphology",
                        "statistics", "serve"])
    if graph == "serve":
        return _unnamed(_case("", graph, 3840, 2160, rng.randint(8, 32), "server"))
    w, h = _log_int(rng, 64, 4096), _log_int(rng, 48, 2160)
    border, response = "replicate", False
    if graph in ("gaussian", "edge"):
        border = rng.choice(["replicate", "replicate", "undefined", "constant"])
    if graph in ("harris", "tomasi"):
        border = rng.choice(["undefined", "undefined", "replicate"])
        response = graph == "harris" and rng.random() < 0.3
    if graph == "statistics":
        return _unnamed(_case("", graph, max(64, w // 2 * 2), h))
    if rng.random() < 0.4:
        return _unnamed(_case("", graph, w, h, 1, "frame", border, response))
    most = max(2, min(64, int(MAX_PIXELS / (w * h))))
    mixed = graph in ("edge", "gaussian") and rng.random() < 0.3
    return _unnamed(_case("", graph, w, h, _log_int(rng, 2, most), "batch", border, response,
                          mixed))


def _unnamed(case):
    del case["name"]
    return case


# ---------------------------------------------------------------------------
# What a case computes

def _sizes(case):
    """(width, height) of every frame."""
    w, h, n = case["w"], case["h"], case["n"]
    if case["graph"] == "serve":
        return [SERVE_SIZES[k] for k in _serve_mix(n)[1]]
    if case["mixed"]:
        return synth.batch_sizes(n, seed=4, wlo=max(64, w // 12), whi=w, hlo=max(48, h // 9), hhi=h)
    return [(w, h)] * n


def _serve_mix(n):
    """Graph and size index of every request: half Gaussian3x3, 30 % edge,
    20 % Harris; a third of each size."""
    return (synth.choice(5, 30, n, [0.5, 0.3, 0.2]), synth.choice(5, 31, n, [1, 1, 1]))


def _graphs(case):
    if case["graph"] == "serve":
        return [("gaussian", "edge", "harris")[k] for k in _serve_mix(case["n"])[0]]
    return [case["graph"]] * case["n"]


def _outputs(graph, case):
    """name -> hvx format of a graph's output images."""
    if graph == "edge":
        return {"phase": H.HVX_DF_U8, "mask": H.HVX_DF_U8}
    if graph in ("harris", "tomasi"):
        out = {"mask": H.HVX_DF_U8}
        if case["response"]:
            out["response"] = H.HVX_DF_F32
        return out
    if graph in ("unsharp", "laplacian", "sobel_x"):
        return {"out": H.HVX_DF_S16}
    return {"out": H.HVX_DF_U8}


# operations a pixel: adds, multiplies, compares of the definitions with
# separable filters done by rows and columns
_OPS = {"gaussian": 9, "edge": 9 + 10 + 5 + 20, "harris": 10 + 3 + 24 + 8, "tomasi": 10 + 3 + 24 + 12,
        "fchain": 9 + 17 + 7, "unsharp": 12, "laplacian": 6, "gauss5": 17, "sobel": 15, "sobel_x": 6,
        "edgfig2": 9 + 5 + 4, "morphology": 8 + 8 + 38 + 4, "statistics": 10}


def work(case):
    nbytes = ops = 0
    for (w, h), g in zip(_sizes(case), _graphs(case)):
        inb = 2 if g == "statistics" else 1
        outb = sum(H.BYTES_PER_PIXEL[f] for f in _outputs(g, case).values())
        nbytes += w * h * (inb + outb)
        ops += w * h * _OPS[g]
    return {"bytes": nbytes, "flops": ops}


# ---------------------------------------------------------------------------
# Inputs

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _scene(w, h, gen, dev):
    """Rectangles on a background, float32 (h, w)."""
    n = max(8, min(200, w * h // 20000))
    u = torch.rand((n, 5), generator=gen, device=dev).cpu().numpy()
    img = torch.full((h, w), float(int(u[0, 4] * 256)), device=dev)
    for a, b, c, d, v in u:
        rw = max(1, w // 50) + int(a * (w // 4 - w // 50 + 1))
        rh = max(1, h // 50) + int(b * (h // 4 - h // 50 + 1))
        x, y = int(c * (w - rw + 1)), int(d * (h - rh + 1))
        img[y:y + rh, x:x + rw] = float(int(v * 256))
    return img


def _noisy(scene, gen):
    noise = torch.randn(scene.shape, generator=gen, device=scene.device)
    return (scene + 10.0 * noise + 0.5).floor_().clamp_(0, 255).to(torch.uint8)


def _inputs(case, seed):
    """One U8 (h, w) tensor per frame; (h, 2 w) UYVY bytes for statistics."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    sizes = _sizes(case)
    bw, bh = max(s[0] for s in sizes), max(s[1] for s in sizes)
    scenes = [_scene(bw, bh, gen, dev) for _ in range(min(4, len(sizes)))]
    frames = []
    for i, (w, h) in enumerate(sizes):
        s = scenes[i % len(scenes)]
        x, y = (bw - w) // 2, (bh - h) // 2
        frames.append(_noisy(s[y:y + h, x:x + w], gen))
    if case["graph"] == "statistics":
        chroma = torch.randint(0, 256, frames[0].shape, generator=gen, device=dev,
                               dtype=torch.uint8)
        frames = [torch.stack((chroma, frames[0]), dim=2).reshape(frames[0].shape[0], -1)]
    return frames


_TORCH = {H.HVX_DF_U8: torch.uint8, H.HVX_DF_S16: torch.int16, H.HVX_DF_F32: torch.float32}


class _Images:
    """Frames of one format in one allocation, rows 16-byte aligned."""

    def __init__(self, ctx, sizes, fmt):
        self.bpp = H.BYTES_PER_PIXEL[fmt]
        self.sizes, self.fmt = sizes, fmt
        pitches = [(w * self.bpp + 15) // 16 * 16 for w, _ in sizes]
        at = [0]
        for (_, h), p in zip(sizes, pitches):
            at.append(at[-1] + h * p)
        self.bytes = torch.zeros(at[-1], dtype=torch.uint8, device="cuda")
        self.rows = [self.bytes[a:b].view(-1, p) for a, b, p in zip(at, at[1:], pitches)]
        self.images = [H.hvxCreateImageFromHandle(ctx, w, h, fmt, r.data_ptr(), p)
                       for (w, h), r, p in zip(sizes, self.rows, pitches)]

    def whole(self):
        """Every pixel: (n, h, w) for frames of one size, else the allocation."""
        if len(set(self.sizes)) > 1:
            return self.bytes if self.fmt == H.HVX_DF_U8 else self.bytes.view(_TORCH[self.fmt])
        (w, h), n = self.sizes[0], len(self.sizes)
        return self.bytes.view(_TORCH[self.fmt]).view(n, h, -1)[:, :, :w]


class State:
    """What a program holds: a context, images, verified graphs."""

    def __init__(self):
        self.ctx = H.hvxCreateContext()
        self.server = None
        self.nodes = {}

    def __del__(self):
        if self.server is not None:
            H.hvxReleaseServer(self.server)
        H.hvxReleaseContext(self.ctx)


def _border(node, mode):
    H.hvxSetNodeBorder(node, mode, 0)
    return node


def _morphology(ctx, src, out):
    """Closing, its difference from the input, and the input's median where
    that difference is large."""
    g = H.hvxCreateGraph(ctx)
    d, c, diff, mask, med = (H.hvxCreateVirtualImage(g) for _ in range(5))
    H.hvxDilate3x3Node(g, src, d)
    H.hvxErode3x3Node(g, d, c)
    H.hvxMedian3x3Node(g, src, med)
    H.hvxAbsDiffNode(g, c, src, diff)
    H.hvxThresholdNode(g, diff, H.HVX_THRESHOLD_BINARY, 20, 0, 255, 0, mask)
    H.hvxAndNode(g, med, mask, out)
    H.hvxVerifyGraph(g)
    return g


def _statistics(ctx, src, out, nodes):
    g = H.hvxCreateGraph(ctx)
    luma = H.hvxCreateVirtualImage(g)
    H.hvxChannelExtractNode(g, src, H.HVX_CHANNEL_Y, luma)
    nodes["moments"] = H.hvxMeanStdDevNode(g, luma)
    nodes["extrema"] = H.hvxMinMaxLocNode(g, luma)
    nodes["histogram"] = H.hvxHistogramNode(g, luma, 256, 0, 256)
    H.hvxEqualizeHistNode(g, luma, out)
    H.hvxVerifyGraph(g)
    return g


def _convolve(ctx, src, out, coeffs, shift):
    g = H.hvxCreateGraph(ctx)
    k = coeffs.shape[0]
    _border(H.hvxConvolveNode(g, src, coeffs.ravel(), k, k, shift, out), H.HVX_BORDER_REPLICATE)
    H.hvxVerifyGraph(g)
    return g


def _fchain(ctx, src, out):
    g = H.hvxCreateGraph(ctx)
    a, b = (H.hvxCreateVirtualImage(g, 0, 0, H.HVX_DF_U8) for _ in range(2))
    for i, o, c, shift in ((src, a, A.B3, 4), (a, b, A.B5, 8), (b, out, A.SHARPEN, 2)):
        k = c.shape[0]
        _border(H.hvxConvolveNode(g, i, c.ravel(), k, k, shift, o), H.HVX_BORDER_REPLICATE)
    H.hvxVerifyGraph(g)
    return g


def _unsharp(ctx, src, out):
    g = H.hvxCreateGraph(ctx)
    blur = H.hvxCreateVirtualImage(g)
    d, d2 = (H.hvxCreateVirtualImage(g, 0, 0, H.HVX_DF_S16) for _ in range(2))
    _border(H.hvxGaussian3x3Node(g, src, blur), H.HVX_BORDER_REPLICATE)
    H.hvxSubtractNode(g, src, blur, H.HVX_POLICY_SATURATE, d)
    H.hvxAddNode(g, d, d, H.HVX_POLICY_SATURATE, d2)
    H.hvxAddNode(g, src, d2, H.HVX_POLICY_SATURATE, out)
    H.hvxVerifyGraph(g)
    return g


def _sobel_graph(ctx, src, out, graph):
    """The Sobel applications: the gradient mask, gx alone, and Listing 1's
    graph (a Gaussian first, Magnitude of gy alone)."""
    g = H.hvxCreateGraph(ctx)
    gx, gy, m = (H.hvxCreateVirtualImage(g) for _ in range(3))
    if graph == "sobel_x":
        _border(H.hvxSobel3x3Node(g, src, out, None), H.HVX_BORDER_REPLICATE)
    else:
        if graph == "edgfig2":
            blur = H.hvxCreateVirtualImage(g)
            _border(H.hvxGaussian3x3Node(g, src, blur), H.HVX_BORDER_REPLICATE)
            src = blur
        _border(H.hvxSobel3x3Node(g, src, gx, gy), H.HVX_BORDER_REPLICATE)
        H.hvxMagnitudeNode(g, gy if graph == "edgfig2" else gx, gy, m)
        H.hvxThresholdNode(g, m, H.HVX_THRESHOLD_BINARY, THRESHOLD, 0, 255, 0, out)
    H.hvxVerifyGraph(g)
    return g


def _build(graph, case, st, src, out):
    """The verified graph of one frame; `out` maps output names to images."""
    border = BORDERS[case["border"]]
    ctx = st.ctx
    if graph == "gaussian":
        return PG.gaussian_graph(ctx, src, out["out"], border=border)
    if graph == "edge":
        return PG.edge_graph(ctx, src, out["phase"], out["mask"], border=border, thr=THRESHOLD)
    if graph in ("harris", "tomasi"):
        if case["graph"] == "serve":
            border = H.HVX_BORDER_UNDEFINED
        return PG.harris_graph(ctx, src, out["mask"], out.get("response"), border=border,
                               thr=CORNER_THRESHOLD[graph], tomasi=graph == "tomasi")
    if graph == "fchain":
        return _fchain(ctx, src, out["out"])
    if graph == "unsharp":
        return _unsharp(ctx, src, out["out"])
    if graph == "laplacian":
        return _convolve(ctx, src, out["out"], A.LAPLACE, 0)
    if graph == "gauss5":
        return _convolve(ctx, src, out["out"], A.B5, 8)
    if graph == "morphology":
        return _morphology(ctx, src, out["out"])
    if graph == "statistics":
        return _statistics(ctx, src, out["out"], st.nodes)
    return _sobel_graph(ctx, src, out["out"], graph)


def prepare(case, seed):
    st = State()
    st.case = case
    st.stream = torch.cuda.current_stream().cuda_stream
    sizes, graphs = _sizes(case), _graphs(case)
    frames = _inputs(case, seed)
    in_fmt = H.HVX_DF_UYVY if case["graph"] == "statistics" else H.HVX_DF_U8
    st.src = _Images(st.ctx, sizes, in_fmt)
    for rows, f in zip(st.src.rows, frames):
        rows[:, :f.shape[1]] = f
    st.out, per_frame = {}, [{} for _ in sizes]
    for name in sorted({o for g in graphs for o in _outputs(g, case)}):
        have = [i for i, g in enumerate(graphs) if name in _outputs(g, case)]
        fmt = _outputs(graphs[have[0]], case)[name]
        st.out[name] = _Images(st.ctx, [sizes[i] for i in have], fmt)
        for i, img in zip(have, st.out[name].images):
            per_frame[i][name] = img
    st.graphs = [_build(g, case, st, src, out)
                 for g, src, out in zip(graphs, st.src.images, per_frame)]
    if case["call"] == "server":
        st.server = H.hvxCreateServer(st.ctx, 40 << 30, 16, 8)
    st.results = {name: o.whole() for name, o in st.out.items()}  # the program's own buffers
    torch.cuda.synchronize()
    return st


def run(st):
    call = st.case["call"]
    if call == "batch":
        H.hvxProcessGraphBatch(st.graphs, st.stream)
    elif call == "server":
        for t in H.hvxServerSubmitMany(st.server, st.graphs):
            status, _ = H.hvxServerWait(st.server, t)
            if status != H.HVX_SUCCESS:
                raise H.HvxError(status, "request")
    elif st.nodes:  # results on the host
        H.hvxProcessGraph(st.graphs[0])
    else:
        H.hvxScheduleGraph(st.graphs[0], st.stream)
    if not st.nodes:
        return st.results
    out = dict(st.results)
    m = H.hvxGetNodeResult(st.nodes["moments"], H.HvxMeanStdDev())
    x = H.hvxGetNodeResult(st.nodes["extrema"], H.HvxMinMaxLoc())
    out["moments"] = {"mean": m.mean, "stddev": m.stddev, "sum": m.sum,
                      "sum_squares": m.sum_squares, "count": m.count}
    out["extrema"] = {f: getattr(x, f) for f, _ in H.HvxMinMaxLoc._fields_}
    out["histogram"] = H.hvxGetNodeResult(st.nodes["histogram"], np.zeros(256, np.uint32))
    return out


# ---------------------------------------------------------------------------
# The same results in 64-bit torch arithmetic

class _Grid:
    """An int64 image and how many pixels of its rim are not valid (0)."""

    def __init__(self, v, rim=0):
        self.v, self.rim = v, rim

    def map(self, f):
        return _Grid(_rimmed(f(self.v), self.rim), self.rim)


def _rimmed(v, m):
    if m == 0:
        return v
    out = torch.zeros_like(v)
    h, w = v.shape
    if h > 2 * m and w > 2 * m:
        out[m:h - m, m:w - m] = v[m:h - m, m:w - m]
    return out


def _taps(img, r, border):
    """f(dx, dy): the image shifted, read under the border mode."""
    h, w = img.v.shape
    if border == "replicate":
        ys = torch.arange(-r, h + r, device=img.v.device).clamp(0, h - 1)
        xs = torch.arange(-r, w + r, device=img.v.device).clamp(0, w - 1)
        p = img.v[ys][:, xs]
    else:
        p = torch.zeros((h + 2 * r, w + 2 * r), dtype=img.v.dtype, device=img.v.device)
        p[r:r + h, r:r + w] = img.v
    return lambda dx, dy: p[r + dy:r + dy + h, r + dx:r + dx + w]


def _local(img, r, border, f):
    rim = img.rim + (r if border == "undefined" else 0)
    return _Grid(_rimmed(f(_taps(img, r, border)), rim), rim)


def _corr(img, coeffs, border):
    k = coeffs.shape[0]
    r = k // 2

    def total(t):
        acc = 0
        for dy in range(k):
            for dx in range(k):
                if coeffs[dy, dx]:
                    acc = acc + int(coeffs[dy, dx]) * t(dx - r, dy - r)
        return acc
    return _local(img, r, border, total)


_SX = np.array([[-1, 0, 1], [-2, 0, 2], [-1, 0, 1]])


def _clamp(lo, hi):
    return lambda v: v.clamp(lo, hi)


def _shift_sat(img, shift, lo=0, hi=255):
    return img.map(lambda v: (v >> shift).clamp(lo, hi))


def _isqrt_round(s):
    """floor(sqrt(s) + 1/2) of int64 below 2^40."""
    r = torch.sqrt(s.double()).floor().long()
    return r + (s - r * r > r).long()


def _mask(cond):
    return cond.long() * 255


def _exact_frame(graph, case, f):
    """name -> result of one frame (int64 or float64)."""
    b = case["border"]
    if graph == "statistics":
        return _exact_statistics(f)
    img = _Grid(f.long())
    if graph == "gaussian":
        return {"out": _shift_sat(_corr(img, A.B3, b), 4).v}
    if graph == "edge":
        g = _shift_sat(_corr(img, A.B3, b), 4)
        gx, gy = _corr(g, _SX, b), _corr(g, _SX.T, b)
        angle = torch.atan2(gy.v.double(), gx.v.double()) * (128.0 / math.pi)
        mag = _isqrt_round(gx.v ** 2 + gy.v ** 2)
        return {"phase": _rimmed((angle + 0.5).floor().long() % 256, gx.rim),
                "mask": _rimmed(_mask(mag > THRESHOLD), gx.rim)}
    if graph in ("harris", "tomasi"):
        if case["graph"] == "serve":
            b = "undefined"
        gx, gy = _corr(img, _SX, b), _corr(img, _SX.T, b)
        box = np.ones((5, 5), np.int64)
        sxx, syy, sxy = (_corr(_Grid(p * q, gx.rim), box, b) for p, q in
                         ((gx.v, gx.v), (gy.v, gy.v), (gx.v, gy.v)))
        rim, a, d, c = sxx.rim, sxx.v, syy.v, sxy.v
        det, tr = a * d - c * c, a + d
        if graph == "harris":
            q = 25 * det - tr * tr  # 25 R, exact
            out = {"mask": _rimmed(_mask(q > int(25 * CORNER_THRESHOLD[graph])), rim)}
            if case["response"]:
                out["response"] = _rimmed(q.double() / 25.0, rim)
            return out
        root = torch.sqrt(((a - d) ** 2 + 4 * c * c).double())
        den = tr.double() + root
        lam = torch.where(den > 0, 2.0 * det.double() / den.clamp_min(1.0), tr.double())
        return {"mask": _rimmed(_mask(lam > CORNER_THRESHOLD[graph]), rim)}
    if graph == "gauss5":
        return {"out": _shift_sat(_corr(img, A.B5, b), 8).v}
    if graph == "laplacian":
        return {"out": _corr(img, A.LAPLACE, b).map(_clamp(-32768, 32767)).v}
    if graph == "fchain":
        x = _shift_sat(_corr(img, A.B3, b), 4)
        x = _shift_sat(_corr(x, A.B5, b), 8)
        return {"out": _shift_sat(_corr(x, A.SHARPEN, b), 2).v}
    if graph == "unsharp":
        g = _shift_sat(_corr(img, A.B3, b), 4)
        return {"out": (img.v + 2 * (img.v - g.v)).clamp(-32768, 32767)}
    if graph == "sobel_x":
        return {"out": _corr(img, _SX, b).v}
    if graph in ("sobel", "edgfig2"):
        if graph == "edgfig2":
            img = _shift_sat(_corr(img, A.B3, b), 4)
        gy = _corr(img, _SX.T, b).v
        gx = gy if graph == "edgfig2" else _corr(img, _SX, b).v
        return {"out": _mask(_isqrt_round(gx ** 2 + gy ** 2) > THRESHOLD)}
    # morphology
    def nine(t):
        return torch.stack([t(dx, dy) for dy in (-1, 0, 1) for dx in (-1, 0, 1)])
    small = _Grid(f.to(torch.int16))
    dil = _local(small, 1, b, lambda t: nine(t).amax(0))
    closed = _local(dil, 1, b, lambda t: nine(t).amin(0))
    med = _local(small, 1, b, lambda t: nine(t).sort(0)[0][4])
    diff = (closed.v.long() - img.v).abs()
    return {"out": med.v.long() & _mask(diff > 20)}


def _exact_statistics(f):
    y = f[:, 1::2].long()
    n, s1, s2 = y.numel(), int(y.sum()), int((y * y).sum())
    hist = torch.bincount(y.reshape(-1), minlength=256)
    cum = hist.cumsum(0)
    lo, hi = int(y.min()), int(y.max())
    cmin, left = int(cum[lo]), n - int(cum[lo])
    table = torch.arange(256, device=y.device)
    if left:
        table = (2 * 255 * (cum - cmin) + left) // (2 * left)  # halves up
        table = table.clamp(0, 255)
    flat = y.reshape(-1)
    at = {k: int((flat == v).nonzero()[0]) for k, v in (("min", lo), ("max", hi))}
    w = y.shape[1]
    return {"out": table[y],
            "moments": {"mean": s1 / n, "stddev": math.sqrt(n * s2 - s1 * s1) / n, "sum": s1,
                        "sum_squares": s2, "count": n},
            "extrema": {"min": lo, "max": hi, "min_count": int(hist[lo]),
                        "max_count": int(hist[hi]), "min_x": at["min"] % w, "min_y": at["min"] // w,
                        "max_x": at["max"] % w, "max_y": at["max"] // w},
            "histogram": hist}


def exact(case, seed):
    sizes, graphs = _sizes(case), _graphs(case)
    got = [_exact_frame(g, case, f) for g, f in zip(graphs, _inputs(case, seed))]
    out = {}
    for name in sorted({o for g in graphs for o in _outputs(g, case)}):
        have = [i for i, g in enumerate(graphs) if name in _outputs(g, case)]
        fmt = _outputs(graphs[have[0]], case)[name]
        to = torch.float64 if fmt == H.HVX_DF_F32 else _TORCH[fmt]
        vals = [got[i][name].to(to) for i in have]
        if len({sizes[i] for i in have}) == 1:
            out[name] = torch.stack(vals)
            continue
        per = 16 // H.BYTES_PER_PIXEL[fmt]  # as the allocation holds them, padding 0
        out[name] = torch.cat([torch.nn.functional.pad(v, (0, -v.shape[1] % per)).reshape(-1)
                               for v in vals])
    for name in ("moments", "extrema", "histogram"):
        if name in got[0]:
            out[name] = got[0][name]
    return out
