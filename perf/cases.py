"""Work that users of the library have it do, as cases to be timed.

A case is a dict of plain values.  `prepare` makes what a program holds before
the call -- pixels on the device (or in pinned host memory), output buffers
and the stream, server or graph it keeps -- and `run` makes one pass through
the public entry points.  Every output is a histogram, a sum of histograms, a
pattern or a change result: whole numbers, exact.

The ranges (`draw` takes from all of them):
  plain     hist_plain of one image, 4 KiB .. 1 GiB
  adaptive  hist_adaptive with the pattern of the frame before, then the
            pattern of the next frame, 4 KiB .. 1 GiB, budgets 256 .. 8192
  push      one chunk pushed to a stream, 16 B .. 1 MiB
  stream    one push_many of 2 .. 1024 chunks of 1 KiB .. 16 MiB, at most
            1 GiB in all, every mode, budget, window, whole and ragged sizes
  host      chunks in pinned host memory, pushed through staging buffers
  batch     many images of uneven sizes in one call, or as a replayed graph
  serve     a burst of requests on many independent streams
"""
import ctypes
import math
import random

import numpy as np
import torch

import paper_1011_0235_gb300 as hl
from paper_1011_0235_gb300 import _abi

KiB, MiB = 1 << 10, 1 << 20
GEN_STEP = 32 * MiB  # pixels generated at a time (the generator's temporaries are four bytes a pixel)
MODES = {"auto": hl.MODE_AUTO, "plain": hl.MODE_PLAIN, "adaptive": hl.MODE_ADAPTIVE}


def listed():
    return [
        # the smallest call of a monitoring loop: one jumbo-frame packet, pushed
        # to a stream as it arrives
        {"name": "push_packet", "kind": "push", "n": 9001, "law": "normal", "mode": "auto", "budget": 8192},
        # one 1024 x 1024 image of random pixels, the plain kernel
        {"name": "image_1mib", "kind": "plain", "n": 1 << 20, "off": 0, "law": "uniform"},
        # the paper's 8192 x 8192 slice of random pixels, the plain kernel
        {"name": "slice_8192_plain", "kind": "plain", "n": 1 << 26, "off": 0, "law": "uniform"},
        # frames of a camera with the paper's 960-slot table: count one frame
        # with the pattern of the one before, derive the next (an odd size at
        # an odd address, as a crop of a larger buffer)
        {"name": "frames_960", "kind": "adaptive", "n": 200_000_003, "off": 13, "law": "normal", "budget": 960},
        # small slices gathered into one call, ragged, kernel by the switch
        {"name": "stream_64k_chunks", "kind": "stream", "chunk": 64 * KiB, "chunks": 1024, "ragged": True,
         "law": "normal", "mode": "auto", "budget": 8192, "window": 1, "overlap": False, "layout": 3},
        # the accumulated and the moving-window histogram of a stream compared
        # for a change, window of 32 chunks
        {"name": "stream_window32", "kind": "stream", "chunk": 1 * MiB, "chunks": 128, "ragged": False,
         "law": "phases", "mode": "auto", "budget": 8192, "window": 32, "overlap": False, "layout": 1},
        # the X-ray-like stream, 1 GiB in 16 MiB chunks, resident
        {"name": "stream_xray_1gib", "kind": "stream", "chunk": 16 * MiB, "chunks": 64, "ragged": False,
         "law": "normal", "mode": "adaptive", "budget": 8192, "window": 1, "overlap": True, "layout": 1},
        # the stream that turns degenerate and back every 8 chunks, kernel by
        # the switch, running totals
        {"name": "stream_degenerate_1gib", "kind": "stream", "chunk": 16 * MiB, "chunks": 64, "ragged": False,
         "law": "phases", "mode": "auto", "budget": 8192, "window": 1, "overlap": False, "layout": 1},
        # an acquisition's chunks in pinned host memory, copies overlapped
        {"name": "host_fed", "kind": "host", "chunk": 16 * MiB, "chunks": 16, "depth": 2, "law": "normal",
         "mode": "auto", "budget": 8192},
        # thumbnails and tiles: many small images in one call
        {"name": "batch_thumbnails", "kind": "batch", "count": 2048, "lo": 16, "hi": 256, "graph": False,
         "regimes": False, "layout": 5},
        # 4096 images of 64 .. 4096 pixels a side, one replayed graph
        {"name": "batch_4096_images", "kind": "batch", "count": 4096, "lo": 64, "hi": 4096, "graph": True,
         "regimes": False, "layout": 4},
        # a burst of requests of 4 KiB .. 64 MiB on 256 streams
        {"name": "serve_burst", "kind": "serve", "requests": 600, "streams": 256, "lo": 4 * KiB, "hi": 64 * MiB,
         "mode": "auto", "layout": 7},
    ]


def _log(rng, lo, hi):
    """A whole number, log-uniform in [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["plain", "plain", "adaptive", "push", "stream", "stream", "stream", "stream", "host", "batch",
                       "batch", "serve"])
    law = rng.choice(["uniform", "normal", "normal", "mixture", "degenerate"])
    mode = rng.choice(["auto", "auto", "adaptive", "plain"])
    budget = rng.choice([8192, 8192, 256, 960, 2048, 4096])
    if kind == "plain":
        return {"kind": kind, "n": _log(rng, 4 * KiB, 1 << 30), "off": rng.choice([0, rng.randrange(128)]), "law": law}
    if kind == "adaptive":
        return {"kind": kind, "n": _log(rng, 4 * KiB, 1 << 30), "off": rng.choice([0, rng.randrange(128)]), "law": law,
                "budget": budget}
    if kind == "push":
        return {"kind": kind, "n": _log(rng, 16, MiB), "law": law, "mode": mode, "budget": budget}
    if kind == "stream":
        chunk = _log(rng, KiB, 16 * MiB)
        chunks = _log(rng, 2, min(1024, (1 << 30) // chunk))
        return {"kind": kind, "chunk": chunk, "chunks": chunks, "ragged": rng.random() < 0.5,
                "law": rng.choice([law, law, "phases"]), "mode": mode, "budget": budget,
                "window": rng.choice([1, 1, 1, 2 + rng.randrange(255)]), "overlap": rng.random() < 0.3,
                "layout": rng.randrange(1 << 30)}
    if kind == "host":
        chunk = _log(rng, 64 * KiB, 16 * MiB)
        return {"kind": kind, "chunk": chunk, "chunks": _log(rng, 2, min(64, 256 * MiB // chunk)),
                "depth": rng.choice([2, 3, 4]), "law": law, "mode": mode, "budget": budget}
    if kind == "batch":
        lo = _log(rng, 8, 512)
        hi = _log(rng, lo, 4096)
        return {"kind": kind, "count": _log(rng, 1, 4096), "lo": lo, "hi": hi, "graph": rng.random() < 0.5,
                "regimes": rng.random() < 0.3, "layout": rng.randrange(1 << 30)}
    lo = _log(rng, KiB, MiB)
    return {"kind": kind, "requests": _log(rng, 16, 600), "streams": rng.choice([16, 64, 256]), "lo": lo,
            "hi": _log(rng, lo, 64 * MiB), "mode": mode, "layout": rng.randrange(1 << 30)}


# ---------------------------------------------------------------- inputs --

class _Laws:
    """Pixels of a law, on the device, from one generator."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)
        self.r = random.Random(seed)

    def params(self, law):
        """The law's parameters: an image's mean and spread are its own."""
        if law == "image":
            law = self.r.choice(["uniform", "normals", "mixture"])
        if law == "serve":
            law = "degenerate" if self.r.random() < 0.2 else self.r.choice(["uniform", "normals", "mixture"])
        if law == "normals":
            return ("normal", self.r.uniform(40, 215), self.r.uniform(4, 40))
        if law == "normal":
            return ("normal", 128.0, 8.0)
        if law == "mixture":
            return ("mixture", self.r.uniform(0.2, 0.8), self.r.uniform(40, 215), self.r.uniform(4, 40),
                    self.r.uniform(40, 215), self.r.uniform(4, 40))
        return (law,)

    def _normal(self, n, mu, sigma):
        return torch.randn(n, generator=self.g, device="cuda").mul_(sigma).add_(mu).round_().clamp_(0, 255).to(torch.uint8)

    def _uniform(self, n):
        return torch.randint(0, 256, (n,), dtype=torch.uint8, generator=self.g, device="cuda")

    def fill(self, x, p):
        for at in range(0, x.numel(), GEN_STEP):
            y = x[at:at + GEN_STEP]
            n = y.numel()
            if p[0] == "normal":
                y.copy_(self._normal(n, p[1], p[2]))
            elif p[0] == "mixture":
                first = torch.rand(n, generator=self.g, device="cuda") < p[1]
                y.copy_(torch.where(first, self._normal(n, p[2], p[3]), self._normal(n, p[4], p[5])))
            elif p[0] == "degenerate":  # 95 % of the pixels equal 90, the others uniform
                hot = torch.rand(n, generator=self.g, device="cuda") < 0.95
                y.copy_(self._uniform(n).masked_fill_(hot, 90))
            else:
                y.copy_(self._uniform(n))


def _sizes(case):
    """Sizes of a case's pieces and their byte offsets in one buffer."""
    kind = case["kind"]
    r = random.Random(case.get("layout", 0))
    if kind in ("plain", "adaptive"):
        return [case["n"]], [case["off"]]
    if kind == "push":
        return [case["n"]], [0]
    if kind == "host":
        return [case["chunk"]] * case["chunks"], [case["chunk"] * c for c in range(case["chunks"])]
    if kind == "stream":
        if not case["ragged"]:
            return [case["chunk"]] * case["chunks"], [case["chunk"] * c for c in range(case["chunks"])]
        sizes = [r.randint((case["chunk"] + 1) // 2, case["chunk"]) for _ in range(case["chunks"])]
    elif kind == "batch":
        sizes, offs, at = [], [], 0
        for _ in range(case["count"]):
            side = int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            sizes.append(side * int(round(side * r.uniform(1.0, 4.0 / 3.0))))
            offs.append(at)
            at = (at + sizes[-1] + 255) // 256 * 256
        return sizes, offs
    else:  # serve: each request lies in its stream's region, at any byte
        region = case["hi"]
        sizes, offs = [], []
        for s in _request_streams(case):
            n = int(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]))))
            sizes.append(min(n, region))
            offs.append(s * region + r.randint(0, region - sizes[-1]))
        return sizes, offs
    offs = [0]
    for n in sizes[:-1]:
        offs.append(offs[-1] + n)
    return sizes, offs


def _request_streams(case):
    r = random.Random(case["layout"] + 1)
    return [r.randrange(case["streams"]) for _ in range(case["requests"])]


def _pixels(case, seed):
    """The case's pixels (one device buffer), its pieces' sizes and offsets."""
    laws = _Laws(seed)
    sizes, offs = _sizes(case)
    if case["kind"] == "serve":
        x = torch.empty(case["streams"] * case["hi"], dtype=torch.uint8, device="cuda")
        for s in range(case["streams"]):
            laws.fill(x[s * case["hi"]:(s + 1) * case["hi"]], laws.params("serve"))
        return x, sizes, offs
    x = torch.empty(max(o + n for o, n in zip(offs, sizes)), dtype=torch.uint8, device="cuda")
    if case["kind"] == "batch":
        x.zero_()
        for n, o in zip(sizes, offs):
            laws.fill(x[o:o + n], laws.params("image"))
    elif case.get("law") == "phases":  # degenerate and uniform, 8 chunks each in turn
        for c, (n, o) in enumerate(zip(sizes, offs)):
            laws.fill(x[o:o + n], laws.params("degenerate" if (c // 8) % 2 == 0 else "uniform"))
    else:
        laws.fill(x, laws.params(case["law"]))
    return x, sizes, offs


# ----------------------------------------------------------------- state --

class _Graph:
    """A batch's graph, destroyed with it."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        hl.lib().hist_batch_graph_destroy(self.handle)


def prepare(case, seed):
    kind = case["kind"]
    x, sizes, offs = _pixels(case, seed)
    st = {"case": case, "x": x}
    k = len(sizes)
    if kind in ("plain", "adaptive"):
        st["img"] = x[offs[0]:offs[0] + sizes[0]]
        st["out"] = hl.empty_hist()
        if kind == "adaptive":  # the pattern of the frame before, another one of the same law
            before = torch.empty(MiB, dtype=torch.uint8, device="cuda")
            laws = _Laws(seed + (1 << 20))
            laws.fill(before, laws.params(case["law"]))
            st["pattern"] = hl.binning_pattern(hl.hist_plain(before), case["budget"])
            st["next"] = hl.empty_pattern()
        return st
    if kind == "push":
        st["stream"] = hl.Stream(budget=case["budget"], mode=MODES[case["mode"]])
        st["out"] = hl.empty_hist()
        return st
    st["outs"] = torch.empty((k, 256), dtype=torch.int32, device="cuda")
    out_ptrs = [st["outs"].data_ptr() + 1024 * i for i in range(k)]
    if kind == "stream":
        st["stream"] = hl.Stream(budget=case["budget"], mode=MODES[case["mode"]], window=case["window"],
                                 overlap=case["overlap"])
        st["ptrs"] = np.array([x.data_ptr() + o for o in offs], dtype=np.uint64)
        st["sizes"] = np.array(sizes, dtype=np.uint64)
        st["out_ptrs"] = np.array(out_ptrs, dtype=np.uint64)
        st["totals"] = torch.empty(256, dtype=torch.int64, device="cuda")
        st["window"] = torch.empty(256, dtype=torch.int64, device="cuda")
    elif kind == "host":
        st["host"] = torch.empty(x.numel(), dtype=torch.uint8, pin_memory=True)
        st["host"].copy_(x)
        del st["x"]
        st["stream"] = hl.Stream(budget=case["budget"], mode=MODES[case["mode"]])
        st["stream"].attach_staging(case["chunk"], case["depth"])
        st["calls"] = [(st["host"].data_ptr() + o, n, p) for o, n, p in zip(offs, sizes, out_ptrs)]
        st["totals"] = torch.empty(256, dtype=torch.int64, device="cuda")
    elif kind == "batch":
        st["ptrs"] = torch.tensor([x.data_ptr() + o for o in offs], dtype=torch.int64).cuda()
        st["sizes"] = torch.tensor(sizes, dtype=torch.int64).cuda()
        st["regime"] = torch.empty(k, dtype=torch.uint8, device="cuda")
        if case["graph"]:
            g = ctypes.c_void_p()
            a = (st["ptrs"].data_ptr(), st["sizes"].data_ptr(), k, st["outs"].data_ptr())
            torch.cuda.synchronize()
            if case["regimes"]:
                rc = hl.lib().hist_batch_regimes_capture(*a, st["regime"].data_ptr(), None, ctypes.byref(g))
            else:
                rc = hl.lib().hist_batch_capture(*a, None, ctypes.byref(g))
            _abi.check("hist_batch_capture", rc)
            st["graph"] = _Graph(g)
    else:
        st["server"] = hl.Server(streams=case["streams"], mode=MODES[case["mode"]])
        reqs = (_abi.Request * k)()
        for i, s in enumerate(_request_streams(case)):
            reqs[i].arrival_ns, reqs[i].stream, reqs[i].tag = 0, s, i
            reqs[i].d_in, reqs[i].n, reqs[i].d_out = x.data_ptr() + offs[i], sizes[i], out_ptrs[i]
        st["reqs"] = reqs
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "plain":
        return hl.hist_plain(st["img"], st["out"])
    if kind == "adaptive":
        h = hl.hist_adaptive(st["img"], st["pattern"], st["out"])
        return [h, hl.binning_pattern(h, case["budget"], st["next"])]
    if kind == "push":
        st["stream"].push(st["x"], st["out"])
        return st["out"]
    if kind == "stream":
        s = st["stream"]
        s.push_many(st["ptrs"], st["sizes"], st["out_ptrs"])
        got = [st["outs"], s.totals(st["totals"])]
        if case["window"] > 1:
            got += [s.window(st["window"]), s.change()]
        return got
    if kind == "host":
        s = st["stream"]
        for ptr, n, out in st["calls"]:
            s.push_host(ptr, n, out)
        return [st["outs"], s.totals(st["totals"])]
    if kind == "batch":
        if case["graph"]:
            rc = hl.lib().hist_batch_graph_launch(st["graph"].handle, torch.cuda.current_stream().cuda_stream)
        else:
            a = (st["ptrs"].data_ptr(), st["sizes"].data_ptr(), case["count"], st["outs"].data_ptr())
            s = torch.cuda.current_stream().cuda_stream
            if case["regimes"]:
                rc = hl.lib().hist_batch_regimes(*a, st["regime"].data_ptr(), None, s)
            else:
                rc = hl.lib().hist_batch(*a, None, s)
        _abi.check("hist_batch", rc)
        return [st["outs"], st["regime"]] if case["regimes"] else st["outs"]
    st["server"].replay(st["reqs"], timeout_ms=60000)
    return st["outs"]


def work(case):
    sizes, _ = _sizes(case)
    out = 1024 * len(sizes)
    if case["kind"] in ("stream", "host"):
        out += 2048
    return {"bytes": sum(sizes) + out, "flops": 0}


def exact(case, seed):
    """The histograms by torch.bincount, in int64; the patterns, the regimes
    and the change result have no such value."""
    x, sizes, offs = _pixels(case, seed)
    rows = []
    for n, o in zip(sizes, offs):
        h = torch.zeros(256, dtype=torch.int64, device="cuda")
        for at in range(0, n, GEN_STEP):
            h += torch.bincount(x[o + at:o + min(n, at + GEN_STEP)], minlength=256)
        rows.append(h)
    outs = torch.stack(rows)
    kind = case["kind"]
    if kind in ("plain", "push"):
        return outs[0]
    if kind == "adaptive":
        return [outs[0], None]
    if kind == "host":
        return [outs, outs.sum(0)]
    if kind == "stream":
        got = [outs, outs.sum(0)]
        return got + [outs[-case["window"]:].sum(0), None] if case["window"] > 1 else got
    if kind == "batch" and case["regimes"]:
        return [outs, None]
    return outs
