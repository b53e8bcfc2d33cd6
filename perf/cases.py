"""The workloads that the library's speed is judged by, from the smallest call to the largest.

A case is one pass through the public entry points of ``paper_1603_09180_gb300.thin`` on seeded
synthetic images: value noise in three octaves with dark line segments, the recipe of the package's
``synth`` module made on the GPU so that many inputs can be drawn quickly.  Thinning works in place, so
a pass first copies the pristine images over the working ones, as a program that keeps its inputs does.

kind   run     thin.run, the default call (waits for its stats)
       batch   BatchPlan.run: job records marshalled once, one device-driven thin_batch call a pass
       plan    GraphPlan.run: the batch prepared once, one graph launch a pass; images of many sizes
       serve   Server: host images submitted at once, collected as they finish

All outputs are whole numbers: thinned images, lowering counts and last changing phases (16-bit images
as int16: the same bits in a type that every tensor operation takes).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1603_09180_gb300 import thin

SIGMAS = (2.0, 8.0, 32.0)
WEIGHTS = (0.2, 0.3, 0.5)
N_LINES = 20
VMAX = {"u8": 255, "u16": 4095}


def _case(name, kind, w, h, n=1, dtype="u8", lams="0", op="thinning", adj="8,4", rule="max", sizes=0):
    c = dict(kind=kind, w=w, h=h, n=n, dtype=dtype, lams=lams, op=op, adj=adj, rule=rule, sizes=sizes)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a thumbnail or region of interest in an interactive tool: one call's latency
        _case("run_64", "run", 64, 64, lams="10"),
        # the paper's image size, one image, homotopic thinning without filtering
        _case("run_512", "run", 512, 512, lams="0"),
        # 64 sections of a series, each at three contrasts (the benchmark's default step)
        _case("batch192_u8", "batch", 512, 512, n=64, lams="0,5,20"),
        # the same series under the paper's own operator
        _case("batch192_skeleton", "batch", 512, 512, n=64, lams="0,5,20", op="skeleton"),
        # the same series at 12 bits, the same contrasts in grey levels
        _case("batch192_u16", "batch", 512, 512, n=64, dtype="u16", lams="0,80,320"),
        # bright objects taken as 4-connected: the other adjacency pair
        _case("batch64_adj48", "batch", 512, 512, n=64, lams="5", adj="4,8"),
        # a scanned page or micrograph, without and with filtering
        _case("run_4096_l0", "run", 4096, 4096, lams="0"),
        _case("run_4096_l30", "run", 4096, 4096, lams="30"),
        # a 12-bit slide, the largest image of the benchmark
        _case("run_8192_u16_l0", "run", 8192, 8192, dtype="u16", lams="0"),
        _case("run_8192_u16_l30", "run", 8192, 8192, dtype="u16", lams="30"),
        # a data set of images of every size, odd widths among them, processed again and again
        _case("plan_uneven1024", "plan", 2048, 2048, n=1024, lams="0,10,25", sizes=64),
        # a service: requests of all sizes and both types, host images in and out
        _case("serve_48", "serve", 4096, 4096, n=48, dtype="mix", lams="0,10", sizes=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "batch", "batch", "batch", "plan", "plan", "serve"])
    if kind == "serve":
        return _case(None, kind, _log_int(rng, 256, 3000), _log_int(rng, 256, 3000), n=rng.randint(8, 48), dtype="mix",
                     lams="0,10", sizes=rng.choice([64, 128]))
    dtype = rng.choice(["u8", "u8", "u16"])
    lams = {"u8": ["0", "5", "10", "20", "30"], "u16": ["0", "30", "80", "160"]}[dtype]
    if kind == "plan":
        most = 512 if dtype == "u8" else 256
        return _case(None, kind, _log_int(rng, 256, 2048), _log_int(rng, 256, 2048), n=_log_int(rng, 16, most), dtype=dtype,
                     lams=",".join(sorted(rng.sample(lams, 2), key=int)), sizes=64)
    # the options beside the common mode: the skeleton, the other adjacency pair, the other reading of F^-
    op, adj, rule = rng.choice([("thinning", "8,4", "max")] * 5 + [("skeleton", "8,4", "max"), ("thinning", "4,8", "max"),
                                                                   ("thinning", "8,4", "min")])
    common = op == "thinning" and adj == "8,4" and rule == "max"
    if kind == "run":
        hi = 4096 if common else 1024
        return _case(None, kind, _log_int(rng, 64, hi), _log_int(rng, 64, hi), dtype=dtype, lams=rng.choice(lams), op=op,
                     adj=adj, rule=rule)
    w, h = _log_int(rng, 64, 1024), _log_int(rng, 64, 1024)
    picked = sorted(rng.sample(lams, rng.randint(1, 3)), key=int)
    jobs = (96 if common else 32) * 512 * 512 / (w * h * len(picked))
    return _case(None, kind, w, h, n=max(1, min(64, int(rng.uniform(0.1, 1.0) * jobs))), dtype=dtype, lams=",".join(picked),
                 op=op, adj=adj, rule=rule)


def _sizes(case):
    """(h, w) of every input image: one size, or sides log-uniform up to the case's."""
    if not case["sizes"]:
        return [(case["h"], case["w"])] * case["n"]
    rng = np.random.Generator(np.random.PCG64(case["n"] * 7919 + case["w"] * 31 + case["h"]))
    a = math.log(case["sizes"])
    hs = np.rint(np.exp(rng.uniform(a, math.log(case["h"]), case["n"]))).astype(int)
    ws = np.rint(np.exp(rng.uniform(a, math.log(case["w"]), case["n"]))).astype(int)
    return [(int(h), int(w)) for h, w in zip(hs, ws)]


def _dtypes(case):
    if case["dtype"] != "mix":
        return [case["dtype"]] * case["n"]
    return ["u16" if k % 2 else "u8" for k in range(case["n"])]


def _lams(case):
    return [int(v) for v in case["lams"].split(",")]


def _image(h, w, dtype, gen, rng):
    """One image on the GPU: three blurred octaves of noise, dark lines, rescaled to 0..vmax."""
    dev = torch.device("cuda")
    hh, ww = (h + 255) // 256 * 256, (w + 255) // 256 * 256  # few distinct FFT sizes
    fy = torch.fft.fftfreq(hh, device=dev)[:, None]
    fx = torch.fft.rfftfreq(ww, device=dev)[None, :]
    v = torch.zeros((h, w), device=dev)
    for sigma, weight in zip(SIGMAS, WEIGHTS):
        f = torch.fft.rfft2(torch.rand((hh, ww), device=dev, generator=gen))
        f *= torch.exp((fy * fy + fx * fx) * (-2.0 * math.pi ** 2 * sigma ** 2))
        o = torch.fft.irfft2(f, s=(hh, ww))[:h, :w]
        lo, hi = torch.aminmax(o)
        v += weight * ((o - lo) / (hi - lo).clamp_min(1e-12))
    ends = rng.uniform(0.0, 1.0, (N_LINES, 4)) * np.array([w, h, w, h])
    half = rng.integers(2, 5, N_LINES) / 2.0
    table = torch.from_numpy(np.concatenate([ends, half[:, None]], 1).astype(np.float32)).to(dev)
    y = torch.arange(h, device=dev, dtype=torch.float32)[None, :, None]
    x = torch.arange(w, device=dev, dtype=torch.float32)[None, None, :]
    chunk = max(1, min(N_LINES, (1 << 26) // (h * w)))
    for i in range(0, N_LINES, chunk):
        x0, y0, x1, y1, r = (table[i:i + chunk, k][:, None, None] for k in range(5))
        dx, dy = x1 - x0, y1 - y0
        t = (((x - x0) * dx + (y - y0) * dy) / (dx * dx + dy * dy).clamp_min(1e-6)).clamp_(0.0, 1.0)
        d2 = (x - x0 - t * dx).square_() + (y - y0 - t * dy).square_()
        v -= (40.0 / 255.0) * (d2 <= r * r).sum(0)
    lo, hi = torch.aminmax(v)
    v = ((v - lo) * (VMAX[dtype] / (hi - lo).clamp_min(1e-12))).round_().to(torch.int32)
    return v.to(torch.uint8 if dtype == "u8" else torch.uint16)


def _options(case):
    return dict(op=case["op"], adj=case["adj"], rule=case["rule"])


class _Service:
    """A server that ends with the state that holds it."""

    def __init__(self, n):
        self.server = thin.Server(1 << 30, max_slots=256, queue_cap=max(64, n))

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    images = [_image(h, w, d, gen, rng) for (h, w), d in zip(_sizes(case), _dtypes(case))]
    kind, lams = case["kind"], _lams(case)
    if kind == "run":
        return {"kind": kind, "lam": lams[0], "src": images[0], "img": torch.empty_like(images[0]), "opt": _options(case)}
    if kind == "serve":
        order = [lams[k // 2 % len(lams)] for k in range(case["n"])]
        return {"kind": kind, "images": [t.cpu().numpy() for t in images], "lams": order, "service": _Service(case["n"])}
    if kind == "batch":
        src = torch.stack([t.view(torch.int16) if t.dtype == torch.uint16 else t for t in images]).repeat(len(lams), 1, 1)
        out = torch.empty_like(src)
        views = list(out.view(images[0].dtype))
        plan = thin.BatchPlan(views, [lam for lam in lams for _ in images], **_options(case))
        return {"kind": kind, "src": src, "out": out, "views": views, "plan": plan}
    # plan: the images in one buffer, each at a 512-byte boundary, rows packed
    es = images[0].element_size()
    off, at = [], 0
    for t in images:
        off.append(at)
        at += (t.numel() * es + 511) // 512 * 512
    src = torch.zeros(at, dtype=torch.uint8, device="cuda")
    for o, t in zip(off, images):
        src[o:o + t.numel() * es] = t.view(-1).view(torch.uint8)
    out = src.clone()
    views = [out[o:o + t.numel() * es].view(t.dtype).view(t.shape) for o, t in zip(off, images)]
    pick = np.random.Generator(np.random.PCG64(case["n"])).integers(0, len(lams), len(images))
    order = [lams[k] for k in pick]
    return {"kind": kind, "src": src, "out": out, "views": views, "plan": thin.GraphPlan(views, order, **_options(case))}


def run(state):
    kind = state["kind"]
    if kind == "run":
        img = state["img"]
        img.copy_(state["src"])
        st = thin.run(img, state["lam"], **state["opt"])
        return {"image": img.view(torch.int16) if img.dtype == torch.uint16 else img, "lowered": st["lowered"],
                "last_change_phase": st["last_change_phase"]}
    if kind == "serve":
        server, place, got = state["service"].server, {}, [None] * len(state["images"])
        for k, (img, lam) in enumerate(zip(state["images"], state["lams"])):
            place[server.submit(img, lam)] = k
        while place:
            ticket = server.wait_any(1000)
            if ticket is not None:
                done, img, _, _ = server.poll(ticket)
                if done:
                    got[place.pop(ticket)] = img.view(np.int16) if img.dtype == np.uint16 else img
        return got
    state["out"].copy_(state["src"])
    state["plan"].run()
    return state["out"]


def work(case):
    """Every pixel read and written once; every pixel compared with its eight neighbours and decided at least once."""
    es = [2 if d == "u16" else 1 for d in _dtypes(case)]
    jobs = len(_lams(case)) if case["kind"] == "batch" else 1
    sizes = _sizes(case)
    return {"bytes": float(jobs * sum(2 * h * w * e for (h, w), e in zip(sizes, es))),
            "flops": float(jobs * sum(9 * h * w for h, w in sizes))}
