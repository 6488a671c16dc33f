"""Performance cases: the work a user of this library has it do, through its
public entry points, over the range of sizes, types, directions and options
the library serves.

Inputs are drawn on the GPU from a seed: a smooth gradient with sensor-like
noise for CDF 9/7 (divided by its scale for 16-bit storage) and 12-bit
integers for LeGall 5/3.  The inverse starts from the coefficients of such an
image, computed here in 64 bits and stored in the case's type.

Kinds of case:
  image   one transform of a device-resident image (or coefficients); with
          direction "both", the forward and the inverse of its result
  batch   many images of uneven sizes through one Batch
  serve   a burst of requests through the serving loop
  host    one forward transform from a pinned host buffer to another
"""
from __future__ import annotations

import math
import random

import torch

from paper_1705_08266_gb300 import dwt2d as D
from paper_1705_08266_gb300 import serve

DEV = "cuda"
TYPES = {"f32": torch.float32, "i32": torch.int32, "f16": torch.float16, "bf16": torch.bfloat16}
# CDF 9/7 lifting pairs (predict, update) and scaling constant
PAIRS = ((-1.586134342059924, -0.052980118572961), (0.882911075530934, 0.443506852043971))
SCALING = 1.230174104914001
PEAK = 263.5  # bound of the float images: values of 16-bit images are stored divided by it


def _image(name, h, w, levels, dtype="f32", direction="fwd", scheme="nonsep_reduced"):
    return {"name": name, "kind": "image", "h": h, "w": w, "levels": levels, "dtype": dtype,
            "direction": direction, "scheme": scheme}


def listed():
    return [
        # the smallest everyday call: one level of a 512 x 512 tile there and
        # back, separable lifting; launches and latency count
        _image("tile_512_l1_sep_both", 512, 512, 1, direction="both", scheme="separable"),
        # a video frame or photograph analysed at the usual depth
        _image("frame_1080p_l5_fwd", 1080, 1920, 5),
        # sizes that divide by nothing: odd rows and columns at every level
        _image("odd_777x3001_l2_fwd", 777, 3001, 2),
        # synthesis of an odd-sized scan kept in 16 bits
        _image("odd_4099x2051_l6_f16_inv", 4099, 2051, 6, "f16", "inv"),
        # the headline workload, both directions
        _image("large_8192_l5_fwd", 8192, 8192, 5),
        _image("large_8192_l5_inv", 8192, 8192, 5, direction="inv"),
        # lossless coding of large 12-bit scans, both directions
        _image("large_8192_l5_i32_fwd", 8192, 8192, 5, "i32"),
        _image("large_8192_l5_i32_inv", 8192, 8192, 5, "i32", "inv"),
        # the largest images, whose 16-bit storage halves the memory they take
        _image("huge_16384_l6_f16_fwd", 16384, 16384, 6, "f16"),
        # a dataset batch: 256 images of uneven sizes, three quarters CDF 9/7
        # and a quarter LeGall 5/3
        {"name": "batch_256_mixed_fwd", "kind": "batch", "images": 256, "lo": 65, "hi": 4096,
         "persistent": False, "sizes": 2017},
        # a burst of a serving client: sides log-uniform on 64..8192, both
        # directions, 16-bit CDF 9/7 and LeGall 5/3
        {"name": "serve_32_mixed", "kind": "serve", "requests": 32, "lo": 64, "hi": 8192, "sizes": 2026},
        # an image that lives in host memory and whose coefficients go back there
        {"name": "host_8192_l5_fwd", "kind": "host", "h": 8192, "w": 8192, "levels": 5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    r = rng.random()
    if r < 0.12:
        hi = _log_int(rng, 256, 4096)
        return {"kind": "batch", "images": _log_int(rng, 8, 256), "lo": 65, "hi": hi,
                "persistent": rng.random() < 0.5, "sizes": rng.randrange(1 << 30)}
    if r < 0.2:
        return {"kind": "serve", "requests": rng.randint(4, 32), "lo": 64, "hi": _log_int(rng, 512, 8192),
                "sizes": rng.randrange(1 << 30)}
    if r < 0.26:
        s = _log_int(rng, 512, 8192)
        return {"kind": "host", "h": s, "w": max(64, int(s / rng.uniform(1, 3))), "levels": rng.randint(1, 6)}
    long = _log_int(rng, 128, 16384)
    short = max(32, int(long / rng.uniform(1, 4)))
    h, w = (long, short) if rng.random() < 0.5 else (short, long)
    if rng.random() < 0.4:  # sizes as sensors and tilers have them, the others as they fall
        h, w = max(32, h // 32 * 32), max(32, w // 32 * 32)
    return {"kind": "image", "h": h, "w": w, "levels": rng.randint(1, 6),
            "dtype": rng.choice(("f32", "f32", "f32", "i32", "i32", "f16", "bf16")),
            "direction": rng.choice(("fwd", "fwd", "inv", "both")),
            "scheme": rng.choice(("nonsep_reduced", "nonsep_reduced", "nonsep_reduced", "separable", "nonsep"))}


# ---------------------------------------------------------------- shapes ----
def _jobs(case):
    """[(h, w, levels, dtype, inverse)] of a batch or serving case."""
    rng = random.Random(case["sizes"])
    out = []
    if case["kind"] == "batch":
        for _ in range(case["images"]):
            h, w = rng.randint(case["lo"], case["hi"]), rng.randint(case["lo"], case["hi"])
            out.append((h, w, rng.randint(1, 6), "f32" if rng.random() < 0.75 else "i32", False))
        return out
    for _ in range(case["requests"]):
        long = _log_int(rng, case["lo"], case["hi"])
        short = max(16, int(long / rng.uniform(1, 4)))
        h, w = (long, short) if rng.random() < 0.5 else (short, long)
        out.append((h, w, rng.randint(1, 6), "f16" if rng.random() < 0.5 else "i32", rng.random() < 0.3))
    return out


def _wavelet(dtype):
    return "legall53" if dtype == "i32" else "cdf97"


def work(case):
    """Each image read once and its coefficients written once (or the reverse);
    32 lifting operations per quadruple and level for CDF 9/7, 16 for 5/3."""
    if case["kind"] in ("image", "host"):
        dtype = case.get("dtype", "f32")
        jobs = [(case["h"], case["w"], case["levels"], dtype, False)] * (2 if case.get("direction") == "both" else 1)
    else:
        jobs = _jobs(case)
    total, flops = 0, 0
    for h, w, levels, dtype, _inv in jobs:
        total += 2 * h * w * TYPES[dtype].itemsize
        for _ in range(levels):
            flops += h * w * (4 if dtype == "i32" else 8)
            h, w = (h + 1) // 2, (w + 1) // 2
    return {"bytes": total, "flops": flops}


# ---------------------------------------------------------------- inputs ----
def _picture(gen, h, w, dtype):
    """An (h, w) image of the case's type."""
    if dtype == "i32":
        return torch.randint(0, 4096, (h, w), generator=gen, device=DEV, dtype=torch.int32)
    r = torch.arange(h, device=DEV, dtype=torch.float32)[:, None] * (0.5 / h)
    c = torch.arange(w, device=DEV, dtype=torch.float32)[None, :] * (0.75 / w)
    x = torch.rand((h, w), generator=gen, device=DEV).mul_(16.0).add_(119.5)
    x += torch.sin((r + c).mul_(2.0 * math.pi)).mul_(127.5)
    return x if dtype == "f32" else (x / PEAK).to(TYPES[dtype])


def _input(gen, h, w, levels, dtype, inverse):
    x = _picture(gen, h, w, dtype)
    if not inverse:
        return x
    c = _lift(_wide(x), levels, dtype == "i32")
    return c.to(TYPES[dtype])


def _pitched(x):
    t = D.empty_image(x.shape[0], x.shape[1], x.dtype, DEV)
    t.copy_(x)
    return t


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _flat(shapes, dtype):
    """One zeroed buffer for many outputs and a pitched view of it per shape,
    each starting on a 256-byte boundary."""
    offs, n = [], 0
    for h, w in shapes:
        offs.append(n)
        n += (h * D.pitch_elems(w, TYPES[dtype]) + 63) // 64 * 64
    return n, offs


def _views(buf, shapes, offs, dtype):
    out = []
    for (h, w), o in zip(shapes, offs):
        p = D.pitch_elems(w, TYPES[dtype])
        out.append(buf[o:o + h * p].view(h, p)[:, :w])
    return out


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "image":
        h, w, levels, dtype = case["h"], case["w"], case["levels"], case["dtype"]
        x = _pitched(_input(gen, h, w, levels, dtype, case["direction"] == "inv"))
        plan = D.Plan(h, w, levels, _wavelet(dtype), case["scheme"], TYPES[dtype])
        st = {"plan": plan, "x": x, "out": D.empty_image(h, w, TYPES[dtype], DEV), "ws": plan.workspace(DEV),
              "scale": PEAK if dtype in ("f16", "bf16") else 1.0, "direction": case["direction"]}
        if case["direction"] == "both":
            st["back"] = D.empty_image(h, w, TYPES[dtype], DEV)
        return {"kind": kind, **st}
    if kind == "host":
        h, w = case["h"], case["w"]
        plan = D.Plan(h, w, case["levels"])
        src = torch.empty((h, w), dtype=torch.float32, pin_memory=True)
        src.copy_(_picture(gen, h, w, "f32"))
        return {"kind": kind, "plan": plan, "src": src,
                "dst": torch.empty((h, w), dtype=torch.float32, pin_memory=True),
                "stage_in": D.empty_image(h, w, torch.float32, DEV),
                "stage_out": D.empty_image(h, w, torch.float32, DEV), "ws": plan.workspace(DEV)}
    jobs = _jobs(case)
    xs = [_pitched(_input(gen, h, w, lv, dt, inv)) for h, w, lv, dt, inv in jobs]
    if kind == "serve":
        reqs = [serve.Request(h, w, lv, _wavelet(dt), TYPES[dt], inv, data=x)
                for (h, w, lv, dt, inv), x in zip(jobs, xs)]
        # the inputs are resident before the first request arrives
        torch.cuda.current_stream().synchronize()
        return {"kind": kind, "server": serve.Server(budget_bytes=40 << 30), "requests": reqs}
    bufs, outs = {}, [None] * len(jobs)
    for dt in ("f32", "i32"):
        at = [i for i, j in enumerate(jobs) if j[3] == dt]
        shapes = [jobs[i][:2] for i in at]
        n, offs = _flat(shapes, dt)
        if n:
            bufs[dt] = torch.zeros(n, dtype=TYPES[dt], device=DEV)
            for i, v in zip(at, _views(bufs[dt], shapes, offs, dt)):
                outs[i] = v
    batch = D.Batch([(x, o, lv, _wavelet(dt), int(inv)) for (h, w, lv, dt, inv), x, o in zip(jobs, xs, outs)],
                    tuning={"persistent": 1} if case["persistent"] else None)
    ws = batch.workspace(DEV)
    batch.upload(ws)
    return {"kind": kind, "batch": batch, "ws": ws, "bufs": bufs, "xs": xs}


# ------------------------------------------------------------------- run ----
def run(state):
    kind = state["kind"]
    if kind == "image":
        plan, scale, d = state["plan"], state["scale"], state["direction"]
        if d == "inv":
            return plan.inverse(state["x"], state["out"], state["ws"], scale)
        plan.forward(state["x"], state["out"], state["ws"], scale)
        if d == "fwd":
            return state["out"]
        plan.inverse(state["out"], state["back"], state["ws"], scale)
        return [state["out"], state["back"]]
    if kind == "host":
        return state["plan"].forward_host(state["src"], state["dst"], state["stage_in"], state["stage_out"],
                                          state["ws"])
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(r) for r in state["requests"]]
        outs = [server.result(t) for t in tickets]
        for t in tickets:
            server.release(t)
        return outs
    state["batch"].launch(state["ws"])
    return state["bufs"]


# ----------------------------------------------------------------- exact ----
def _wide(x):
    return x.to(torch.int64) if x.dtype == torch.int32 else x.to(torch.float64)


def _next_even(e, no):
    """Right neighbour e[i + 1] of every odd sample, mirrored past the end."""
    return e[1:no + 1] if e.shape[0] > no else torch.cat([e[1:], e[-1:]])


def _odd_pair(o, ne):
    """(o[i - 1], o[i]) around every even sample, mirrored at both ends."""
    own = o if o.shape[0] == ne else torch.cat([o, o[-1:]])
    return torch.cat([o[:1], o[:ne - 1]]), own


def _split(x):
    return x[0::2].clone(), x[1::2].clone()


def _analyse(x, integer):
    """One level along the first axis: (low, high)."""
    e, o = _split(x)
    if x.shape[0] == 1:
        return e, o
    ne, no = e.shape[0], o.shape[0]
    if integer:
        o -= (e[:no] + _next_even(e, no)) >> 1
        a, b = _odd_pair(o, ne)
        e += (a + b + 2) >> 2
        return e, o
    for p, u in PAIRS:
        o += (e[:no] + _next_even(e, no)).mul_(p)
        a, b = _odd_pair(o, ne)
        e += (a + b).mul_(u)
    return e.div_(SCALING), o.mul_(SCALING)


def _synthesise(e, o, integer):
    ne, no = e.shape[0], o.shape[0]
    e, o = e.clone(), o.clone()
    if no and integer:
        a, b = _odd_pair(o, ne)
        e -= (a + b + 2) >> 2
        o += (e[:no] + _next_even(e, no)) >> 1
    elif no:
        e.mul_(SCALING)
        o.div_(SCALING)
        for p, u in reversed(PAIRS):
            a, b = _odd_pair(o, ne)
            e -= (a + b).mul_(u)
            o -= (e[:no] + _next_even(e, no)).mul_(p)
    x = torch.empty((ne + no,) + tuple(e.shape[1:]), dtype=e.dtype, device=e.device)
    x[0::2], x[1::2] = e, o
    return x


def _lift(x, levels, integer):
    """Mallat coefficients of x in 64 bits.  The reversible 5/3 is defined in
    the order predict along rows, predict along columns, update along rows,
    update along columns; the linear steps commute."""
    out = x.clone()
    h, w = x.shape
    for _ in range(levels):
        a = out[:h, :w]
        ne, we = (h + 1) // 2, (w + 1) // 2
        bands = _level53(a) if integer else _level97(a)
        out[:ne, :we], out[:ne, we:w], out[ne:h, :we], out[ne:h, we:w] = bands
        h, w = ne, we
    return out


def _level97(a):
    lo, hi = _analyse(a.t(), False)
    (ll, lh), (hl, hh) = _analyse(lo.t(), False), _analyse(hi.t(), False)
    return ll, hl, lh, hh


def _level53(a):
    h, w = a.shape
    q = [[a[i::2, j::2].clone() for j in (0, 1)] for i in (0, 1)]
    nw, nh = w // 2, h // 2
    if w > 1:  # predict along rows
        for row in q:
            e = row[0].t()
            row[1] -= ((e[:nw] + _next_even(e, nw)) >> 1).t()
    if h > 1:  # predict along columns
        for j in (0, 1):
            e = q[0][j]
            q[1][j] -= (e[:nh] + _next_even(e, nh)) >> 1
    if w > 1:  # update along rows
        for row in q:
            x, y = _odd_pair(row[1].t(), row[0].shape[1])
            row[0] += ((x + y + 2) >> 2).t()
    if h > 1:  # update along columns
        for j in (0, 1):
            x, y = _odd_pair(q[1][j], q[0][j].shape[0])
            q[0][j] += (x + y + 2) >> 2
    return q[0][0], q[0][1], q[1][0], q[1][1]


def _unlift(c, levels, integer):
    out = c.clone()
    sizes, h, w = [], c.shape[0], c.shape[1]
    for _ in range(levels):
        sizes.append((h, w))
        h, w = (h + 1) // 2, (w + 1) // 2
    for h, w in reversed(sizes):
        ne, we = (h + 1) // 2, (w + 1) // 2
        ll, hl, lh, hh = out[:ne, :we], out[:ne, we:w], out[ne:h, :we], out[ne:h, we:w]
        out[:h, :w] = _unlevel53(ll, hl, lh, hh) if integer else _unlevel97(ll, hl, lh, hh)
    return out


def _unlevel97(ll, hl, lh, hh):
    lo, hi = _synthesise(ll, lh, False), _synthesise(hl, hh, False)
    return _synthesise(lo.t(), hi.t(), False).t()


def _unlevel53(ll, hl, lh, hh):
    q = [[ll.clone(), hl.clone()], [lh.clone(), hh.clone()]]
    h, w = ll.shape[0] + lh.shape[0], ll.shape[1] + hl.shape[1]
    nw, nh = w // 2, h // 2
    if h > 1:
        for j in (0, 1):
            x, y = _odd_pair(q[1][j], q[0][j].shape[0])
            q[0][j] -= (x + y + 2) >> 2
    if w > 1:
        for row in q:
            x, y = _odd_pair(row[1].t(), row[0].shape[1])
            row[0] -= ((x + y + 2) >> 2).t()
    if h > 1:
        for j in (0, 1):
            e = q[0][j]
            q[1][j] += (e[:nh] + _next_even(e, nh)) >> 1
    if w > 1:
        for row in q:
            e = row[0].t()
            row[1] += ((e[:nw] + _next_even(e, nw)) >> 1).t()
    x = torch.empty((h, w), dtype=ll.dtype, device=ll.device)
    for i in (0, 1):
        for j in (0, 1):
            x[i::2, j::2] = q[i][j]
    return x


def exact(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    if kind == "host":
        return _lift(_wide(_picture(gen, case["h"], case["w"], "f32")), case["levels"], False).cpu()
    if kind == "image":
        h, w, levels, dtype, d = case["h"], case["w"], case["levels"], case["dtype"], case["direction"]
        integer = dtype == "i32"
        x = _wide(_input(gen, h, w, levels, dtype, d == "inv"))
        if d == "inv":
            return _unlift(x, levels, integer)
        c = _lift(x, levels, integer)
        # the inverse's input is the forward's result as it is stored, which
        # only for the integers is known without running it
        return c if d == "fwd" else [c, x if integer else None]
    jobs = _jobs(case)
    xs = [_wide(_input(gen, h, w, lv, dt, inv)) for h, w, lv, dt, inv in jobs]
    outs = [(_unlift if inv else _lift)(x, lv, dt == "i32") for x, (h, w, lv, dt, inv) in zip(xs, jobs)]
    if kind == "serve":
        return outs
    bufs = {}
    for dt in ("f32", "i32"):
        at = [i for i, j in enumerate(jobs) if j[3] == dt]
        shapes = [jobs[i][:2] for i in at]
        n, offs = _flat(shapes, dt)
        if n:
            bufs[dt] = torch.zeros(n, dtype=torch.int64 if dt == "i32" else torch.float64, device=DEV)
            for i, v in zip(at, _views(bufs[dt], shapes, offs, dt)):
                v.copy_(outs[i])
    return bufs
