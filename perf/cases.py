"""The work that programs have this library do, as cases that can be timed.

Every case goes through the public calls of paper_1709_07781_gb300 with the
library's default tile shapes. Inputs are uint32 data held as int32 tensors
(bit copies), made on the GPU from a seed. All outputs are whole numbers.

Kinds of case:
  compact     one ka_compact call: caller-owned buffers and workspace
  actors      one request to a composed actor on device references, received
              before the next (the paper's programming model)
  batch       one ka_compact_batch call over many instances
  tick        what a serving loop issues for a group of requests: one
              ka_generate_batch, then one in-place ka_compact_batch per
              pipeline stage, lengths staying on the device
  mandelbrot  one ka_mandelbrot image (the paper's compute workload)
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1709_07781_gb300 as ka

# keep-tests in use: name -> (library kind, share of uniform data that passes)
PREDICATES = {
    "lt": (ka.KA_PRED_LT, None),               # x < floor(sel 2^32)
    "and_mask": (ka.KA_PRED_AND_MASK_EQ0, 0.25),  # (x & 3) == 0
    "topbits": (ka.KA_PRED_TOPBITS_LT, 0.5),   # (x >> 28) < 8
    "popc_odd": (ka.KA_PRED_POPC_ODD, 0.5),
    "mod3": (ka.KA_PRED_MOD_NE0, 2.0 / 3.0),   # x % 3 != 0
    "nonzero": (ka.KA_PRED_NE, None),          # x != 0, on data with a share of zeros
}
PARAMS = {"and_mask": 3, "topbits": 8, "popc_odd": 0, "mod3": 3, "nonzero": 0}

# Stages of the 4-stage pipeline: hash map, then three compactions.
PIPELINE4 = (("map", 1.0), ("topbits", 0.5), ("popc_odd", 0.5), ("mod3", 2.0 / 3.0))

ITEM = np.dtype([("in", "<u8"), ("out", "<u8"), ("n_ptr", "<u8"), ("count", "<u8"), ("n", "<u4"),
                 ("pred", "<i4"), ("param", "<u4"), ("xform", "<u4")])
GEN = np.dtype([("out", "<u8"), ("seed", "<u8"), ("n", "<u4"), ("pad", "<u4")])

# The Mandelbrot rectangle of the paper's workload.
RECT = (-0.5, -0.7375, 0.1, -0.1375)

TICK_ENTRIES = 1 << 28  # input entries that a serving loop groups at most


def listed():
    return [
        # The smallest request of the serving workload: one tile, latency only.
        dict(name="compact_1k", kind="compact", n=1024, pred="lt", sel=0.5, offset=0, hash=False, live=False),
        # A mid-size request of odd length (the serving sizes are log-uniform
        # in 2^10..2^24): many blocks, everything in L2.
        dict(name="compact_100k", kind="compact", n=100003, pred="and_mask", sel=0.25, offset=0, hash=False,
             live=False),
        # A stage inside a pipeline: hashed values, its live length in a
        # device word, a view that starts one entry past a 16-byte boundary.
        dict(name="compact_4m_view", kind="compact", n=4194309, pred="topbits", sel=0.5, offset=1, hash=True,
             live=True),
        # The large single compaction (1 GiB) at its three selectivities.
        dict(name="compact_256m_s01", kind="compact", n=1 << 28, pred="lt", sel=0.01, offset=0, hash=False,
             live=False),
        dict(name="compact_256m_s50", kind="compact", n=1 << 28, pred="lt", sel=0.5, offset=0, hash=False,
             live=False),
        dict(name="compact_256m_s99", kind="compact", n=1 << 28, pred="lt", sel=0.99, offset=0, hash=False,
             live=False),
        # The single pipeline of three actors: predicate, scan, scatter.
        dict(name="actors3_1m", kind="actors", pipe="three", n=1 << 20),
        # The 4-stage pipeline on device-resident data.
        dict(name="pipeline4_64m", kind="actors", pipe="four", n=1 << 26),
        # The paper's index step: chunk ids and literals interleaved, then
        # zeros removed (half of both are zero).
        dict(name="index_16m_pairs", kind="actors", pipe="index", n=(1 << 24) + 4),
        # 4096 instances of uneven size, each with its own threshold.
        dict(name="batch_4096", kind="batch", items=4096, lo=8, hi=20, sizes_seed=4),
        # A serving group: requests of 1 to 4 stages over fresh data.
        dict(name="tick_128", kind="tick", items=128, lo=10, hi=24, sizes_seed=5),
        # The paper's compute workload at 1920 x 1080.
        dict(name="mandelbrot_1080p", kind="mandelbrot", width=1920, height=1080, iters=100),
    ]


def _log_int(rng, lo, hi):
    """An integer log-uniform in [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["compact", "compact", "compact", "actors", "actors", "batch", "tick", "mandelbrot"])
    if kind == "compact":
        pred = rng.choice(sorted(PREDICATES))
        share = PREDICATES[pred][1]
        n = _log_int(rng, 1 << 10, 1 << 28)
        return dict(kind=kind, n=n, pred=pred, sel=round(rng.uniform(0.01, 0.99), 4) if share is None else share,
                    offset=rng.choice([0, 0, 0, 1, 2, 3]), hash=rng.random() < 0.25, live=rng.random() < 0.25)
    if kind == "actors":
        pipe = rng.choice(["three", "four", "index"])
        lo, hi = {"three": (1 << 10, 1 << 24), "four": (1 << 14, 1 << 26), "index": (1 << 12, 1 << 25)}[pipe]
        return dict(kind=kind, pipe=pipe, n=_log_int(rng, lo, hi))
    if kind == "batch":
        return dict(kind=kind, items=_log_int(rng, 256, 4096), lo=8, hi=rng.choice([12, 16, 20]),
                    sizes_seed=rng.randrange(1 << 20))
    if kind == "tick":
        hi = rng.choice([16, 20, 24])
        return dict(kind=kind, items=_log_int(rng, 2, 128 if hi == 24 else 1024), lo=10, hi=hi,
                    sizes_seed=rng.randrange(1 << 20))
    return dict(kind=kind, width=rng.randrange(320, 1921), height=rng.randrange(200, 1081),
                iters=_log_int(rng, 50, 400))


# ---------------------------------------------------------------------------
# Inputs.
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(n, seed):
    """n uniform uint32 values, as int32 bits."""
    return torch.randint(-(1 << 31), 1 << 31, (n,), dtype=torch.int32, device="cuda", generator=_generator(seed))


def _with_zeros(x, share, seed):
    """x with about `share` of its entries set to zero, in place."""
    return x.masked_fill_(torch.rand(x.shape, device="cuda", generator=_generator(seed)) < share, 0)


def _rearranged(x, seed):
    """The values of x in another order, set by the seed: place i gets entry
    (a i + b) mod n with a prime to n. Every seed's data then keeps the same
    number of entries, so results of different seeds have one length."""
    n = x.numel()
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    a = int(r.randint(1, max(2, n)))
    while math.gcd(a, n) != 1:
        a += 1
    i = torch.arange(n, dtype=torch.int64, device="cuda").mul_(a).add_(int(r.randint(0, n))).remainder_(n)
    return x[i]


def _threshold(sel):
    return max(0, min(0xFFFFFFFF, int(math.floor(sel * 4294967296.0))))


def _param(pred, sel):
    return _threshold(sel) if pred == "lt" else PARAMS[pred]


def _sizes(case):
    """Sizes log-uniform in [2^lo, 2^hi), fixed by the case."""
    r = np.random.RandomState(case["sizes_seed"])
    n = np.floor(np.exp2(case["lo"] + (case["hi"] - case["lo"]) * r.random_sample(case["items"]))).astype(np.int64)
    if case["kind"] == "tick":
        n = n[: max(1, int(np.searchsorted(np.cumsum(n), TICK_ENTRIES, side="right")))]
    return n


def _workspace(nbytes):
    """A 256-byte aligned, initialised workspace: (tensor that owns it, address)."""
    t = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    p = (t.data_ptr() + 255) // 256 * 256
    ka.check(ka.ka_workspace_init(p, nbytes, torch.cuda.current_stream()))
    return t, p


def _table(a):
    return torch.from_numpy(np.frombuffer(a.tobytes(), dtype=np.uint8).copy()).cuda()


def _arena(sizes):
    """Element offsets of regions of the given sizes (16-byte aligned), and the total."""
    off = np.concatenate([[0], np.cumsum((sizes + 3) // 4 * 4)])
    return off[:-1], int(off[-1])


# ---------------------------------------------------------------------------
# The actor system of the process and its pipelines: made once and kept, as a
# program that sends requests keeps them.
_kept = {}


def _system():
    if "system" not in _kept:
        s, h = ka.ka_system_create(torch.cuda.current_device())
        ka.check(s)
        _kept["system"] = h
    return _kept["system"]


def _pipeline(name):
    if name not in _kept:
        stages = {
            "three": [(ka.KA_STAGE_PREDICATE, ka.KA_PRED_AND_MASK_EQ0, 3), (ka.KA_STAGE_EXSCAN,),
                      (ka.KA_STAGE_SCATTER,)],
            "four": [(ka.KA_STAGE_MAP_HASH,), (ka.KA_STAGE_COMPACT, ka.KA_PRED_TOPBITS_LT, 8),
                     (ka.KA_STAGE_COMPACT, ka.KA_PRED_POPC_ODD, 0), (ka.KA_STAGE_COMPACT, ka.KA_PRED_MOD_NE0, 3)],
            "index": [(ka.KA_STAGE_PREPARE,), (ka.KA_STAGE_COMPACT, ka.KA_PRED_NE, 0)],
        }[name]
        pipe = None
        for spec in stages:
            s, a = ka.ka_spawn_stage(_system(), *spec)
            ka.check(s)
            if pipe is not None:
                s, a = ka.ka_compose(a, pipe)
                ka.check(s)
            pipe = a
        _kept[name] = pipe
    return _kept[name]


class _DeviceWords:
    """n uint32 words of device memory that the library owns, for torch.as_tensor."""

    def __init__(self, address, n):
        self.__cuda_array_interface__ = {"shape": (n,), "typestr": "<i4", "data": (address, False), "version": 3}


class _ActorState:
    """An actor, its input references and the last result, which is released
    when the next one has come or the state goes."""

    def __init__(self, pipe, inputs):
        self.pipe, self.inputs, self.held = _pipeline(pipe), inputs, ()
        self.refs = []
        for x in inputs:
            s, r = ka.ka_ref_wrap(_system(), x, x.numel(), x.numel())
            ka.check(s)
            self.refs.append(r)

    def release(self):
        for r in self.held:
            ka.ka_ref_release(r)
        self.held = ()

    def request(self):
        self.release()
        s, req = ka.ka_request(self.pipe, ka.make_msg(self.refs))
        ka.check(s)
        s, msg = ka.ka_receive(req)
        ka.check(s)
        self.held = tuple(msg.refs[: msg.n_refs])
        s, address, _, _, _ = ka.ka_ref_info(self.held[0])
        ka.check(s)
        return {"data": torch.as_tensor(_DeviceWords(address, msg.count), device="cuda"), "count": int(msg.count)}

    def __del__(self):
        self.release()
        for r in self.refs:
            ka.ka_ref_release(r)


# ---------------------------------------------------------------------------
def prepare(case, seed):
    stream = torch.cuda.current_stream().cuda_stream
    if case["kind"] == "compact":
        n, off = case["n"], case["offset"]
        whole = _uniform(n + off, seed)
        if case["pred"] == "nonzero":
            _with_zeros(whole, 1.0 - case["sel"], seed + 1)
        s, nbytes = ka.ka_workspace_size(n)
        ka.check(s)
        owner, ws = _workspace(nbytes)
        return dict(kind="compact", x=whole[off:], n=n, live=torch.full((1,), n, dtype=torch.int32, device="cuda")
                    if case["live"] else None, pred=PREDICATES[case["pred"]][0],
                    param=_param(case["pred"], case["sel"]), xform=ka.KA_XFORM_HASH if case["hash"] else ka.KA_XFORM_NONE,
                    out=torch.zeros(n, dtype=torch.int32, device="cuda"),
                    count=torch.zeros(1, dtype=torch.int32, device="cuda"), owner=owner, ws=ws, nbytes=nbytes,
                    stream=stream)
    if case["kind"] == "actors":
        n = case["n"]
        inputs = [_rearranged(_uniform(n, n), seed)]
        if case["pipe"] == "index":
            inputs = [_rearranged(_with_zeros(_uniform(n, n + k), 0.5, n + k + 2), seed + k) for k in range(2)]
        return dict(kind="actors", actors=_ActorState(case["pipe"], inputs))
    if case["kind"] == "batch":
        sizes = _sizes(case)
        off, total = _arena(sizes)
        share = np.random.RandomState(case["sizes_seed"] + 1).uniform(0.01, 0.99, sizes.size)
        x, out = _uniform(total, seed), torch.zeros(total, dtype=torch.int32, device="cuda")
        count = torch.zeros(sizes.size, dtype=torch.int32, device="cuda")
        t = np.zeros(sizes.size, dtype=ITEM)
        t["in"], t["out"] = x.data_ptr() + 4 * off, out.data_ptr() + 4 * off
        t["count"], t["n"] = count.data_ptr() + 4 * np.arange(sizes.size), sizes
        t["pred"], t["param"] = ka.KA_PRED_LT, [_threshold(v) for v in share]
        s, nbytes = ka.ka_batch_workspace_size(sizes.size, int(sizes.sum()))
        ka.check(s)
        owner, ws = _workspace(nbytes)
        return dict(kind="batch", x=x, out=out, count=count, table=_table(t), items=sizes.size, owner=owner, ws=ws,
                    nbytes=nbytes, stream=stream)
    if case["kind"] == "tick":
        sizes = _sizes(case)
        off, total = _arena(sizes)
        r = np.random.RandomState(case["sizes_seed"] + 1)
        depth = r.randint(1, 5, sizes.size)
        stages = r.randint(0, 4, (sizes.size, 4))
        buf = torch.zeros(total, dtype=torch.int32, device="cuda")
        count = torch.zeros((4, sizes.size), dtype=torch.int32, device="cuda")
        g = np.zeros(sizes.size, dtype=GEN)
        g["out"], g["n"] = buf.data_ptr() + 4 * off, sizes
        g["seed"] = np.random.RandomState(seed & 0x7FFFFFFF).randint(0, 1 << 62, sizes.size, dtype=np.int64)
        tables = []
        for d in range(int(depth.max())):
            at = np.nonzero(depth > d)[0]
            t = np.zeros(at.size, dtype=ITEM)
            t["in"] = t["out"] = g["out"][at]
            t["n"], t["count"] = sizes[at], count[d].data_ptr() + 4 * at
            t["n_ptr"] = count[d - 1].data_ptr() + 4 * at if d else 0
            names = [PIPELINE4[k][0] for k in stages[at, d]]
            t["pred"] = [ka.KA_PRED_ALL if v == "map" else PREDICATES[v][0] for v in names]
            t["param"] = [0 if v == "map" else PARAMS[v] for v in names]
            t["xform"] = [ka.KA_XFORM_HASH if v == "map" else ka.KA_XFORM_NONE for v in names]
            tables.append((_table(t), int(at.size)))
        s, nbytes = ka.ka_batch_workspace_size(sizes.size, int(sizes.sum()))
        ka.check(s)
        owner, ws = _workspace(nbytes)
        return dict(kind="tick", buf=buf, count=count, gen=_table(g), tables=tables, items=sizes.size, owner=owner,
                    ws=ws, nbytes=nbytes, stream=stream)
    r = np.random.RandomState(seed & 0x7FFFFFFF)
    dx, dy = r.uniform(-0.01, 0.01, 2)  # the view, moved a little
    return dict(kind="mandelbrot", out=torch.zeros((case["height"], case["width"]), dtype=torch.int32, device="cuda"),
                width=case["width"], height=case["height"], iters=case["iters"],
                rect=(RECT[0] + dx, RECT[1] + dy, RECT[2] + dx, RECT[3] + dy), stream=stream)


def run(state):
    s = state
    if s["kind"] == "compact":
        ka.check(ka.ka_compact(s["x"], s["n"], s["live"], s["pred"], s["param"], s["xform"], s["out"], s["count"],
                               s["ws"], s["nbytes"], stream=s["stream"]))
        return {"data": s["out"], "count": s["count"]}
    if s["kind"] == "actors":
        return s["actors"].request()
    if s["kind"] == "batch":
        ka.check(ka.ka_compact_batch(s["table"], s["items"], s["items"], s["ws"], s["nbytes"], stream=s["stream"]))
        return {"data": s["out"], "count": s["count"]}
    if s["kind"] == "tick":
        ka.check(ka.ka_generate_batch(s["gen"], s["items"], s["items"], s["ws"], s["nbytes"], s["stream"]))
        for table, items in s["tables"]:
            ka.check(ka.ka_compact_batch(table, items, s["items"], s["ws"], s["nbytes"], stream=s["stream"]))
        return {"data": s["buf"], "count": s["count"]}
    ka.check(ka.ka_mandelbrot(s["out"], s["width"], s["height"], *s["rect"], s["iters"], s["stream"]))
    return s["out"]


# ---------------------------------------------------------------------------
def _mean_steps(case):
    """Mean steps per pixel, from a coarse grid of the image."""
    re, im = np.meshgrid(np.linspace(RECT[0], RECT[2], 96), np.linspace(RECT[1], RECT[3], 96))
    c = re + 1j * im
    z, steps = np.zeros_like(c), np.zeros(c.shape)
    for _ in range(case["iters"]):
        inside = np.abs(z) <= 2.0
        z = np.where(inside, z * z + c, z)
        steps += inside
    return float(steps.mean())


def work(case):
    """Bytes: inputs read once and results written once (a chain of stages by
    its ends, except that the calls of a serving group are separate and each
    reads its input and writes its result). One integer operation or so a
    byte is left out; the Mandelbrot step is eight operations."""
    if case["kind"] == "compact":
        return {"bytes": 4 * case["n"] * (1 + case["sel"]), "flops": 0}
    if case["kind"] == "actors":
        n = case["n"]
        return {"bytes": {"three": 4 * n * 1.25, "four": 4 * n * (1 + 1 / 6), "index": 8 * n * 1.5}[case["pipe"]],
                "flops": 0}
    if case["kind"] == "batch":
        n = _sizes(case)
        share = np.random.RandomState(case["sizes_seed"] + 1).uniform(0.01, 0.99, n.size)
        return {"bytes": float((4 * n * (1 + share)).sum()), "flops": 0}
    if case["kind"] == "tick":
        n = _sizes(case)
        r = np.random.RandomState(case["sizes_seed"] + 1)
        depth = r.randint(1, 5, n.size)
        share = np.array([p for _, p in PIPELINE4])[r.randint(0, 4, (n.size, 4))]
        live, moved = n.astype(float), 4.0 * n.sum()
        for d in range(4):
            on = depth > d
            moved += float((4 * live * (1 + share[:, d]) * on).sum())
            live = live * np.where(on, share[:, d], 1.0)
        return {"bytes": float(moved), "flops": 0}
    pixels = case["width"] * case["height"]
    return {"bytes": 4 * pixels, "flops": 8 * pixels * _mean_steps(case)}
