"""What this repository's speed is measured on: the calls that a program around a
memory-bank video-segmentation network makes, through the package's public entry
points, from a 32 x 32 fp32 frame to 48 objects of 16 streams.

Kinds of case:
  start      once per sequence: the seed boxes and grid masks of the first frame's
             pixel masks, and the write keep-set of every object
  select     per frame: the keep-set of every object (prior, energies, top-k)
  readout    per frame: pruned cross-attention over the banks, scattered back
  commit     per frame: the write-pruned append to the banks
  close      per frame: closure of the decoder's masks, palette, masks at grid size
  sequence   several frames, each select + readout + commit, captured once in a CUDA
             graph that is replayed (how a serving program runs the path)

Calls of one kind are issued eagerly, a frame's worth each.  Inputs are drawn on
the GPU from the seed: token grids N(0, 1) with more energy inside the objects,
objects as rotated ellipses, keys and values N(0, 1), queries (or keys) scaled so
that the softmax is peaked as a trained network's is.
"""
import math

import torch

from paper_2608_22526_gb300 import rs3, synth
from paper_2608_22526_gb300.pipeline import Pipeline

DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
R_S, CAP = 4, 14                       # prior radius and growth cap: the defaults


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # The first frame of an 8-object clip at 1024 x 1024: seeds and write keep-sets.
        dict(name="start_8obj", kind="start", U=8, G=1, h=1024, w=1024, s=16, lo=0.02, hi=0.40, D_w=12, union=False),
        # The smallest per-frame call: one object on SAM2's 64 x 64 grid; latency and launches.
        dict(name="select_1obj", kind="select", G=1, per=1, m=64, n=64, C=256, dtype="bf16", rho=0.3,
             lo=0.05, hi=0.30, union=False),
        # The same call for 16 streams of 3 objects on 96 x 96 grids, all streams in one call.
        dict(name="select_16x3", kind="select", G=16, per=3, m=96, n=96, C=256, dtype="bf16", rho=0.3,
             lo=0.03, hi=0.25, union=False),
        # The fp32 configuration (32 x 32 grid, one head of 64, two whole frames in the
        # bank): a whole frame of the smallest workload, nothing but launches and latency.
        dict(name="frame_tiny_fp32", kind="sequence", G=1, per=1, m=32, n=32, H=1, d=64, dtype="f32", frames=1,
             prefill=2, n_cond=0, window=-1, n_ptr=0, rho=0.3, lo=0.08, hi=0.12, union=False, rope=False, sharp=2.0),
        # fp32 networks at the usual grid: four heads of 64, one object, seven frames.
        dict(name="readout_fp32", kind="readout", G=1, per=1, m=64, n=64, H=4, d=64, dtype="f32", n_cond=1, window=6,
             ring_frames=6, n_ptr=16, rho=0.3, lo=0.05, hi=0.30, rope=False, residual="inplace", sharp=2.0),
        # SAM2, one object: one head of 256, conditioning frame + 6 recent + 16 pointer rows.
        dict(name="readout_1obj", kind="readout", G=1, per=1, m=64, n=64, H=1, d=256, dtype="bf16", n_cond=1, window=6,
             ring_frames=6, n_ptr=16, rho=0.3, lo=0.05, hi=0.30, rope=False, residual="inplace", sharp=2.0),
        # Eight objects on one grid, their banks of very different lengths.
        dict(name="readout_8obj", kind="readout", G=1, per=8, m=64, n=64, H=1, d=256, dtype="bf16", n_cond=1, window=6,
             ring_frames=6, n_ptr=0, rho=0.3, lo=0.02, hi=0.40, rope=False, residual="inplace", sharp=2.0),
        # Serving: 16 streams x 3 objects, four heads of 64, RoPE, Eq. 6's literal output
        # (zeros off the keep-set) for a network that adds the residual itself.
        dict(name="readout_16x3", kind="readout", G=16, per=3, m=96, n=96, H=4, d=64, dtype="bf16", n_cond=1, window=6,
             ring_frames=6, n_ptr=16, rho=0.3, lo=0.03, hi=0.25, rope=True, residual="none", sharp=2.0),
        # A long video: one object, 490 frames kept, about 300 000 keys.
        dict(name="readout_long", kind="readout", G=1, per=1, m=64, n=64, H=1, d=256, dtype="bf16", n_cond=1, window=-1,
             ring_frames=490, n_ptr=0, rho=0.3, lo=0.14, hi=0.16, rope=False, residual="inplace", sharp=2.5),
        # The serving workload's commit, keys stored rotated, the window full (one frame evicted).
        dict(name="commit_16x3", kind="commit", G=16, per=3, m=96, n=96, H=4, d=64, dtype="bf16", n_cond=1, window=6,
             n_ptr=16, lo=0.03, hi=0.25, rope=True, masked=True),
        # The serving workload's decoder output: 48 objects at 384 x 384.
        dict(name="close_16x3", kind="close", G=16, per=3, h=384, w=384, radius=4, s=4, lo=0.02, hi=0.25, closed=False),
        # Eight objects, 8 frames from the conditioning frame on, as one CUDA graph.
        dict(name="sequence_8obj", kind="sequence", G=1, per=8, m=64, n=64, H=1, d=256, dtype="bf16", frames=8,
             prefill=0, n_cond=1, window=6, n_ptr=0, rho=0.3, lo=0.02, hi=0.40, union=False, rope=False, sharp=2.0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed kinds, anywhere in their ranges, odd sizes among them."""
    while True:
        kind = rng.choice(["start", "select", "select", "readout", "readout", "readout", "commit", "close", "sequence"])
        lo = rng.choice([0.02, 0.03, 0.05, 0.14])
        cov = dict(lo=lo, hi=rng.choice([0.16, 0.25, 0.30, 0.40]))
        if kind == "start":
            s = rng.choice([8, 16])
            c = dict(kind=kind, U=_log(rng, 1, 48), G=1, h=s * rng.randint(20, 64), w=16 * s * rng.randint(1, 4) // (s // 8),
                     s=s, D_w=rng.choice([4, 12, 24]), union=rng.random() < 0.3, **cov)
        elif kind == "close":
            s = rng.choice([2, 4])
            c = dict(kind=kind, G=_log(rng, 1, 16), per=_log(rng, 1, 8), h=s * rng.randint(24, 128), w=32 * rng.randint(3, 16),
                     radius=rng.choice([4, 4, 4, 2, 7]), s=s, closed=rng.random() < 0.3, **cov)
            if c["G"] * c["per"] * c["h"] * c["w"] > 9e6:
                continue
        else:
            m, n = _log(rng, 24, 112), _log(rng, 24, 112)
            G = _log(rng, 1, 16)
            per = _log(rng, 1, max(1, min(8, 48 // G)))
            dtype = "bf16" if rng.random() < 0.7 else "f32"
            H, d = rng.choice([(1, 256), (4, 64), (2, 128), (8, 64), (1, 64)]) if dtype == "bf16" else \
                rng.choice([(1, 64), (4, 64), (2, 32), (2, 128), (1, 256)])
            rho = rng.choice([0.2, 0.3, 0.3, 0.5, 0.7, 1.0])
            if kind == "select":
                c = dict(kind=kind, G=G, per=per, m=m, n=n, C=H * d, dtype=dtype, rho=rho, union=rng.random() < 0.4, **cov)
            elif kind == "readout":
                window = rng.choice([1, 3, 6, 6, -1])
                c = dict(kind=kind, G=G, per=per, m=m, n=n, H=H, d=d, dtype=dtype, n_cond=rng.choice([0, 1, 1, 2]), window=window,
                         ring_frames=window if window > 0 else _log(rng, 8, 200), n_ptr=rng.choice([0, 4, 16, 61]), rho=rho,
                         rope=rng.random() < 0.4, residual=rng.choice(["inplace", "inplace", "none", "other"]),
                         sharp=rng.choice([1.0, 2.0, 3.0]), **cov)
            elif kind == "commit":
                c = dict(kind=kind, G=G, per=per, m=m, n=n, H=H, d=d, dtype=dtype, n_cond=rng.choice([0, 1]),
                         window=rng.choice([2, 4, 6]), n_ptr=rng.choice([0, 16]), rope=rng.random() < 0.5,
                         masked=rng.random() < 0.8, **cov)
                if G * per * m * n * (c["n_cond"] + c["window"]) * H * d * (2 if dtype == "bf16" else 4) > 1.6e9:
                    continue
            else:
                frames = rng.randint(2, 10)
                c = dict(kind=kind, G=min(G, 4), per=min(per, 8), m=m, n=n, H=H, d=d, dtype=dtype, frames=frames, prefill=0,
                         n_cond=1, window=rng.choice([3, 6]), n_ptr=0, rho=rho, union=rng.random() < 0.3,
                         rope=rng.random() < 0.3, sharp=2.0, **cov)
                if c["G"] * c["per"] * m * n * H * d * frames > 1.6e8:
                    continue
            # no more arithmetic than the largest listed cases; the fp32 path runs on the CUDA cores
            if work(c)["flops"] > (4e11 if dtype == "bf16" else 1e10):
                continue
        return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
class _Gen:
    """Draws from (seed, tag): any part of a case's inputs can be drawn again on its own."""

    def __init__(self, seed):
        self.seed = int(seed)

    def __call__(self, *tag):
        x = self.seed & 0x7FFFFFFF
        for t in tag:
            x = (x * 1000003 + int(t) + 12345) % ((1 << 61) - 1)
        g = torch.Generator(device="cuda")
        g.manual_seed(x)
        return g


def _randn(g, shape, dtype, scale=1.0):
    return (torch.randn(shape, generator=g, device="cuda") * scale).to(DTYPE[dtype])


def _covers(U, lo, hi, frame):
    """Coverage of each unit's object at a frame: spread over [lo, hi], moving a little
    from frame to frame; the same for every seed, so that the work is."""
    return [lo + (hi - lo) * (0.5 + 0.5 * math.sin(1.7 * u + 0.35 * frame + 0.9)) for u in range(U)]


def _ellipses(g, U, h, w, covs):
    """bool [U, h, w]: a filled rotated ellipse each, its centre well inside."""
    r = torch.rand((U, 4), generator=g, device="cuda", dtype=torch.float64)
    area = torch.tensor(covs, device="cuda", dtype=torch.float64) * (h * w)
    aspect = 0.6 + r[:, 0]
    a, b = (area * aspect / math.pi).sqrt(), (area / (aspect * math.pi)).sqrt()
    th = r[:, 1] * math.pi
    cy, cx = (0.35 + 0.3 * r[:, 2]) * h, (0.35 + 0.3 * r[:, 3]) * w
    ct, st = th.cos(), th.sin()

    def over(x):
        return x[:, None, None]

    v = torch.arange(h, device="cuda", dtype=torch.float64)[None, :, None] + 0.5 - over(cy)
    u = torch.arange(w, device="cuda", dtype=torch.float64)[None, None, :] + 0.5 - over(cx)
    return ((u * over(ct) + v * over(st)) / over(a)) ** 2 + ((v * over(ct) - u * over(st)) / over(b)) ** 2 <= 1.0


def _masks(g, c, frame):
    U = c["G"] * c["per"]
    return _ellipses(g(3, frame), U, c["m"], c["n"], _covers(U, c["lo"], c["hi"], frame)).reshape(U, -1).to(torch.uint8)


def _z(g, c, frame, masks, scale=1.0):
    """[G, mn, C]: N(0, 1), 1.25 times that inside the group's objects."""
    G, mn = c["G"], c["m"] * c["n"]
    C = c["C"] if "C" in c else c["H"] * c["d"]
    z = torch.randn((G, mn, C), generator=g(4, frame), device="cuda") * scale
    inside = masks.view(G, -1, mn).amax(1).bool()
    z *= torch.where(inside, 1.25, 1.0)[..., None]
    return z.to(DTYPE[c["dtype"]])


def _kv(g, c, frame, scale=1.0):
    shape = (c["G"] * c["per"], c["m"] * c["n"], c["H"] * c["d"])
    return _randn(g(5, frame), shape, c["dtype"], scale), _randn(g(6, frame), shape, c["dtype"])


def _pointers(g, c):
    shape = (c["G"] * c["per"], c["n_ptr"], c["H"] * c["d"])
    return _randn(g(7, 0), shape, c["dtype"]), _randn(g(8, 0), shape, c["dtype"])


def _rope(c):
    """[mn, d/2, 2] (cos, sin): half of the pairs turn with the column, half with the row."""
    m, n, half = c["m"], c["n"], c["d"] // 4
    cell = torch.arange(m * n, device="cuda", dtype=torch.float64)
    freq = 10000.0 ** (-torch.arange(half, device="cuda", dtype=torch.float64) / half)
    ang = torch.cat([(cell % n)[:, None] * freq, (cell // n)[:, None] * freq], 1)
    return torch.stack([ang.cos(), ang.sin()], -1).float().contiguous()


def _dilate(masks, m, n, r):
    x = masks.reshape(-1, 1, m, n).float()
    return torch.nn.functional.max_pool2d(x, 2 * r + 1, 1, r).reshape(-1, m * n) > 0


def _unit_group(c):
    return torch.arange(c["G"], dtype=torch.int32, device="cuda").repeat_interleave(c["per"])


def _kmax(rho, mn):
    return int(math.floor(rho * mn))


def _top(score, prior, k):
    """(idx int32 [U, k] ascending, count): the k best of the prior's cells."""
    U, mn = score.shape
    val, pos = torch.where(prior, score, -1.0).topk(k, dim=1)
    pos = torch.where(val >= 0, pos, mn).sort(dim=1).values
    return torch.where(pos < mn, pos, 0).to(torch.int32), (pos < mn).sum(1).to(torch.int32)


def _readout_inputs(c, seed):
    g, mn, U = _Gen(seed), c["m"] * c["n"], c["G"] * c["per"]
    last = c["n_cond"] + c["ring_frames"]
    q = _z(g, c, last, _masks(g, c, last), c["sharp"])
    prior = _dilate(_masks(g, c, last - 1), c["m"], c["n"], R_S)
    score = torch.rand((U, mn), generator=g(9, 0), device="cuda")
    idx, count = _top(score, prior, max(1, _kmax(c["rho"], mn)))
    res = _randn(g(10, 0), (U, mn, c["H"] * c["d"]), c["dtype"]) if c["residual"] != "none" else None
    return g, q, idx, count, res


def _close_inputs(c, seed):
    """Logits positive inside an ellipse; one pixel in a hundred of it turned negative,
    one in five hundred outside turned positive."""
    g, U, h, w = _Gen(seed), c["G"] * c["per"], c["h"], c["w"]
    inside = _ellipses(g(3, 0), U, h, w, _covers(U, c["lo"], c["hi"], 0))
    mag = torch.randn((U, h, w), generator=g(4, 0), device="cuda").abs() + 0.5
    noise = torch.rand((U, h, w), generator=g(5, 0), device="cuda")
    return torch.where(inside ^ (noise < torch.where(inside, 0.01, 0.002)), mag, -mag)


def _workload(c):
    return synth.Workload("case", 0, c["m"], c["n"], c["H"], c["d"], c["dtype"], c["G"], c["per"], c["frames"], c["lo"], c["hi"],
                          c["n_cond"], c["window"], c["n_ptr"], prefill_frames=c["prefill"], union_mode=int(c["union"]),
                          rho=c["rho"], r_s=R_S, c=CAP)


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _status():
    return torch.zeros(1, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    c = dict(case)
    return {"start": _prepare_start, "select": _prepare_select, "readout": _prepare_readout, "commit": _prepare_commit,
            "close": _prepare_close, "sequence": _prepare_sequence}[c["kind"]](c, seed)


def run(state):
    return state["run"](state)


def _prepare_start(c, seed):
    g, U = _Gen(seed), c["U"]
    m, n = c["h"] // c["s"], c["w"] // c["s"]
    masks = _ellipses(g(3, 0), U, c["h"], c["w"], _covers(U, c["lo"], c["hi"], 0)).to(torch.uint8) * 255

    def cells():
        return torch.empty((U, m * n), dtype=torch.uint8, device="cuda")

    return dict(run=_run_start, c=c, m=m, n=n, masks=masks, track=torch.zeros((U, 6), dtype=torch.int32, device="cuda"),
                grid=cells(), box=cells(), kw=cells(), unit_group=torch.zeros(U, dtype=torch.int32, device="cuda"),
                params=rs3.default_params(D_w=c["D_w"], union_mode=int(c["union"])), status=_status())


def _run_start(s):
    c = s["c"]
    rs3.rs3_seed_from_masks(s["masks"], c["U"], c["h"], c["w"], c["s"], s["track"], s["grid"], s["box"])
    rs3.rs3_write_keepset(s["grid"], s["unit_group"], c["U"], s["m"], s["n"], s["params"], s["kw"], s["status"])
    return s["track"], s["grid"], s["box"], s["kw"]


def _prepare_select(c, seed):
    g, mn, U = _Gen(seed), c["m"] * c["n"], c["G"] * c["per"]
    params = rs3.default_params(rho=c["rho"], r_s=R_S, c=CAP, union_mode=int(c["union"]))
    ws = torch.empty(rs3.rs3_select_workspace_bytes(c["G"], U, c["m"], c["n"]), dtype=torch.uint8, device="cuda")
    return dict(run=_run_select, c=c, U=U, z=_z(g, c, 1, _masks(g, c, 1)), prev=_masks(g, c, 0), unit_group=_unit_group(c),
                track=torch.zeros((U, 6), dtype=torch.int32, device="cuda"), params=params,
                idx=torch.zeros((U, max(1, _kmax(c["rho"], mn))), dtype=torch.int32, device="cuda"),
                count=torch.zeros(U, dtype=torch.int32, device="cuda"), ws=ws, status=_status())


def _run_select(s):
    c = s["c"]
    rs3.rs3_select_queries(s["z"], c["dtype"], c["G"], c["m"], c["n"], c["C"], s["prev"], s["unit_group"], s["U"], s["track"],
                           s["params"], s["idx"], s["count"], s["ws"], s["status"])
    return s["idx"], s["count"], s["track"]


def _ring_rows(c):
    """Rows of an unbounded bank: what the objects' greatest coverage can fill."""
    mn = c["m"] * c["n"]
    return c["window"] * mn if c["window"] > 0 else c["ring_frames"] * min(mn, int(math.ceil(c["hi"] * 1.1 * mn)) + 8)


def _prepare_readout(c, seed):
    g, q, idx, count, res = _readout_inputs(c, seed)
    mn, U = c["m"] * c["n"], c["G"] * c["per"]
    status = _status()
    bank = rs3.Bank(U, c["H"], c["d"], c["dtype"], mn, c["n_cond"], c["window"], _ring_rows(c), max(1, c["ring_frames"]), c["n_ptr"])
    rope = _rope(c) if c["rope"] else None
    for f in range(c["n_cond"] + c["ring_frames"]):
        k, v = _kv(g, c, f)
        if rope is None:
            rs3.rs3_bank_commit(bank, k, v, _masks(g, c, f), int(f < c["n_cond"]), status)
        else:
            rs3.rs3_bank_commit_rope(bank, k, v, _masks(g, c, f), int(f < c["n_cond"]), rope, status)
    if c["n_ptr"]:
        rs3.rs3_bank_set_pointers(bank, *_pointers(g, c), status)
    out = res if c["residual"] == "inplace" else torch.empty((U, mn, c["H"] * c["d"]), dtype=DTYPE[c["dtype"]], device="cuda")
    k_max = idx.shape[1]
    ws = torch.empty(rs3.rs3_readout_workspace_bytes(U, c["H"], c["d"], k_max, c["dtype"]), dtype=torch.uint8, device="cuda")
    return dict(run=_run_readout, c=c, mn=mn, q=q, unit_group=_unit_group(c), idx=idx, count=count, k_max=k_max, bank=bank, rope=rope,
                res=res, out=out, ws=ws, status=status)


def _run_readout(s):
    c = s["c"]
    rs3.rs3_memory_readout(s["q"], c["dtype"], c["G"], s["mn"], c["H"], c["d"], s["unit_group"], s["idx"], s["count"], s["k_max"],
                           s["bank"], s["rope"], s["res"], s["out"], 0.0, s["ws"], s["status"])
    return s["out"]


def _prepare_commit(c, seed):
    g, mn, U = _Gen(seed), c["m"] * c["n"], c["G"] * c["per"]
    status = _status()
    bank = rs3.Bank(U, c["H"], c["d"], c["dtype"], mn, c["n_cond"], c["window"], c["window"] * mn, c["window"], c["n_ptr"])
    s = dict(run=_run_commit, c=c, bank=bank, rope=_rope(c) if c["rope"] else None, status=status, is_cond=0)
    last = c["n_cond"] + c["window"]
    for f in range(last):                        # the window full, as in the middle of a sequence
        s["kv"], s["mask"], s["is_cond"] = _kv(g, c, f), _masks(g, c, f), int(f < c["n_cond"])
        _run_commit(s)
    s["kv"], s["mask"], s["is_cond"] = _kv(g, c, last), _masks(g, c, last) if c["masked"] else None, 0
    return s


def _run_commit(s):
    bank, (k, v) = s["bank"], s["kv"]
    if s["rope"] is None:
        rs3.rs3_bank_commit(bank, k, v, s["mask"], s["is_cond"], s["status"])
    else:
        rs3.rs3_bank_commit_rope(bank, k, v, s["mask"], s["is_cond"], s["rope"], s["status"])
    return bank.k_store, bank.v_store, s["status"]


def _prepare_close(c, seed):
    U = c["G"] * c["per"]

    def u8(*shape):
        return torch.empty(shape, dtype=torch.uint8, device="cuda")

    return dict(run=_run_close, c=c, U=U, logits=_close_inputs(c, seed),
                start=torch.arange(c["G"] + 1, dtype=torch.int32, device="cuda") * c["per"], palette=u8(c["G"], c["h"], c["w"]),
                closed=u8(U, c["h"], c["w"]) if c["closed"] else None,
                grid=u8(U, c["h"] // c["s"], c["w"] // c["s"]) if c["w"] % c["s"] == 0 else None, status=_status())


def _run_close(s):
    c = s["c"]
    rs3.rs3_close_argmax(s["logits"], s["start"], c["G"], s["U"], c["h"], c["w"], c["radius"], c["s"], s["palette"], s["closed"],
                         s["grid"], s["status"])
    return [t for t in (s["palette"], s["closed"], s["grid"]) if t is not None]


def _frames(c):
    """Frames committed whole before the sequence, and the frames of the sequence."""
    return range(c["prefill"]), range(c["prefill"], c["prefill"] + c["frames"])


def _prepare_sequence(c, seed):
    g, w = _Gen(seed), _workload(c)
    pipe = Pipeline(w)
    before, during = _frames(c)
    kv = {f: _kv(g, c, f, c["sharp"]) for f in [*before, *during]}
    masks = {f: _masks(g, c, f) for f in [*before, *during]}
    z = {f: _z(g, c, f, masks[f]) for f in during}
    rope = _rope(c) if c["rope"] else None
    first = during[0] + (1 if c["n_cond"] else 0)   # the conditioning frame is only committed
    blank = torch.zeros_like(masks[during[0]])
    if c["n_cond"] == 0 and c["prefill"] == 0:
        raise ValueError("an empty bank")
    x = {f: z[f].repeat_interleave(c["per"], 0).contiguous() for f in during if f >= first}

    def frames(x):
        pipe.reset()
        for f in before:
            pipe.commit(*kv[f], None, 0, rope)
        for f in during:
            if f >= first:
                pipe.select(z[f], masks.get(f - 1, blank))
                pipe.readout(z[f], x[f], x[f], rope)
            pipe.commit(*kv[f], masks[f], int(f < first), rope)

    frames({f: t.clone() for f, t in x.items()})     # first use of every kernel, before the capture
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        frames(x)
    return dict(run=_run_sequence, c=c, pipe=pipe, x=x, graph=graph, keep=(kv, masks, z, rope, blank))


def _run_sequence(s):
    s["graph"].replay()
    p = s["pipe"]
    return dict(out=list(s["x"].values()), idx=p.idx, count=p.count, track=p.track, k=p.bank.k_store, v=p.bank.v_store, status=p.status)


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _prior_cells(c, frame):
    """Cells of each unit's dilated ellipse, on average over its angle."""
    mn = c["m"] * c["n"]
    out = []
    for cov in _covers(c["G"] * c["per"], c["lo"], c["hi"], frame):
        r = math.sqrt(cov * mn / math.pi)
        out.append(min(mn, cov * mn + 2 * R_S * (4 * r) + 4 * R_S * R_S))
    return out


def _attend(c, frame, lengths):
    """(bytes, flops) of one frame's readout over banks of these lengths."""
    mn, D, es = c["m"] * c["n"], c["H"] * c["d"], 2 if c["dtype"] == "bf16" else 4
    kept = [min(p, _kmax(c["rho"], mn)) for p in _prior_cells(c, frame - 1)]
    flops = sum(4.0 * k * L * D for k, L in zip(kept, lengths))
    nbytes = 2 * sum(lengths) * D * es + sum(kept) * (D * es + 4)
    residual = c.get("residual", "inplace")
    if residual == "inplace":
        nbytes += 2 * sum(kept) * D * es
    else:
        nbytes += (1 if residual == "none" else 2) * len(kept) * mn * D * es
    if c["rope"]:
        nbytes += mn * c["d"] * 4
    return nbytes, flops


def _lengths(c, frames, whole=()):
    """Rows that each unit's bank holds of these frames."""
    mn, U = c["m"] * c["n"], c["G"] * c["per"]
    out = [float(c["n_ptr"])] * U
    for f in frames:
        out = [a + (mn if f in whole else cov * mn) for a, cov in zip(out, _covers(U, c["lo"], c["hi"], f))]
    return out


def _commit_bytes(c, frame, whole=False):
    mn, U, es = c["m"] * c["n"], c["G"] * c["per"], 2 if c["dtype"] == "bf16" else 4
    rows = U * mn if whole else sum(_covers(U, c["lo"], c["hi"], frame)) * mn
    return rows * 4 * c["H"] * c["d"] * es + (0 if whole else U * mn) + (mn * c["d"] * 4 if c["rope"] else 0)


def _select_work(c, frame):
    mn, U, C = c["m"] * c["n"], c["G"] * c["per"], c["C"] if "C" in c else c["H"] * c["d"]
    prior = _prior_cells(c, frame - 1)
    rows = sum(min(mn, sum(prior[g * c["per"]:(g + 1) * c["per"]])) for g in range(c["G"]))
    kept = sum(min(p, _kmax(c["rho"], mn)) for p in prior)
    return U * mn + rows * C * (2 if c["dtype"] == "bf16" else 4) + 4 * kept, 2.0 * rows * C


def work(case):
    c = case
    if c["kind"] == "start":
        cells = c["h"] * c["w"] // c["s"] ** 2
        return {"bytes": c["U"] * (c["h"] * c["w"] + 3 * cells + 24), "flops": 0}
    if c["kind"] == "close":
        px, U = c["h"] * c["w"], c["G"] * c["per"]
        return {"bytes": U * px * (5 if c["closed"] else 4) + c["G"] * px + U * px // c["s"] ** 2, "flops": 0}
    if c["kind"] == "select":
        b, f = _select_work(c, 1)
        return {"bytes": b, "flops": f}
    if c["kind"] == "commit":
        return {"bytes": _commit_bytes(c, c["n_cond"] + c["window"], not c["masked"]), "flops": 0}
    if c["kind"] == "readout":
        last = c["n_cond"] + c["ring_frames"]
        b, f = _attend(c, last, _lengths(c, range(last)))
        return {"bytes": b, "flops": f}
    before, during = _frames(c)
    nbytes = flops = 0.0
    held = list(before)
    for f in [*before, *during]:
        if f in during and not (c["n_cond"] and f == during[0]):
            b, n = _select_work(c, f)
            p, q = _attend(c, f, _lengths(c, held, before))
            nbytes, flops = nbytes + b + p, flops + n + q
        nbytes += _commit_bytes(c, f, f in before)
        if f in during:
            held.append(f)
        if c["window"] > 0:                        # the conditioning frame stays
            held = held[:c["n_cond"]] + held[c["n_cond"]:][-c["window"]:]
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# tolerance and the same in 64 bits
# ---------------------------------------------------------------------------
def tolerance(case):
    c = case
    if c["kind"] in ("start", "select", "close") or (c["kind"] == "commit" and not c["rope"]):
        return "exact"                             # whole numbers, or rows copied as they are
    if c["dtype"] == "f32":
        return {"rel": 4e-6}                       # fp32 sums of thousands of terms in another order
    if c["kind"] == "commit":
        return {"rel": 1e-3}                       # one rounding to bf16, seldom the other way
    # one rounding of the output, and of each probability, to bf16: four times the error
    # against 64 bits (0.0042 of the attention alone, 0.0009 with the residual added)
    return {"rel": 1.6e-2 if c.get("residual") == "none" else 4e-3}


def _turn(x, rope, H):
    """x f64 [rows, D] turned by its own cells' angles [rows, d/2, 2]."""
    r, (cs, sn) = x.reshape(x.shape[0], H, -1, 2), rope.double().unbind(-1)
    a, b = r[..., 0], r[..., 1]
    cs, sn = cs[:, None], sn[:, None]
    return torch.stack([a * cs - b * sn, a * sn + b * cs], -1).reshape(x.shape)


def _attention(c, q, K, V):
    """f64 [rows, D] softmax attention by heads."""
    H, d = c["H"], c["d"]
    out = torch.empty_like(q)
    for h in range(H):
        s = slice(h * d, (h + 1) * d)
        p = q[:, s] @ K[:, s].T
        p *= 1.0 / math.sqrt(d)
        p -= p.amax(1, keepdim=True)
        p.exp_()
        out[:, s] = (p @ V[:, s]) / p.sum(1, keepdim=True)
        del p
    return out


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "readout":
        return _exact_readout(c, seed)
    if c["kind"] == "commit" and c["rope"]:
        return _exact_commit(c, seed)
    if c["kind"] == "sequence":
        return _exact_sequence(c, seed)
    return None                                    # whole numbers and copies


def _exact_readout(c, seed):
    g, q, idx, count, res = _readout_inputs(c, seed)
    U, mn, D, per = c["G"] * c["per"], c["m"] * c["n"], c["H"] * c["d"], c["per"]
    rope = _rope(c) if c["rope"] else None
    K, V = [[] for _ in range(U)], [[] for _ in range(U)]
    for f in range(c["n_cond"] + c["ring_frames"]):
        (k, v), keep = _kv(g, c, f), _masks(g, c, f).bool()
        for u in range(U):
            x = k[u][keep[u]]
            # rows are stored in the bank's type: turned, then rounded once
            K[u].append(x if rope is None else _turn(x.double(), rope[keep[u]], c["H"]).to(x.dtype))
            V[u].append(v[u][keep[u]])
    if c["n_ptr"]:
        kp, vp = _pointers(g, c)
        for u in range(U):
            K[u].append(kp[u])
            V[u].append(vp[u])
    out = torch.zeros((U, mn, D), dtype=torch.float64, device="cuda") if res is None else res.double()
    for u in range(U):
        cells = idx[u, :int(count[u])].long()
        x = q[u // per][cells].double()
        if rope is not None:
            x = _turn(x, rope[cells], c["H"])
        out[u, cells] += _attention(c, x, torch.cat(K[u]).double(), torch.cat(V[u]).double())
    return out


def _exact_commit(c, seed):
    g, mn, U = _Gen(seed), c["m"] * c["n"], c["G"] * c["per"]
    rows = (c["n_cond"] + c["window"]) * mn + c["n_ptr"]
    K = torch.zeros((U, rows, c["H"] * c["d"]), dtype=torch.float64, device="cuda")
    rope = _rope(c)
    tail = [0] * U
    pinned, last = c["n_cond"] * mn, c["n_cond"] + c["window"]
    for f in range(last + 1):
        (k, _), keep = _kv(g, c, f), _masks(g, c, f).bool()
        if f == last and not c["masked"]:
            keep = torch.ones_like(keep)
        for u in range(U):
            x = _turn(k[u][keep[u]].double(), rope[keep[u]], c["H"])
            if f < c["n_cond"]:                    # one pinned frame at most in these cases
                K[u, :len(x)] = x
            else:
                at = pinned + (tail[u] + torch.arange(len(x), device="cuda")) % (c["window"] * mn)
                K[u, at] = x
                tail[u] += len(x)
    return K, None, None


def _exact_sequence(c, seed):
    g, mn, U, per = _Gen(seed), c["m"] * c["n"], c["G"] * c["per"], c["per"]
    before, during = _frames(c)
    rope = _rope(c) if c["rope"] else None
    first = during[0] + (1 if c["n_cond"] else 0)
    held, outs, masks = [], [], {}
    for f in [*before, *during]:
        masks[f] = _masks(g, c, f)
        k, v = _kv(g, c, f, c["sharp"])
        if f in during and f >= first:
            z = _z(g, c, f, masks[f])
            prior = _dilate(masks[f - 1] if f - 1 in masks else torch.zeros_like(masks[f]), c["m"], c["n"], R_S)
            if c["union"]:
                prior = prior.view(c["G"], per, mn).any(1).repeat_interleave(per, 0)
            energy = z.double().square().sum(-1).repeat_interleave(per, 0)
            idx, count = _top(energy, prior, _kmax(c["rho"], mn))
            out = z.double().repeat_interleave(per, 0)
            for u in range(U):
                cells = idx[u, :int(count[u])].long()
                x = z[u // per][cells].double()
                if rope is not None:
                    x = _turn(x, rope[cells], c["H"])
                out[u, cells] += _attention(c, x, torch.cat([h[0][u] for h in held]).double(), torch.cat([h[1][u] for h in held]).double())
            outs.append(out)
        keep = (torch.ones_like(masks[f]) if f in before else masks[f]).bool()
        rows = []
        for u in range(U):
            x = k[u][keep[u]]
            rows.append(x if rope is None else _turn(x.double(), rope[keep[u]], c["H"]).to(x.dtype))
        held.append((rows, [v[u][keep[u]] for u in range(U)]))
        if c["window"] > 0:
            held = held[:c["n_cond"]] + held[c["n_cond"]:][-c["window"]:]
    return dict(out=outs, idx=None, count=None, track=None, k=None, v=None, status=None)
