"""Performance cases: the renders that users of the library ask for.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``frame``       one map in device memory, ``Context.render`` (ASK);
* ``noalloc``     the same through ``ask.render_noalloc`` (a frame loop that
                  may not allocate);
* ``host``        one map in pinned host memory, ``Context.render_host``;
* ``exhaustive``  every pixel's own dwell, ``Context.render``;
* ``batch``       frames of mixed size and zoom in one ``render_batch``;
* ``graph``       the same captured once, ``Context.graph_batch``, replayed;
* ``deep``        a zoom past 1e4 with ``Context.render64`` (ASK), in
                  binary64 or, ``ff``, in float-float arithmetic.

Sizes, dwell caps and subdivision parameters come from the paper's
configurations (Sec. 6.1-6.2, ``inputs.C0`` to ``C2``), from the batched,
served and deep-zoom workloads of ``inputs`` and from the tests.  ``spot``
says where a window lies: ``paper`` and ``wide`` are the windows that show
the whole set, a number is a stored boundary pixel that the window is
centred on at ``zoom``, other names are ``inputs.DEEP_SPOTS`` (a zoom below
1 widens them).  The seed
moves and scales a window by at most a few hundredths of its side, as a
user who pans and zooms does, so every seed gives another map of the same
kind.  All outputs are whole numbers (dwells).
"""
import math
import random

import numpy as np
import torch

from paper_2206_02255_gb300 import ask, inputs


def listed():
    return [
        # The smallest request of the served workload: an image of 256 x 256
        # near the boundary.  Launches and one orbit's latency decide.
        dict(name="frame_256", kind="frame", n=256, max_dwell=512, spot="17", zoom=40.0,
             g=2, r=4, B=8),
        # The paper's smallest map (n = 1024, dwell 512, its g=16 r=2 B=32).
        dict(name="frame_1024", kind="frame", n=1024, max_dwell=512, spot="paper", zoom=1.0,
             g=16, r=2, B=32),
        # A frame of an interactive loop that may not allocate: odd side,
        # ragged regions, a zoom of some hundreds.
        dict(name="noalloc_1999", kind="noalloc", n=1999, max_dwell=1024, spot="405", zoom=300.0,
             g=16, r=4, B=8),
        # A served request of ordinary size: odd side, ragged regions,
        # dwell cap and zoom from the middle of their ranges.
        dict(name="frame_3001", kind="frame", n=3001, max_dwell=1777, spot="1033", zoom=60.0,
             g=24, r=4, B=8),
        # The headline map: n = 16384, dwell 2048 over the paper's window.
        dict(name="frame_16384", kind="frame", n=16384, max_dwell=2048, spot="paper", zoom=1.0,
             g=16, r=4, B=16),
        # The largest map the library takes (17.2 GB): n = 65536, dwell 4096.
        dict(name="frame_65536", kind="frame", n=65536, max_dwell=4096, spot="wide", zoom=1.0,
             g=32, r=2, B=16),
        # The headline map delivered to host memory, as a program that saves
        # or shows it needs it.
        dict(name="host_16384", kind="host", n=16384, max_dwell=2048, spot="paper", zoom=1.0,
             g=16, r=4, B=16),
        # A quarter of the batched workload: 64 frames, sides 512 to 8192,
        # zooms 1 to 1e4, dwell caps 256 to 8192.
        dict(name="batch_64", kind="batch", frames=64, n_min=512, n_max=8192, dwell_min=256,
             dwell_max=8192, r=4, B=8),
        # A page of previews rendered again and again: 12 small frames
        # captured as a CUDA graph.
        dict(name="graph_12", kind="graph", frames=12, n_min=256, n_max=1024, dwell_min=256,
             dwell_max=2048, r=4, B=8),
        # The plain map, every pixel computed: the check on a subdivided map.
        dict(name="exhaustive_4096", kind="exhaustive", n=4096, max_dwell=2048, spot="paper",
             zoom=1.0, block_x=16, block_y=16),
        # Deep zoom in binary64, where float-float's 48 bits are too few.
        dict(name="deep_f64_1024", kind="deep", n=1024, max_dwell=4096, spot="seahorse_2^-30",
             zoom=1.0, g=32, r=4, B=16, ff=False),
        # Deep zoom in float-float arithmetic, the fast option.
        dict(name="deep_ff_3000", kind="deep", n=3000, max_dwell=2048, spot="antenna_2^-20",
             zoom=1.0, g=64, r=4, B=8, ff=True),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(_log_uniform(rng, lo, hi)))))


def _any_spot(rng):
    """(spot, zoom): mostly a zoom on the boundary, else the whole set."""
    if rng.random() < 0.25:
        return rng.choice(["paper", "wide"]), 1.0
    # (single frames up to 500: a stored boundary pixel lies within 2e-3 of the
    # boundary, so a window of a wider zoom may hold nothing but one dwell; the
    # batches go to 1e4)
    return str(rng.randrange(2048)), round(_log_uniform(rng, 1.0, 500.0), 3)


def _grid_of(n, side):
    """Initial regions per axis for regions of about `side` pixels."""
    return max(1, min(64, -(-n // side)))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "noalloc", "host", "exhaustive",
                       "batch", "graph", "deep", "deep"])
    if kind in ("frame", "noalloc", "host"):
        n = _log_int(rng, 256, 4096 if kind == "noalloc" else 16384)
        spot, zoom = _any_spot(rng)
        md = _log_int(rng, 256, 8192 if n <= 8192 else 2048)
        r, B = rng.choice([2, 4, 4, 8]), rng.choice([8, 16, 32])
        g = _grid_of(n, rng.choice([64, 128, 256]))
        return dict(kind=kind, n=n, max_dwell=md, spot=spot, zoom=zoom, g=g, r=r, B=B)
    if kind == "exhaustive":
        n = _log_int(rng, 256, 4096)
        spot, zoom = _any_spot(rng)
        bx, by = rng.choice(inputs.BLOCK_SHAPES)
        return dict(kind=kind, n=n, max_dwell=_log_int(rng, 256, 4096), spot=spot, zoom=zoom,
                    block_x=bx, block_y=by)
    if kind in ("batch", "graph"):
        n_max = rng.choice([512, 1024, 2048] if kind == "graph" else [1024, 2048, 4096])
        return dict(kind=kind, frames=_log_int(rng, 2, 16 if kind == "graph" else 48), n_min=256,
                    n_max=n_max, dwell_min=256, dwell_max=rng.choice([1024, 2048, 4096, 8192]),
                    r=rng.choice([2, 4, 8]), B=rng.choice([8, 16]))
    ff = rng.random() < 0.5
    n = _log_int(rng, 256, 2048 if ff else 1024)
    # (below its own cap a spot's window may be all at the cap)
    spot, _, _, _, cap = rng.choice(inputs.DEEP_SPOTS)
    zoom = round(_log_uniform(rng, 1.0 / 64, 1.0), 5)
    return dict(kind=kind, n=n, max_dwell=rng.randint(cap, cap + cap // 2), spot=spot, zoom=zoom,
                g=_grid_of(n, rng.choice([32, 64])), r=rng.choice([2, 4]),
                B=rng.choice([8, 16, 32]), ff=ff)


def _spot_window(spot, zoom):
    if spot == "paper":
        return inputs.WINDOW_PAPER
    if spot == "wide":
        return inputs.WINDOW_WIDE
    for name, re0, im0, w, _ in inputs.DEEP_SPOTS:
        if name == spot:
            return (re0, re0 + w / zoom, im0, im0 + w / zoom)
    cr, ci = inputs.boundary_centers()[int(spot)]
    return (cr - 1.0 / zoom, cr + 1.0 / zoom, ci - 1.0 / zoom, ci + 1.0 / zoom)


def _window(case, seed):
    """The case's window, moved by up to 2% and scaled by up to 1% by the seed."""
    return _moved(_spot_window(case["spot"], case["zoom"]), random.Random(seed))


def _moved(window, rng):
    re0, re1, im0, im1 = window
    w, h = re1 - re0, im1 - im0
    cr = 0.5 * (re0 + re1) + w * rng.uniform(-0.02, 0.02)
    ci = 0.5 * (im0 + im1) + h * rng.uniform(-0.02, 0.02)
    k = 0.5 * rng.uniform(0.99, 1.01)
    return (cr - k * w, cr + k * w, ci - k * h, ci + k * h)


def _side(n):
    """Initial-region side of a batched frame."""
    return 128 if n <= 4096 else 256


def _frame_specs(case, seed):
    """The frames of a batch: sizes, places and dwell caps from the workload's
    own generator, each window moved by the seed."""
    rng = random.Random(seed)
    out = inputs.batch_frames(case["frames"], 0, sides=(case["n_min"], case["n_max"]),
                              dwells=(case["dwell_min"], case["dwell_max"]))
    for f in out:
        f.update(window=_moved(f["window"], rng), g=-(-f["n"] // _side(f["n"])), r=case["r"],
                 B=case["B"])
    return out


class _State:
    pass


def prepare(case, seed):
    """A context with its scratch reserved, the window, and the output buffers."""
    st = _State()
    st.kind = kind = case["kind"]
    st.ctx = ask.Context(0)
    if kind in ("batch", "graph"):
        st.frames = _frame_specs(case, seed)
        for f in st.frames:
            f["out"] = torch.empty((f["n"], f["n"]), dtype=torch.int32, device="cuda:0")
        if kind == "graph":
            st.graph = st.ctx.graph_batch(st.frames)
        return st
    n = case["n"]
    st.n, st.max_dwell = n, case["max_dwell"]
    st.window = _window(case, seed)
    if kind == "exhaustive":
        st.params = ask.make_params(block=(case["block_x"], case["block_y"]))
        st.ctx.reserve("exhaustive", n, st.params)
    else:
        flags = ask.FLAG_FLOAT_FLOAT if case.get("ff") else 0
        st.params = ask.make_params(case["g"], case["r"], case["B"], flags=flags)
        if kind != "noalloc":
            st.ctx.reserve("ask", n, ask.make_params(case["g"], case["r"], case["B"]))
    if kind == "host":
        st.out = torch.empty((n, n), dtype=torch.int32, pin_memory=True)
    else:
        st.out = torch.empty((n, n), dtype=torch.int32, device="cuda:0")
    return st


def run(st):
    if st.kind == "frame":
        return st.ctx.render("ask", st.window, st.n, st.max_dwell, st.params, out=st.out)
    if st.kind == "exhaustive":
        return st.ctx.render("exhaustive", st.window, st.n, st.max_dwell, st.params, out=st.out)
    if st.kind == "noalloc":
        return ask.render_noalloc(st.window, st.n, st.max_dwell, st.params, st.out)
    if st.kind == "host":
        return st.ctx.render_host("ask", st.window, st.n, st.max_dwell, st.params, out=st.out)
    if st.kind == "deep":
        return st.ctx.render64("ask", st.window, st.n, st.max_dwell, st.params, out=st.out)
    if st.kind == "graph":
        st.graph.launch()
    else:
        st.ctx.render_batch(st.frames)
    return [f["out"] for f in st.frames]


def exact(case, seed):
    """Dwells are whole numbers: there is no 64-bit value to be near to."""
    return None


_FLOPS_PER_UPDATE = 7  # three fused multiply-adds and one sum


def _mean_escaping_dwell(window, max_dwell, k=48):
    """Mean updates of the escaping points of a k x k sample of the window
    (points inside the set count as none: their updates are not a need)."""
    re = np.linspace(window[0], window[1], k)
    im = np.linspace(window[2], window[3], k)
    c = re[None, :] + 1j * im[:, None]
    z = np.zeros_like(c)
    d = np.zeros(c.shape)
    alive = np.ones(c.shape, dtype=bool)
    for _ in range(max_dwell):
        z[alive] = z[alive] * z[alive] + c[alive]
        d[alive] += 1
        alive &= np.abs(z) < 2
    return float(np.where(alive, 0.0, d).sum() / d.size)


def _work_frame(window, n, max_dwell, g):
    """Each output pixel written once; the updates of the pixels that no rule
    spares: all of them (g = 0), or the perimeters of the initial regions."""
    s0 = -(-n // g) if g else 0
    pixels = g * g * max(1, 4 * s0 - 4) if g else n * n
    ups = pixels * _mean_escaping_dwell(window, max_dwell)
    return 4.0 * n * n, _FLOPS_PER_UPDATE * ups


def work(case):
    if case["kind"] in ("batch", "graph"):
        parts = [_work_frame(f["window"], f["n"], min(f["max_dwell"], 512), f["g"])
                 for f in _frame_specs(case, 0)]
    else:
        parts = [_work_frame(_spot_window(case["spot"], case["zoom"]), case["n"],
                             case["max_dwell"], case.get("g", 0))]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
