"""Perimeter queries: spread chunks, orbits proven to stay in the set, cheap
regions several to a ticket, children probed in parallel.  Maps and counts
against the CPU reference at the sizes and places where each can go wrong."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

# windows: the set; the main cardioid's cusp, its root points with the period-2
# and period-3 bulbs; the period-2 bulb's rim; wholly inside either; a window
# whose corner points have |c| near 2; far outside
WINDOWS = [
    inputs.WINDOW_PAPER, inputs.WINDOW_WIDE, (0.24, 0.26, -0.01, 0.01), (-0.76, -0.74, -0.01, 0.01),
    (-0.135, -0.115, 0.64, 0.66), (-1.26, -1.24, -0.01, 0.01), (-0.3, -0.1, -0.1, 0.1),
    (-1.05, -0.95, -0.05, 0.05), (-2.05, -1.95, -0.05, 0.05), (1.0, 2.2, 1.0, 2.2),
]
# (n, max_dwell, g, r, B): perimeters around 32 and 64 pixels (sides 9, 17, 18),
# one chunk and many, chunks of one perimeter longer than the rest, children
# more than 64 a region (r > 8), caps below and beside the block lengths, high
# caps (slow captures)
CASES = [
    (144, 4096, 16, 2, 4), (153, 2000, 9, 2, 9), (162, 129, 9, 3, 3), (200, 3000, 1, 2, 8),
    (255, 33, 2, 16, 4), (300, 31, 5, 4, 8), (96, 8191, 3, 12, 1), (64, 7, 4, 2, 1),
    (257, 32, 1, 64, 2), (180, 96, 20, 3, 2),
]


def _check(ctx, asklib, orc, win, n, md, g, r, B, flags):
    want, ost = orc.render_ms(win, n, md, g, r, B)
    out, st = ctx.render("ask", win, n, md, asklib.make_params(g, r, B, flags=flags), stats=True)
    got = out.cpu().numpy().view(np.uint32)
    assert np.array_equal(got, want), (win, n, md, g, r, B, int((got != want).sum()))
    for key in ("regions_per_level", "fills_per_level"):
        mine, ref = st[key], ost[key]  # (the reference lists no levels without regions)
        assert mine[:len(ref)] == ref and not any(mine[len(ref):]), key
    assert st["leaves"] == ost["leaves"]


@pytest.mark.parametrize("n,md,g,r,B", CASES)
@pytest.mark.parametrize("win", WINDOWS)
def test_queries_match_oracle(ctx, orc, asklib, win, n, md, g, r, B):
    _check(ctx, asklib, orc, win, n, md, g, r, B, 0)
    if n < 200:
        _check(ctx, asklib, orc, win, n, md, g, r, B, asklib.FLAG_COUNT)


def test_queries_in_a_batch_and_noalloc(ctx, orc, asklib):
    import torch
    specs = [(WINDOWS[k % len(WINDOWS)],) + CASES[k % len(CASES)] for k in range(3, 23)]
    frames = [dict(window=w, n=n, max_dwell=md, g=g, r=r, B=B,
                   out=torch.full((n, n), -1, dtype=torch.int32, device="cuda"))
              for w, n, md, g, r, B in specs]
    maps = [orc.render_ms(w, n, md, g, r, B)[0] for w, n, md, g, r, B in specs]
    for flags in (0, asklib.FLAG_PERSISTENT, asklib.FLAG_EXACT_BORDERS):
        ctx.render_batch(frames, flags=flags)
        for f, want in zip(frames, maps):
            assert np.array_equal(f["out"].cpu().numpy().view(np.uint32), want), (flags, f["n"])
            f["out"].fill_(-1)
    for f, want in zip(frames, maps):
        asklib.render_noalloc(f["window"], f["n"], f["max_dwell"],
                              asklib.make_params(f["g"], f["r"], f["B"]), f["out"])
        assert np.array_equal(f["out"].cpu().numpy().view(np.uint32), want), f["n"]


@pytest.mark.slow
def test_many_cheap_regions_to_a_ticket(ctx, orc, asklib):
    """Enough light regions that a ticket stands for several."""
    win, n, md, g, r, B = inputs.WINDOW_WIDE, 4099, 300, 64, 2, 4
    want, ost = orc.render_ms(win, n, md, g, r, B)
    out, st = ctx.render("ask", win, n, md, asklib.make_params(g, r, B), stats=True)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
    assert st["regions_per_level"] == ost["regions_per_level"]
    assert st["leaves"] == ost["leaves"]
