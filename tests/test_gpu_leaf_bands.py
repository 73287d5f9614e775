"""Leaves handed out as row bands (few leaves for the GPU's warps): maps and
counts against the CPU reference at the sizes where the cut can go wrong."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

# (n, max_dwell, g, r, B): one leaf, leaves of fewer rows than bands, ragged
# leaves, one wide leaf, leaves of one pixel, many leaves (no cut), caps below
# and at one block
CASES = [
    (1, 50, 1, 2, 1), (2, 50, 1, 2, 4), (7, 63, 1, 2, 8), (33, 64, 1, 2, 64), (97, 65, 3, 2, 32),
    (250, 300, 4, 2, 64), (513, 700, 2, 4, 256), (777, 1, 5, 3, 64), (1000, 40, 16, 2, 32),
    (256, 2048, 2, 2, 256), (200, 3001, 1, 2, 256),  # orbits that repeat themselves, to odd caps
    (1024, 512, 16, 2, 32), (1025, 129, 1, 2, 2048), (1200, 200, 300, 2, 4),
]


@pytest.mark.parametrize("exact", [False, True], ids=["query", "exact_borders"])
@pytest.mark.parametrize("n,md,g,r,B", CASES)
def test_leaf_bands_match_oracle(ctx, orc, asklib, n, md, g, r, B, exact):
    flags = asklib.FLAG_EXACT_BORDERS if exact else 0
    for win in (inputs.WINDOW_PAPER, (-2.1, 0.4, -0.2, 1.3)):
        want, ost = orc.render_ms(win, n, md, g, r, B)
        out, st = ctx.render("ask", win, n, md,
                             asklib.make_params(g, r, B, flags=flags | asklib.FLAG_COUNT), stats=True)
        got = out.cpu().numpy().view(np.uint32)
        assert np.array_equal(got, want), int((got != want).sum())
        assert st["leaves"] == ost["leaves"]
        out2 = ctx.render("ask", win, n, md, asklib.make_params(g, r, B, flags=flags))
        assert np.array_equal(out2.cpu().numpy().view(np.uint32), want)


def test_leaf_bands_in_a_batch(ctx, orc, asklib):
    import torch
    frames = [dict(window=inputs.WINDOW_PAPER, n=n, max_dwell=md, g=g, r=r, B=B,
                   out=torch.full((n, n), -1, dtype=torch.int32, device="cuda"))
              for n, md, g, r, B in CASES]
    for exact in (0, asklib.FLAG_EXACT_BORDERS):
        ctx.render_batch(frames, flags=exact)
        for f in frames:
            want, _ = orc.render_ms(f["window"], f["n"], f["max_dwell"], f["g"], f["r"], f["B"])
            assert np.array_equal(f["out"].cpu().numpy().view(np.uint32), want), f["n"]
            f["out"].fill_(-1)
