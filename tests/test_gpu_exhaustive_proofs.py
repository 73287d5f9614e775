"""The dwell loop with proofs (exhaustive maps, tiled leaves, exact perimeters)
against the CPU reference: caps beside its block lengths and looks, windows
where proofs come early, late and never."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

CAPS = [1, 15, 16, 17, 31, 47, 48, 49, 79, 80, 81, 144, 145, 1000, 4097]
WINDOWS = [inputs.WINDOW_PAPER, (0.24, 0.26, -0.01, 0.01), (-0.76, -0.74, -0.01, 0.01),
           (-1.26, -1.24, -0.01, 0.01), (-2.05, -1.95, -0.05, 0.05), (0.28, 0.30, 0.56, 0.58)]


@pytest.mark.parametrize("md", CAPS)
def test_exhaustive_proofs(ctx, orc, asklib, md):
    for k, win in enumerate(WINDOWS):
        n = 120 + k
        want = orc.render_exhaustive(win, n, md)
        for flags in (0, asklib.FLAG_COUNT):
            out = ctx.render("exhaustive", win, n, md, asklib.make_params(flags=flags))
            got = out.cpu().numpy().view(np.uint32)
            assert np.array_equal(got, want), (win, md, int((got != want).sum()))
        ms, _ = orc.render_ms(win, n, md, 3, 2, 8)
        for flags in (asklib.FLAG_LEAF_TILED, asklib.FLAG_EXACT_BORDERS):
            out = ctx.render("ask", win, n, md, asklib.make_params(3, 2, 8, flags=flags))
            assert np.array_equal(out.cpu().numpy().view(np.uint32), ms), (win, md, flags)
