"""Deep-zoom leaves handed out as row bands and queried in rounds of 16, against
the CPU reference, in both arithmetics."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

# (n, max_dwell, g, r, B): one leaf, leaves of fewer rows than bands, of one
# pixel, ragged ones, caps below, at and beside the round length, regions of
# many perimeter groups, many leaves (no cut)
CASES = [(1, 20, 1, 2, 1), (5, 15, 1, 2, 8), (33, 16, 1, 2, 64), (64, 17, 2, 2, 64),
         (97, 300, 3, 2, 64), (150, 1024, 1, 3, 16), (200, 33, 50, 2, 2), (256, 1500, 4, 4, 64)]


@pytest.mark.parametrize("ff", [False, True], ids=["f64", "ff"])
@pytest.mark.parametrize("n,md,g,r,B", CASES)
def test_deep_leaf_bands(ctx, orc, asklib, n, md, g, r, B, ff):
    for win in (inputs.deep_window("spiral_2^-28")[0], (-0.76, -0.74, -0.01, 0.01),
                (-2.05, -1.95, -0.05, 0.05)):
        want, ost = orc.render_ms(win, n, md, g, r, B, fp64=True, flags=4 if ff else 0)
        for count in (0, asklib.FLAG_COUNT):
            flags = count | (asklib.FLAG_FLOAT_FLOAT if ff else 0)
            out, st = ctx.render64("ask", win, n, md, asklib.make_params(g, r, B, flags=flags), stats=True)
            got = out.cpu().numpy().view(np.uint32)
            assert np.array_equal(got, want), (win, int((got != want).sum()))
            assert st["leaves"] == ost["leaves"]
