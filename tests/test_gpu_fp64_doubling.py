"""Binary64 blocks double x on its exponent: states with x = 0 (c = -1, c = i),
rows with ci = 0, rows whose ci is tiny, at or beside the limit below which
tested updates run, and points that escape at once, against the CPU reference."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

WINDOWS = [
    (-2.0, 2.0, -2.0, 2.0), (-1.5, -0.5, -0.5, 0.5), (-0.5, 0.5, 0.5, 1.5),
    (-2.0, 0.0, -2.0**-395, 2.0**-395), (-2.0, 0.0, -2.0**-398, 2.0**-398),
    (-2.0, 0.0, -2.0**-900, 2.0**-900), (-2.0, 0.5, -2.0**-1060, 2.0**-1060),
    (-2.0**-1040, 2.0**-1040, -2.0**-1040, 2.0**-1040), (1.0, 1.9, -0.3, 0.6),
    inputs.deep_window("seahorse_2^-30")[0],
]


@pytest.mark.parametrize("n,md,g,r,B", [(64, 1000, 4, 2, 4), (61, 47, 1, 2, 64)])
@pytest.mark.parametrize("win", WINDOWS)
def test_doubling_on_the_exponent(ctx, orc, asklib, win, n, md, g, r, B):
    for method, want in (("ask", orc.render_ms(win, n, md, g, r, B, fp64=True)[0]),
                         ("exhaustive", orc.render_exhaustive(win, n, md, fp64=True))):
        out = ctx.render64(method, win, n, md, asklib.make_params(g, r, B))
        got = out.cpu().numpy().view(np.uint32)
        assert np.array_equal(got, want), (method, int((got != want).sum()))
