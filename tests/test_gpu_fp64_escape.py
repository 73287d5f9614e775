"""Binary64 escape test by leading bits: points whose first states lie within,
across and beside the band around |z|^2 = 4 in which the exact test decides."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [2.0**-48, 1e-9, 1e-5, 6e-5, 1e-3])
@pytest.mark.parametrize("cr,ci", [(1.2, 1.6), (-1.6, 1.2), (-2.0, 0.0), (0.0, -2.0), (-2.0**0.5, 2.0**0.5)])
def test_escape_near_the_circle(ctx, orc, asklib, cr, ci, half):
    win = (cr - half, cr + half, ci - half, ci + half)
    n, md = 96, 200
    for method, want in (("ask", orc.render_ms(win, n, md, 4, 2, 4, fp64=True)[0]),
                         ("exhaustive", orc.render_exhaustive(win, n, md, fp64=True))):
        got = ctx.render64(method, win, n, md, asklib.make_params(4, 2, 4)).cpu().numpy().view(np.uint32)
        assert np.array_equal(got, want), (method, int((got != want).sum()))
