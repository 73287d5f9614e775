"""Perimeters that hold both points of |c| >= 2 and points of the set: the query
ends with the first escape, not with the orbits that stay.  The updates that a
level counts, and the maps, against the CPU reference."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

CAP = 200000
# (window, n, g, r, B): one region in chunks, four, one CTA a region, and more
# regions of 16 x 16 than that (one orbit a lane)
CASES = [((-2.5, -0.5, -1.0, 1.0), 512, 1, 2, 256), ((-2.0, 2.0, -2.0, 2.0), 400, 2, 2, 200),
         ((-2.5, 1.5, -2.0, 2.0), 64, 4, 2, 16), ((-24.5, 23.5, -24.3, 23.7), 768, 48, 2, 16),
         ((-0.001, 8.0, -0.001, 8.0), 1100, 1, 2, 550)]


@pytest.mark.parametrize("win,n,g,r,B", CASES)
def test_first_escape_ends_the_query(ctx, orc, asklib, win, n, g, r, B):
    # (the reference's own map, at a cap that the CPU can run)
    want, ost = orc.render_ms(win, n, 300, g, r, B)
    p = asklib.make_params(g, r, B, flags=asklib.FLAG_COUNT)
    out, st = ctx.render("ask", win, n, 300, p, stats=True)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
    assert st["fills_per_level"][:1] == ost["fills_per_level"][:1]
    st = ctx.render("ask", win, n, CAP, p, out=out, stats=True)[1]
    border = (4 * (n // g) - 4) * g * g
    # (the first rounds of a query are of 8 updates, of one with a large perimeter 64)
    assert st["iterations_per_level"][0] <= 64 * border
    frame = dict(window=win, n=n, max_dwell=300, g=g, r=r, B=B, out=out)
    for flags in (0, asklib.FLAG_PERSISTENT):
        out.fill_(-1)
        ctx.render_batch([frame], flags=flags)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), want), flags
