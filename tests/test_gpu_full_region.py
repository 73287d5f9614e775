"""A uniform region of 65536 x 65536, whose pixel count does not fit 32 bits, is
filled and counted like any other."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.slow
def test_uniform_region_of_2_to_the_32_pixels(ctx, asklib):
    import torch
    n, win = 65536, (10.0, 11.0, 10.0, 11.0)   # every point escapes at once
    out = torch.zeros((n, n), dtype=torch.int32, device="cuda")
    frame = dict(window=win, n=n, max_dwell=50, g=1, r=2, B=16, out=out)
    for go in (lambda: ctx.render("ask", win, n, 50, asklib.make_params(1, 2, 16, flags=asklib.FLAG_COUNT),
                                  out=out, stats=True)[1],
               lambda: ctx.render_batch([frame], flags=asklib.FLAG_COUNT, stats=True),
               lambda: ctx.render_batch([frame], flags=asklib.FLAG_PERSISTENT, stats=True)):
        out.zero_()
        st = go()
        assert int(out.min()) == int(out.max()) == 1
        assert st["fills_per_level"][0] == 1 and st["leaves"] == 0
        assert st["ms_total"] < 100.0   # over the whole GPU, not by one warp
        if st["fill_pixels"] or st["border_pixels"]:   # counted
            assert st["fill_pixels"] == n * n
            assert st["deferred_fill_pixels"] == n * n
