"""A level with so many regions of the cheap kind (whose centre escapes within
the probe's 64 updates) that a ticket of its kernel stands for several: the
number of them is checked against what the kernel needs at any residency."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PROBE, TICKETS_PER_WARP, WARPS_PER_SM = 64, 4, 64


def test_tickets_of_several_regions(ctx, orc, asklib):
    import torch
    win, n, md, g, r, B = (0.42, 0.62, 0.2, 0.4), 3000, 300, 50, 2, 2
    want, ost, log = orc.render_ms(win, n, md, g, r, B, log=True)
    ex = orc.render_exhaustive(win, n, PROBE + 1)
    centre = ex[log["y0"] + log["h"] // 2, log["x0"] + log["w"] // 2]
    light = np.bincount(log["level"][centre <= PROBE], minlength=ost["levels"])
    warps = torch.cuda.get_device_properties(0).multi_processor_count * WARPS_PER_SM
    assert light.max() >= 2 * TICKETS_PER_WARP * warps   # else every ticket is of one region
    out, st = ctx.render("ask", win, n, md, asklib.make_params(g, r, B), stats=True)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
    for key in ("regions_per_level", "fills_per_level", "subdivisions_per_level", "leaves"):
        assert st[key] == ost[key], key
    frame = dict(window=win, n=n, max_dwell=md, g=g, r=r, B=B, out=torch.full_like(out, -1))
    st = ctx.render_batch([frame], stats=True)
    assert np.array_equal(frame["out"].cpu().numpy().view(np.uint32), want)
    assert st["regions_per_level"] == ost["regions_per_level"]
