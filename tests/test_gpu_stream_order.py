"""Renders of every kind queued on one stream and one context without a
synchronisation between them: ASK chains and batches directly after CDP2
renders, whose grids launch the rest of their work from the device and share
the context's tables and counters with what follows."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu


def test_chains_behind_device_launches(ctx, orc, asklib):
    import torch
    win, win2 = inputs.WINDOW_PAPER, (-0.8, -0.6, 0.05, 0.30)
    n, md, g, r, B = 700, 900, 4, 2, 8
    want = orc.render_ms(win, n, md, g, r, B)[0]
    want2, ost2 = orc.render_ms(win2, n, md, g, r, B)
    p = asklib.make_params(g, r, B, (16, 16))
    kinds = [0, asklib.FLAG_CDP2_FIRE_AND_FORGET, asklib.FLAG_MBR,
             asklib.FLAG_MBR | asklib.FLAG_CDP2_FIRE_AND_FORGET]
    q = [asklib.make_params(g, r, B, (16, 16), f) for f in kinds]

    def new():
        return torch.full((n, n), -1, dtype=torch.int32, device="cuda")

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx.render("cdp2", win, n, md, q[0], out=new())   # sets the device runtime's limits
        s.synchronize()
        outs = []
        for _ in range(3):
            for k in q:
                shared = new()   # written by the CDP2 render first, by the chain behind it then
                ctx.render("cdp2", win, n, md, k, out=shared)
                ctx.render("ask", win2, n, md, p, out=shared)
                outs.append((shared, want2))
                outs.append((ctx.render("cdp2", win2, n, md, k, out=new()), want2))
                frames = [dict(window=w, n=n, max_dwell=md, g=g, r=r, B=B, out=new()) for w in (win, win2)]
                ctx.render_batch(frames)
                outs += [(frames[0]["out"], want), (frames[1]["out"], want2)]
                outs.append((ctx.render("cdp2", win, n, md, k, out=new()), want))
                last = new()
                asklib.render_noalloc(win2, n, md, p, last, stream=s)
                outs.append((last, want2))
                outs.append((ctx.render("cdp2", win, n, md, k, out=new()), want))
        out, st = ctx.render("ask", win2, n, md, p, out=new(), stats=True)
    s.synchronize()
    ctx.check(s)
    for k, (o, w) in enumerate(outs + [(out, want2)]):
        assert np.array_equal(o.cpu().numpy().view(np.uint32), w), k
    L = ost2["levels"]
    assert st["regions_per_level"][:L] == ost2["regions_per_level"]
    assert st["fills_per_level"][:L] == ost2["fills_per_level"]
    assert st["leaves"] == ost2["leaves"]
