"""Leaves of the persistent batch kernel that are larger than an entry of its
leaf list: they go in as bands of rows.  Maps, leaf counts and pixel counts
against the CPU reference."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

# (window, n, max_dwell, g, r, B): leaves of 2^20 pixels (one entry), of a row
# more, of several bands with a short last one, four such leaves of a frame
SPECS = [(inputs.WINDOW_WIDE, 1024, 60, 1, 2, 1024), (inputs.WINDOW_WIDE, 1025, 60, 1, 2, 1025),
         (inputs.WINDOW_PAPER, 2051, 150, 1, 2, 1500), ((-1.8, 0.3, -0.9, 1.1), 2500, 90, 2, 2, 900)]


def test_leaves_in_bands(ctx, orc, asklib):
    import torch
    frames = [dict(window=w, n=n, max_dwell=md, g=g, r=r, B=B,
                   out=torch.full((n, n), -1, dtype=torch.int32, device="cuda"))
              for w, n, md, g, r, B in SPECS]
    wants = [orc.render_ms(*s) for s in SPECS]
    graph = ctx.graph_batch(frames, flags=asklib.FLAG_PERSISTENT)
    for k, go in enumerate([
            lambda: ctx.render_batch(frames, flags=asklib.FLAG_PERSISTENT, stats=True),
            lambda: ctx.render_batch(frames, flags=asklib.FLAG_PERSISTENT | asklib.FLAG_COUNT, stats=True),
            graph.launch]):
        for f in frames:
            f["out"].fill_(-1)
        st = go()
        torch.cuda.synchronize()
        for f, (want, _) in zip(frames, wants):
            assert np.array_equal(f["out"].cpu().numpy().view(np.uint32), want), (k, f["n"])
        if st is not None:
            assert st["leaves"] == sum(o["leaves"] for _, o in wants) == 7
        if k == 1:
            assert st["leaf_pixels"] == sum(s[1] ** 2 for s in SPECS)
    graph.close()
