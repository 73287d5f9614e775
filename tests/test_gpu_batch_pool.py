"""Small batches pool their survivors for a second kernel; batches just above
the size do not; a full pool leaves the rest with their warps.  Maps against
the CPU reference and against the frames rendered alone."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu


def _frame(win, n, md, g, r, B):
    import torch
    return dict(window=win, n=n, max_dwell=md, g=g, r=r, B=B,
                out=torch.full((n, n), -1, dtype=torch.int32, device="cuda"))


@pytest.mark.parametrize("specs", [
    [(inputs.WINDOW_PAPER, 1, 50, 1, 2, 1)],
    [(inputs.WINDOW_PAPER, 64, 70, 1, 2, 64), ((0.28, 0.30, 0.56, 0.58), 65, 2000, 2, 2, 33)],
    [((-0.76, -0.74, 0.05, 0.07), 300, 3000, 3, 4, 8), (inputs.WINDOW_WIDE, 97, 40, 3, 2, 4),
     ((-2.05, -1.95, -0.05, 0.05), 150, 500, 5, 3, 16)],
], ids=["one_pixel", "one_leaf", "mixed"])
@pytest.mark.parametrize("exact", [False, True])
def test_pooled_batches(ctx, orc, asklib, specs, exact):
    import torch
    frames = [_frame(*s) for s in specs]
    flags = asklib.FLAG_EXACT_BORDERS if exact else 0
    wants = [orc.render_ms(*s)[0] for s in specs]
    graph = ctx.graph_batch(frames, flags=flags)
    for go in (lambda: ctx.render_batch(frames, flags=flags),
               lambda: ctx.render_batch(frames, flags=flags | asklib.FLAG_COUNT), graph.launch,
               graph.launch):
        for f in frames:
            f["out"].fill_(-1)
        go()
        torch.cuda.synchronize()
        for f, want in zip(frames, wants):
            assert np.array_equal(f["out"].cpu().numpy().view(np.uint32), want)
    graph.close()


def test_full_pool_and_no_pool(ctx, asklib):
    """Sixteen 1024 x 1024 frames all of whose pixels survive the pre-pass (16.8
    million survivors for 4.2 million pool entries), and the same with one
    frame more (too many pixels for a pool)."""
    import torch
    win = (-0.7436, -0.7430, 0.1310, 0.1316)
    want = ctx.render("ask", win, 1024, 700, asklib.make_params(1, 2, 1024))
    ex = ctx.render("exhaustive", win, 1024, 700)
    assert torch.equal(want, ex) and int((ex > 64).sum()) > 1 << 19
    for count in (16, 17):
        frames = [_frame(win, 1024, 700, 1, 2, 1024) for _ in range(count)]
        ctx.render_batch(frames)
        torch.cuda.synchronize()
        for f in frames:
            assert torch.equal(f["out"], want)
