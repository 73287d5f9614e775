"""Updates that proofs of staying spare: counted with the others (an orbit of
the set counts max_dwell), reported apart, so that what was run is known."""
import numpy as np
import pytest

from paper_2206_02255_gb300 import inputs

pytestmark = pytest.mark.gpu

INSIDE = (-0.15, 0.15, -0.15, 0.15)     # the main cardioid
OUTSIDE = (0.5, 0.9, 0.3, 0.7)
CAP = 100000


def _params(asklib, g=4, r=2, B=8, flags=0):
    return asklib.make_params(g, r, B, flags=flags | asklib.FLAG_COUNT)


@pytest.mark.parametrize("method", ["exhaustive", "ask", "cdp2"])
def test_long_orbits_are_not_run(ctx, asklib, method):
    n = 96
    out, st = ctx.render(method, INSIDE, n, CAP, _params(asklib), stats=True)
    assert int(out.min()) == CAP
    run = st["iterations"] - st["spared_iterations"]
    if method == "cdp2":                # its queries run every orbit to the cap
        assert st["spared_iterations"] == 0
        return
    pixels = n * n if method == "exhaustive" else st["border_pixels"]
    assert st["iterations"] == pixels * CAP
    # proofs are looked for after 64 and more updates, and found here by 2000
    assert 64 * pixels <= run <= 2000 * pixels
    if method == "ask":
        assert st["spared_iterations"] == sum(st["spared_iterations_per_level"]) + st["spared_leaf_iterations"]


def test_every_kernel_reports(ctx, asklib):
    """Counts as ever, and parts that add up, in leaves, batches (pooled, not
    pooled, persistent), exact borders and CDP2 leaves."""
    import torch
    win, n, md = (-0.3, 0.1, 0.2, 0.7), 400, 20000
    ex, est = ctx.render("exhaustive", win, n, md, _params(asklib), stats=True)
    assert 0 < est["spared_iterations"] < est["iterations"] == int(ex.to(torch.int64).sum())
    frame = dict(window=win, n=n, max_dwell=md, g=1, r=2, B=300, out=torch.empty_like(ex))
    for go in (lambda: ctx.render("ask", win, n, md, _params(asklib, 1, 2, 300), stats=True)[1],
               lambda: ctx.render_batch([frame], flags=asklib.FLAG_COUNT, stats=True),
               lambda: ctx.render_batch([frame], flags=asklib.FLAG_COUNT | asklib.FLAG_PERSISTENT, stats=True),
               lambda: ctx.render("cdp2", win, n, md, _params(asklib, 1, 2, 300), stats=True)[1]):
        st = go()
        assert 0 < st["spared_iterations"] < st["iterations"]
        if st["leaf_iterations"]:
            assert st["leaf_iterations"] == est["iterations"]     # one leaf, the whole map
            assert 0 < st["spared_leaf_iterations"] < st["leaf_iterations"]
            assert st["spared_iterations"] == (sum(st["spared_iterations_per_level"]) +
                                               st["spared_leaf_iterations"])
    _, st = ctx.render("ask", win, n, md, _params(asklib, 4, 2, 16, asklib.FLAG_EXACT_BORDERS), stats=True)
    assert 0 < st["spared_iterations_per_level"][-1] < st["iterations_per_level"][-1]


def test_nothing_spared(ctx, asklib):
    """No proofs outside the set, at caps below the first look, in the double
    precision kernels, or where nothing was counted."""
    for win, md in ((OUTSIDE, 5000), (INSIDE, 64)):
        for method in ("exhaustive", "ask", "cdp2"):
            _, st = ctx.render(method, win, 120, md, _params(asklib), stats=True)
            assert st["spared_iterations"] == 0 < st["iterations"], (win, method)
    _, st = ctx.render64("ask", INSIDE, 64, 3000, _params(asklib), stats=True)
    assert st["spared_iterations"] == 0 < st["iterations"]
    ctx.render("ask", INSIDE, 120, 5000, _params(asklib), stats=True)
    _, st = ctx.render("ask", INSIDE, 120, 5000, asklib.make_params(4, 2, 8), stats=True)
    assert st["spared_iterations"] == st["iterations"] == 0


def test_rate_of_run_updates_fits_the_pipe(ctx, asklib):
    """152 SMs x 128 lanes x 2.07 GHz / 4 instructions an update."""
    n, md = 4096, 2048
    p = asklib.make_params()
    _, st = ctx.render("exhaustive", inputs.WINDOW_PAPER, n, md, _params(asklib), stats=True)
    ms = min(ctx.render("exhaustive", inputs.WINDOW_PAPER, n, md, p, stats=True)[1]["ms_total"] for _ in range(5))
    assert (st["iterations"] - st["spared_iterations"]) / (ms / 1e3) < 10.07e12


def test_first_escape_in_batches(ctx, asklib):
    """Perimeters with points beyond |c| = 2 and points of the set, in batches:
    few updates are run, whatever the cap."""
    import torch
    for win, n, g in (((-2.5, -0.5, -1.0, 1.0), 512, 1), ((-2.0, 2.0, -2.0, 2.0), 400, 2)):
        frame = dict(window=win, n=n, max_dwell=200000, g=g, r=2, B=n // g,
                     out=torch.empty((n, n), dtype=torch.int32, device="cuda"))
        for flags in (0, asklib.FLAG_PERSISTENT):
            st = ctx.render_batch([frame], flags=flags | asklib.FLAG_COUNT, stats=True)
            run = st["iterations_per_level"][0] - st["spared_iterations_per_level"][0]
            assert run <= 64 * g * g * (4 * (n // g) - 4), (win, flags)
