"""Perimeters that lie on both sides of the limit of |c| above which an orbit is
tested at every update, with one dwell that is a multiple of the rounds'
length: uniform, whichever way each orbit runs.  Two columns of pixels beside
c = -1.99975, a hair above the real axis, against the CPU reference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

RE = (-1.999750018119812, -1.999749779701233)   # two float steps, the limit between the columns
RE64 = (-1.999725341796875, -1.9997253417968182)  # the same of binary64
IM16, IM32 = (1.8197008557763183e-06, 1.8215205273008905e-06), (2.2908676691746344e-11, 2.2931585449970093e-11)
IM16_64 = (2.0892961308540237e-06, 2.0897139900801943e-06)


def _check(render, want, ost, dwell):
    assert want.min() == want.max() == dwell and ost["fills_per_level"][0] == 1
    out, st = render()
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want)
    assert st["fills_per_level"][0] == 1 and st["subdivisions_per_level"][0] == 0


@pytest.mark.parametrize("kind", ["ask", "SBR", "MBR", "cdp2", "cdp2 MBR"])
@pytest.mark.parametrize("im,dwell", [(IM16, 16), (IM32, 32)])
def test_single(ctx, orc, asklib, kind, im, dwell):
    win = RE + im
    want, ost = orc.render_ms(win, 2, 300, 1, 2, 1)
    flags = sum(getattr(asklib, "FLAG_" + f) for f in kind.split() if f in ("SBR", "MBR"))
    method = "cdp2" if kind.startswith("cdp2") else "ask"
    p = asklib.make_params(1, 2, 1, (8, 4), flags)
    _check(lambda: ctx.render(method, win, 2, 300, p, stats=True), want, ost, dwell)


@pytest.mark.parametrize("ff", [False, True], ids=["f64", "ff"])
def test_wide(ctx, orc, asklib, ff):
    win = RE + IM16 if ff else RE64 + IM16_64
    want, ost = orc.render_ms(win, 2, 300, 1, 2, 1, fp64=True, flags=4 if ff else 0)
    p = asklib.make_params(1, 2, 1, flags=asklib.FLAG_FLOAT_FLOAT if ff else 0)
    _check(lambda: ctx.render64("ask", win, 2, 300, p, stats=True), want, ost, 16)
