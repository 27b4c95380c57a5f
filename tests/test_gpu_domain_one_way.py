"""Exchange periods of one launch each, in pairs over the caller's buffers and the workspace's copy:
bit for bit against the undivided chain for odd and even numbers of periods, with and without a rest,
through the graph (eight periods) and around it, in both precisions and with the wide tiles."""
import numpy as np
import pytest

import chain_inputs as ci
from test_gpu_domain import FIX, HAR, PER, ROE, domain, rk, whole  # noqa: F401 (rk is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ghost,tiling", [(4, (128, 2, 1)), (12, (128, 4, 3)), (20, (256, 2, 5))])
@pytest.mark.parametrize("nsteps", ["1p", "2p", "3p", "5p+1", "8p", "9p", "17p+2"])
def test_periods(rk, prec, ghost, tiling, nsteps):  # noqa: F811
    n, k = 6007, ghost // 4
    periods, rest = (nsteps.split("p+") + ["0"])[:2] if "+" in nsteps else (nsteps[:-1], "0")
    steps = int(periods) * k + min(int(rest), k - 1)
    y0 = ci.uniform_state(n, 3, seed=1300 + ghost)
    if prec:
        y0 = y0.astype(np.float32)
    bc = PER if prec else FIX
    ref, rc, _ = whole(rk, y0, ROE, prec, bc, steps)
    got, gc, _ = domain(rk, y0, ROE, prec, bc, 3, ghost, steps, tiling=tiling)
    assert np.array_equal(got, ref)
    if prec:
        assert np.array_equal(gc, rc)


@pytest.mark.parametrize("model", [ROE, HAR])
def test_wide_tiles(rk, model):  # noqa: F811
    n = (1 << 20) + 77
    y0 = ci.uniform_state(n, 3 if model == ROE else 2, seed=1310).astype(np.float32)
    ref, rc, _ = whole(rk, y0, model, 1, PER, 51)
    got, gc, _ = domain(rk, y0, model, 1, PER, 4, 64, 51)
    assert np.array_equal(got, ref)
    assert np.array_equal(gc, rc)
