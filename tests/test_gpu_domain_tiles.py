"""The tiles of a decomposed FP32 chain on either side of the lengths at which they change, bit for bit
against the undivided chain (state and Kahan compensation)."""
import numpy as np
import pytest

import chain_inputs as ci
from test_gpu_domain import HAR, PER, ROE, domain, rk, whole  # noqa: F401 (rk is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model", [ROE, HAR])
@pytest.mark.parametrize("n,ghost,tile", [((1 << 19) - 1, 64, (256, 4)), (1 << 19, 64, (128, 8)), ((1 << 19) + 3, 32, (128, 8)),
                                          (1 << 20, 16, (256, 4)), ((1 << 22) - 1, 64, (128, 8)), (1 << 22, 32, (128, 8)),
                                          ((1 << 22) + 1, 64, (256, 8))])
def test_tiles(rk, model, n, ghost, tile):  # noqa: F811
    d = rk.rk4_domain_create(model, 1, n, 0.01, PER, 4, ghost)
    t = rk.rk4_chain_get_tiling(rk.rk4_domain_chain(d))
    rk.rk4_domain_destroy(d)
    assert (t["block"], t["v"], t["k"]) == (*tile, ghost // 4)
    y0 = ci.uniform_state(n, 3 if model == ROE else 2, seed=1320).astype(np.float32)
    ref, rc, _ = whole(rk, y0, model, 1, PER, 35)
    got, gc, _ = domain(rk, y0, model, 1, PER, 4, ghost, 35)
    assert np.array_equal(got, ref)
    assert np.array_equal(gc, rc)
