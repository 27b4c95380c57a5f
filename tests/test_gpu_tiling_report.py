"""rk4_chain_get_tiling says what runs: the tiling that was set, else what the last integration's automatic
choice was, which set explicitly gives the same launches (and so the same bits even where tiles differ in
form: a state some of whose tiles run in the FP64 form)."""
import numpy as np
import pytest

import chain_inputs as ci

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,steps", [(1000, 100), (65537, 64), (300001, 7)])
def test_report(prec, n, steps):
    import torch
    import paper_1412_0544_gb300 as rk
    dtype = torch.float32 if prec else torch.float64
    y0 = ci.uniform_state(n, 3, seed=1280)
    y0[::1777, 1] = 1e-90
    y0 = torch.from_numpy(y0).to(dtype).cuda()

    def run(h):
        st = y0.clone()
        cp = torch.zeros_like(st) if prec else None
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        rk.rk4_chain_integrate(h, st, cp, ws, steps)
        torch.cuda.synchronize()
        return st

    h = rk.rk4_chain_create(0, prec, n, 0.01, 0)
    seed = rk.rk4_chain_get_tiling(h)
    want = run(h)
    ran = rk.rk4_chain_get_tiling(h)
    assert ran != seed and ran["G"] == ran["block"] * ran["v"] - 8 * ran["k"]
    rk.rk4_chain_set_tiling(h, 0)
    assert rk.rk4_chain_get_tiling(h) == seed
    rk.rk4_chain_set_tiling(h, ran["block"], ran["v"], ran["k"])
    assert rk.rk4_chain_get_tiling(h) == ran
    assert torch.equal(run(h), want)
    assert rk.rk4_chain_get_tiling(h) == ran
    rk.rk4_chain_destroy(h)


def test_report_of_a_domain():
    """The parts of a decomposed FP64 chain, which have no tiling set."""
    import torch
    import paper_1412_0544_gb300 as rk
    n = 1 << 20
    d = rk.rk4_domain_create(0, 0, n, 0.01, 0, 4, 32)
    h = rk.rk4_domain_chain(d)
    seed = rk.rk4_chain_get_tiling(h)
    rows, D = rk.rk4_domain_shape(d)
    c = torch.from_numpy(ci.uniform_state(n, 3, seed=1281)).cuda()
    st = torch.zeros((rows, D), dtype=torch.float64, device="cuda")
    ws = torch.empty(rk.rk4_domain_workspace_bytes(d), dtype=torch.uint8, device="cuda")
    rk.rk4_domain_scatter(d, c, None, st, None)
    rk.rk4_domain_integrate(d, st, None, ws, 100)
    torch.cuda.synchronize()
    assert rk.rk4_chain_get_tiling(h) != seed
    rk.rk4_domain_destroy(d)
