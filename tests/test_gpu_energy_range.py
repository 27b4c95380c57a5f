"""The energy sums the squares first and weights them once, where the sums stay in range: values on
either side of that range, and chains of zeros, against long double.  Each of n <= 20000 terms of one sign
carries at most six roundings and the summation tree 20 more: 26 x 1.1e-16 < 1e-14; 1e-13 is
asserted."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROE, HAR = 0, 1


def energy(y0, model, prec, bc, params, kappa2=0.0):
    import torch
    import paper_1412_0544_gb300 as rk
    dtype = torch.float32 if prec else torch.float64
    h = rk.rk4_chain_create(model, prec, y0.shape[0], 0.01, bc, params)
    try:
        if kappa2:
            rk.rk4_chain_set_coupling2(h, kappa2)
        st = torch.from_numpy(y0).to(dtype).cuda()
        cp = torch.zeros_like(st) if prec else None
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        return rk.rk4_chain_energy(h, st, cp, ws)[0]
    finally:
        rk.rk4_chain_destroy(h)


def exact(y0, model, bc, kappa, w2, kappa2):
    y = y0.astype(np.longdouble)
    if model == ROE:
        return float(np.sum(y ** 2) / 2)
    q, p = y[:, 0], y[:, 1]
    e = np.sum(p ** 2) / 2 + np.longdouble(w2) * np.sum(q ** 2) / 2
    for r, k in ((1, kappa), (2, kappa2)):
        if k:
            ext = np.concatenate([q[-r:], q, q[:r]]) if bc == 0 else np.concatenate([np.zeros(r), q, np.zeros(r)])
            d = ext[r:] - ext[:-r]
            e += np.longdouble(k) * np.sum((d[r:] if bc == 0 else d) ** 2) / 2
    return float(e)


@pytest.mark.parametrize("model,prec", [(ROE, 0), (HAR, 0), (HAR, 1)])
@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 20000])
def test_ordinary_and_zero_values(model, prec, bc, n):
    rng = np.random.default_rng(5)
    y0 = rng.uniform(-1, 1, (n, 3 if model == ROE else 2)).astype(np.float32 if prec else np.float64)
    y0[n // 3: 2 * n // 3] = 0.0
    for k2 in (0.0, 0.5):
        if model == ROE and k2:
            continue
        got = energy(y0, model, prec, bc, dict(kappa=1.3, omega0=0.9), k2)
        assert got == pytest.approx(exact(y0, model, bc, 1.3, 0.9 * 0.9, k2), rel=1e-13)


@pytest.mark.parametrize("scale,omega0", [(1e-160, 1e20), (1e-130, 1.0), (1e120, 1.0), (1e150, 1e-10)])
def test_out_of_range_values(scale, omega0):
    n = 3000
    y0 = np.random.default_rng(6).uniform(-1, 1, (n, 2)) * scale
    y0[: n // 2, 1] = 0.0
    got = energy(y0, HAR, 0, 1, dict(kappa=0.0, omega0=omega0))
    assert got == pytest.approx(exact(y0, HAR, 1, 0.0, omega0 * omega0, 0.0), rel=1e-13)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_is_reported(bad):
    import paper_1412_0544_gb300 as rk
    y0 = np.ones((4000, 2))
    y0[3777, 1] = bad
    with pytest.raises(rk.RK4Error):
        energy(y0, HAR, 0, 0, None)
