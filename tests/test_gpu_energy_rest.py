"""The energy of states with components that are zero throughout (a chain released at rest, a uniform one, a
pulse): in one pass like any other, and right beside values whose squares underflow.

Tolerance as in test_gpu_energy_range.py (26 roundings of terms of one sign < 1e-14): 1e-13.  Time: the term
by term pass took such a state 2.1 times a random one's (2^22 sites); 1.5 is asserted of medians."""
import numpy as np
import pytest

from test_gpu_energy_range import ROE, HAR, energy, exact

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [0, 1])
@pytest.mark.parametrize("kappa2", [0.0, 0.5])
@pytest.mark.parametrize("kind", ["rest", "uniform", "pulse", "zero", "tiny"])
def test_values(bc, kappa2, kind):
    n = 5001
    y0 = np.random.default_rng(7).uniform(-1, 1, (n, 2))
    omega0 = 0.9
    if kind == "rest":
        y0[:, 1] = 0.0
    elif kind == "uniform":
        y0[:] = (0.5, -0.25)
    elif kind == "pulse":
        y0[:] = 0.0
        y0[1234] = (1.0, 0.5)
    elif kind == "zero":
        y0[:] = -0.0
    else:  # the squares of q underflow, but not their weight times them
        y0 *= (1e-170, 0.0)
        omega0 = 1e30
    got = energy(y0, HAR, 0, bc, dict(kappa=1.3, omega0=omega0), kappa2)
    assert got == pytest.approx(exact(y0, HAR, bc, 1.3, omega0 * omega0, kappa2), rel=1e-13, abs=0.0)


@pytest.mark.parametrize("model,prec", [(ROE, 0), (HAR, 0), (HAR, 1)])
def test_time(model, prec):
    import torch
    import paper_1412_0544_gb300 as rk
    n, D = 1 << 22, 3 if model == ROE else 2
    h = rk.rk4_chain_create(model, prec, n, 0.01, 0)
    ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")

    def median(st):
        cp = torch.zeros_like(st) if prec else None
        t = []
        for _ in range(25):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            rk.rk4_chain_energy(h, st, cp, ws)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        return float(np.median(t[5:]))

    random = torch.rand((n, D), dtype=torch.float32 if prec else torch.float64, device="cuda") + 0.5
    rest = random.clone()
    rest[:, 1] = 0.0
    pulse = torch.zeros_like(random)
    pulse[12345] = 1.0
    base = median(random)
    for name, st in (("at rest", rest), ("pulse", pulse)):
        r = median(st) / base
        print(f"model {model} precision {prec}: {name} takes {r:.2f} of a random state's time ({base * 1e3:.0f} us)")
        assert r <= 1.5
    rk.rk4_chain_destroy(h)
