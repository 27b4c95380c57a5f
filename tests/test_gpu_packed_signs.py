"""The packed FP32 forms hold some coordinates with the other sign: values on which that could
show (zeros of both signs, sums that cancel, infinities, NaN, the largest and the smallest floats)
against the scalar one-stage-per-launch kernel.  Rounding is symmetric, so the values are the same;
the bits too, NaN payloads aside, except for the sign of a zero that the input itself holds as -0."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROE, HAR = 0, 1
STAGED, BLOCKED, PERSISTENT = 1, 2, 3
F = np.finfo(np.float32)
ODD = [0.0, -0.0, 1.0, -1.0, F.max, -F.max, F.tiny, -F.tiny, 1e-45, np.inf, -np.inf, np.nan]


def run(y0, model, kernel, tiling, nsteps, bc, b):
    import torch
    import paper_1412_0544_gb300 as rk
    h = rk.rk4_chain_create(model, 1, y0.shape[0], 0.01, bc, dict(b=b))
    try:
        rk.rk4_chain_set_kernel(h, kernel)
        if tiling:
            rk.rk4_chain_set_tiling(h, *tiling)
        st = torch.from_numpy(y0).cuda()
        cp = torch.zeros_like(st)
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        rk.rk4_chain_integrate(h, st, cp, ws, nsteps)
        torch.cuda.synchronize()
        return st.cpu().numpy(), cp.cpu().numpy()
    finally:
        rk.rk4_chain_destroy(h)


@pytest.mark.parametrize("model", [ROE, HAR])
@pytest.mark.parametrize("kernel,tiling", [(BLOCKED, (128, 2, 2)), (BLOCKED, (256, 4, 3)), (BLOCKED, (128, 8, 4)),
                                           (PERSISTENT, (128, 4, 2))])
def test_odd_values(model, kernel, tiling):
    D = 3 if model == ROE else 2
    n = 2500
    y0 = np.random.default_rng(7).uniform(-1, 1, (n, D)).astype(np.float32)
    y0[:600] = 0.0
    for i, v in enumerate(ODD):
        y0[900 + 70 * i, i % D] = v
    for bc in (0, 1):
        want = run(y0, model, STAGED, None, 6, bc, 0.0)
        got = run(y0, model, kernel, tiling, 6, bc, 0.0)
        for g, w in zip(got, want):
            assert np.array_equal(g, w, equal_nan=True)


@pytest.mark.parametrize("model", [ROE, HAR])
@pytest.mark.parametrize("tiling", [(128, 2, 2), (256, 4, 3), (128, 8, 4)])
def test_rest_stays_positive_zero(model, tiling):
    y0 = np.zeros((1500, 3 if model == ROE else 2), dtype=np.float32)
    st, cp = run(y0, model, BLOCKED, tiling, 5, 1, 0.0)
    for a in (st, cp):
        assert not np.any(a) and not np.any(np.signbit(a))
