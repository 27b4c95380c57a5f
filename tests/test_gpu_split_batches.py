"""A batch chain's FP64 result does not depend on the chains it shares launches, tiles or flags with: one
chain leaving the split form's range (for the FP64 form) changes no bit of the others, in full tiles, in
packed tiles and in the one-stage-per-launch scheme."""
import numpy as np
import pytest

import chain_inputs as ci

pytestmark = pytest.mark.gpu

ROE, HAR = 0, 1
STAGED, BLOCKED, PERSISTENT = 1, 2, 3
SCHEMES = [(STAGED, None), (BLOCKED, (256, 4, 1)), (BLOCKED, (128, 8, 4)), (BLOCKED, (256, 2, 3)), (BLOCKED, (512, 4, 8)),
           (BLOCKED, (256, 1, 2)), (PERSISTENT, (128, 4, 4)), (PERSISTENT, (256, 1, 1))]
LENGTHS = np.array([3000, 40, 7, 2100, 33, 64, 1, 500, 12, 90], dtype=np.int64)


@pytest.mark.parametrize("kernel,tiling", SCHEMES)
@pytest.mark.parametrize("model,value", [(ROE, 1e-120), (ROE, 1e4), (ROE, np.nan), (HAR, 1e-120), (HAR, 1e14), (HAR, np.nan)])
def test_other_chains_keep_their_bits(kernel, tiling, model, value):
    import torch
    import paper_1412_0544_gb300 as rk
    m = len(LENGTHS)
    off = np.concatenate(([0], np.cumsum(LENGTHS)))
    D = 3 if model == ROE else 2
    kappas, bcs = np.linspace(0.4, 1.6, m), (np.arange(m) % 2).astype(np.int8)
    y0 = ci.uniform_state(int(LENGTHS.sum()), D, seed=1260)
    h = rk.rk4_batch_create(model, rk.RK4_FP64, LENGTHS, kappas, bcs, 0.01)
    rk.rk4_chain_set_kernel(h, kernel)
    if tiling:
        rk.rk4_chain_set_tiling(h, *tiling)
    ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")

    def run(y):
        st = torch.from_numpy(y.copy()).cuda()
        rk.rk4_chain_integrate(h, st, None, ws, 9)
        status = rk.rk4_chain_status(h, ws)
        return st.cpu().numpy(), status

    want, status = run(y0)
    assert status == rk.RK4_OK
    for out in ([1], [3], [2, 4, 8], [0, 9]):  # chains that leave the range
        y = y0.copy()
        for c in out:
            y[off[c] + LENGTHS[c] // 2, 1] = value  # enters linearly
        got, status = run(y)
        assert status == (rk.RK4_ENONFINITE if np.isnan(value) else rk.RK4_OK)
        for c in range(m):
            same = np.array_equal(got[off[c]:off[c + 1]], want[off[c]:off[c + 1]])
            assert same == (c not in out), (out, c)
    rk.rk4_chain_destroy(h)
