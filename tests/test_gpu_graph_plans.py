"""The cached graph of a batch against changes of the tiling: the automatic choice and a set tiling of
the same block, v and k divide the same steps differently (48 steps at k = 16: 16 + 16 + 4 x 4 and
16 + 16 + 8 + 8), so a graph of the one must not be replayed over the tables of the other.  The same
scheme whatever the tiles, so bit for bit."""
import numpy as np
import pytest

import chain_inputs as ci

pytestmark = pytest.mark.gpu

BLOCKED, PERSISTENT = 2, 3
SHAPES = {0: [(64, 1), (128, 1), (256, 1), (512, 1), (128, 2), (128, 4), (256, 4)],
          1: [(256, 1), (128, 2), (256, 2), (128, 4), (256, 4), (512, 4), (128, 8), (256, 8)]}


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kernel", [BLOCKED, PERSISTENT])
def test_automatic_and_set_tilings_take_turns(kernel, prec):
    import torch
    import paper_1412_0544_gb300 as rk
    lens = np.array([700, 4000, 17, 2500, 33, 1200, 64, 9], dtype=np.int64)
    kappas, bcs = np.linspace(0.5, 1.5, len(lens)), (np.arange(len(lens)) % 2).astype(np.int8)
    dtype = torch.float32 if prec else torch.float64
    y0 = torch.from_numpy(ci.uniform_state(int(lens.sum()), 3, seed=1240)).to(dtype).cuda()
    steps = 48

    def create():
        h = rk.rk4_batch_create(0, prec, lens, kappas, bcs, 0.01)
        rk.rk4_chain_set_kernel(h, kernel)
        return h

    h = create()
    st = y0.clone()
    cp = torch.zeros_like(st) if prec else None
    ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")

    def run():
        st.copy_(y0)
        if prec:
            cp.zero_()
        rk.rk4_chain_integrate(h, st, cp, ws, steps)
        assert rk.rk4_chain_status(h, ws) == rk.RK4_OK
        return st.clone()

    want = run()
    for block, v in SHAPES[prec]:
        for k in (1, 2, 4, 8, 16):
            try:
                rk.rk4_chain_set_tiling(h, block, v, k)
            except rk.RK4Error:
                continue  # too small a tile for k
            assert torch.equal(run(), want), (block, v, k)
            rk.rk4_chain_set_tiling(h, 0, 0, 0)
            assert torch.equal(run(), want), (block, v, k)
    rk.rk4_chain_destroy(h)
