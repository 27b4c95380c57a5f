"""The automatic tiling (a choice by sites and steps) and the split of the steps into launches,
against the seed tiling set explicitly: the same scheme whatever the tiles, so bit for bit, state
and Kahan compensation."""
import numpy as np
import pytest

import chain_inputs as ci

pytestmark = pytest.mark.gpu

PER, FIX = 0, 1
ROE, HAR = 0, 1
STAGED, BLOCKED, PERSISTENT = 1, 2, 3
STEPS = (1, 2, 3, 7, 16, 17, 31, 50)


@pytest.fixture(scope="module")
def gh():
    import gpu_helpers
    return gpu_helpers


def same(a, b):
    assert np.array_equal(a[0], b[0])
    assert (a[1] is None) == (b[1] is None)
    if a[1] is not None:
        assert np.array_equal(a[1], b[1])


@pytest.mark.parametrize("n", [1, 37, 1000, 16001, 65537, 300001])
@pytest.mark.parametrize("model", [ROE, HAR])
@pytest.mark.parametrize("prec", [0, 1])
def test_chain(gh, n, model, prec):
    y0 = ci.uniform_state(n, 3 if model == ROE else 2, seed=1200 + n)
    for s in STEPS if n <= 16001 else (1, 31, 50):
        kw = dict(model=model, precision=prec, bc=FIX if s % 2 else PER, nsteps=s, return_comp=True)
        same(gh.gpu_run(y0, kernel=BLOCKED, **kw), gh.gpu_run(y0, kernel=BLOCKED, tiling=(256, 4, 1), **kw))
        if n <= 1000:
            same(gh.gpu_run(y0, kernel=PERSISTENT, **kw), gh.gpu_run(y0, kernel=STAGED, **kw))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kernel", [BLOCKED, PERSISTENT])
def test_batch_calls_of_many_lengths(gh, kernel, prec):
    """One handle, calls of many lengths: the launches' k come from one set."""
    lens = np.array([5000, 3, 1023, 1, 4096, 777, 20000, 64], dtype=np.int64)
    y0 = ci.uniform_state(int(lens.sum()), 3, seed=1210)
    kw = dict(precision=prec, lengths=lens, kappas=np.linspace(0.5, 1.5, len(lens)),
              bcs=(np.arange(len(lens)) % 2).astype(np.int8), kernel=kernel, return_comp=True, chunks=list(STEPS))
    same(gh.gpu_run(y0, **kw), gh.gpu_run(y0, tiling=(256, 4, 1), **kw))


def run_more(n, prec, nsteps, *, tiling=None, het=False, tableau=False):
    import torch
    import bench
    import paper_1412_0544_gb300 as rk
    dtype = torch.float32 if prec else torch.float64
    h = rk.rk4_chain_create(ROE, prec, n, 0.01, PER)
    try:
        if het:
            g = np.random.default_rng(1220).uniform(size=(n, 4))
            sp = np.stack([.15 + .1 * g[:, 0], .8 + .4 * g[:, 1], 8 + 2 * g[:, 2], .5 + 1.5 * g[:, 3]], 1)
            d_sp = torch.from_numpy(sp).to(dtype).cuda()
            rk.rk4_chain_set_site_params(h, d_sp)
        else:
            if tableau:
                rk.rk4_chain_set_tableau(h, bench.DOPRI5_A, bench.DOPRI5_B)
            rk.rk4_chain_set_coupling2(h, 0.5)
        if tiling:
            rk.rk4_chain_set_tiling(h, *tiling)
        st = torch.from_numpy(ci.uniform_state(n, 3, seed=1221)).to(dtype).cuda()
        cp = torch.zeros_like(st) if prec else None
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        rk.rk4_chain_integrate(h, st, cp, ws, nsteps)
        torch.cuda.synchronize()
        assert rk.rk4_chain_status(h, ws) == rk.RK4_OK
        return st.double().cpu().numpy(), (cp.double().cpu().numpy() if prec else None)
    finally:
        rk.rk4_chain_destroy(h)


@pytest.mark.parametrize("n", [50, 5003, 200003])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("form", ["het", "rk4nnn", "dopri5nnn"])
def test_other_forms(n, prec, form):
    kw = dict(het=form == "het", tableau=form == "dopri5nnn")
    for s in (1, 7, 32):
        same(run_more(n, prec, s, **kw), run_more(n, prec, s, tiling=(128, 2, 1), **kw))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kernel", [BLOCKED, PERSISTENT])
def test_captured_batch_outlives_other_calls(kernel, prec):
    """A batch integration captured into the caller's graph after a call of another length, and
    replayed after a third: the tables it uploads are still the right ones."""
    import torch
    import paper_1412_0544_gb300 as rk
    dtype = torch.float32 if prec else torch.float64
    lens = np.array([900, 4000, 17, 2500], dtype=np.int64)
    N = int(lens.sum())
    y0 = torch.from_numpy(ci.uniform_state(N, 3, seed=1230)).to(dtype).cuda()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = rk.rk4_batch_create(ROE, prec, lens, np.ones(4), np.zeros(4, np.int8), 0.01, stream=s.cuda_stream)
        rk.rk4_chain_set_kernel(h, kernel)
        rk.rk4_chain_set_option(h, rk.RK4_OPT_GRAPHS, 0)
        st, zero = y0.clone(), torch.zeros_like(y0)
        cp = zero.clone() if prec else None
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")

        def reset():
            st.copy_(y0)
            if prec:
                cp.copy_(zero)

        def call(n):
            rk.rk4_chain_integrate(h, st, cp, ws, n)

        call(5)
        reset()
        call(23)
        s.synchronize()
        want = st.clone()
        call(4)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            call(23)
        call(9)
        reset()
        g.replay()
        s.synchronize()
        assert torch.equal(st, want)
        del g
        rk.rk4_chain_destroy(h)
