"""Fronts that run into a chain at rest, where the split FP64 form's differences underflow: the results have
to be the FP64 form's, down to the smallest values, wherever the front lies in a tile (16 steps in one
launch reach 64 sites), and a state at rest has to stay in the split form.

Tolerance: as for the other states whose values span hundreds of decades (60 steps x 40 roundings of 2^-53,
amplified at most e^(60 x 0.05 x 4)), 1e-7 relative per site down to 1e-250."""
import numpy as np
import pytest

import closed_form as cf
import oracle
import oracle_pins as P

pytestmark = pytest.mark.gpu

PER, FIX = 0, 1
HAR = 1
STAGED, BLOCKED, PERSISTENT = 1, 2, 3
# interiors of 896, 1920, 384, 128 sites: fronts near 896 lie at a tile border or within a tile
TILINGS = [(256, 4, 16), (256, 8, 16), (128, 4, 16), (256, 1, 16)]
DISTANCES = (-2, 0, 5, 17, 20, 33, 60, 66, 90)


def check(got, ref, zero):
    assert np.all(got[zero] == 0.0)
    near = np.abs(ref) > 1e-250
    err = np.abs(got - ref)[near] / np.abs(ref)[near]
    assert np.max(err) <= 1e-7, (np.max(err), np.flatnonzero(near.reshape(-1))[np.argmax(err)])
    assert cf.rel_inf(got, ref) <= 1e-12


@pytest.fixture(scope="module")
def gh():
    import gpu_helpers
    return gpu_helpers


def pulse(n, site, amp):
    y0 = np.zeros((n, 2))
    y0[site] = (amp, 0.25 * amp)
    return y0


@pytest.mark.parametrize("amp", [1.0, 1e-20])
@pytest.mark.parametrize("dt,steps", [(0.01, 32), (2.0 ** -16, 32), (0.01, 9)])
@pytest.mark.parametrize("scheme", [(STAGED, None)] + [(BLOCKED, t) for t in TILINGS])
def test_front_beside_a_tile_border(gh, scheme, dt, steps, amp):
    kernel, tiling = scheme
    n = 4001
    for d in DISTANCES if kernel == BLOCKED else (0,):
        site = 896 - d
        y0 = pulse(n, site, amp)
        ref = oracle.rk4_integrate(y0, HAR, FIX, dt, steps)
        got = gh.gpu_run(y0, model=HAR, bc=FIX, dt=dt, nsteps=steps, kernel=kernel, tiling=tiling)
        check(got, ref, np.abs(np.arange(n) - site) > 4 * steps)


@pytest.mark.parametrize("kernel,tiling", [(BLOCKED, (256, 2, 16)), (PERSISTENT, (128, 4, 16)), (STAGED, None)])
def test_fronts_in_a_batch(gh, kernel, tiling):
    """Pulses in some chains of a batch, at rest the others, in full and packed tiles."""
    lengths = np.array([900, 100, 40, 300, 33, 2000, 150], dtype=np.int64)
    off = np.concatenate(([0], np.cumsum(lengths)))
    kappas, bcs = np.linspace(0.5, 1.5, 7), np.array([0, 1, 0, 1, 0, 1, 1], dtype=np.int8)
    y0 = np.zeros((int(lengths.sum()), 2))
    for c in (0, 1, 3, 6):
        y0[off[c] + lengths[c] // 3] = (1.0, 0.25)
    ref = oracle.batch_rk4_integrate(y0, lengths, kappas, bcs, model=HAR, nsteps=16)
    got = gh.gpu_run(y0, model=HAR, nsteps=16, lengths=lengths, kappas=kappas, bcs=bcs, kernel=kernel, tiling=tiling)
    check(got, ref, ref == 0.0)


@pytest.mark.parametrize("tiling", [None, (256, 2, 2), (128, 2, 3)])
@pytest.mark.parametrize("kappa2", [0.0, 0.6])
def test_generic_front(tiling, kappa2):
    import test_gpu_split as tgs
    A, b, _ = P.TABLEAUX["dopri5"]
    n, steps = 3001, 12
    prm = oracle.params(kappa=1.1, omega0=0.9, kappa2=kappa2)
    for site in range(1500, 1530, 7):
        y0 = pulse(n, site, 1.0)
        ref = oracle.rk_integrate(y0, A, b, HAR, FIX, 0.01, steps, prm)
        got = tgs.gen_run(y0, A, b, model=HAR, bc=FIX, nsteps=steps, kappa2=kappa2, kernel=BLOCKED if tiling else STAGED,
                          tiling=tiling)
        check(got, ref, np.abs(np.arange(n) - site) > 6 * (2 if kappa2 else 1) * steps)


@pytest.mark.parametrize("kernel,tiling", [(STAGED, None), (BLOCKED, (256, 4, 1)), (BLOCKED, (128, 4, 16)), (BLOCKED, (256, 1, 2))])
def test_states_at_rest_keep_the_split_form(gh, kernel, tiling):
    """Chains released at rest (all momenta zero), wholly at rest, and with a component that stays zero:
    bit for bit alike in every scheme, which the FP64 form of single tiles would not be."""
    import chain_inputs as ci
    n = 3001
    rest = ci.uniform_state(n, 2, seed=1270)
    rest[:, 1] = 0.0
    for y0, model, params in ((rest, HAR, {}), (np.zeros((n, 2)), HAR, {}), (np.ones((n, 2)) * [0.5, 0.0], HAR, dict(omega0=0.0)),
                              (np.zeros((n, 3)), 0, {}), (ci.uniform_state(n, 3, seed=1271) * [1, 1, 0], 0, dict(b=0.0))):
        want = gh.gpu_run(y0, model=model, nsteps=20, params=params, tiling=(256, 2, 4), kernel=BLOCKED)
        got = gh.gpu_run(y0, model=model, nsteps=20, params=params, kernel=kernel, tiling=tiling)
        assert np.array_equal(got, want)
