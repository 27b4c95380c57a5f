"""The split form of the FP64 step (float-pair differences, csrc/rk4_split.cuh) where it can go
wrong: values that leave its range (tiles then run in the FP64 form), exact zeros, coefficients
on either side of its limits, its conversions' corner cases, and its accuracy.

Tolerances.  Against the oracle 1e-12 as everywhere in FP64.  Where a chain's values span hundreds
of decades the error is taken site by site: one step has 4 stages of at most 10 roundings each of
2^-53, amplified at most (1 + dt |J|)^4 per step, so 60 steps at dt |J| <= 0.05 stay below
60 x 40 x 1.2e-16 x e^(60 x 0.05 x 4) ~ 5e-8 relative for a linear chain whose terms all have one
sign; 1e-7 is asserted."""
import numpy as np
import pytest

import chain_inputs as ci
import closed_form as cf
import oracle

pytestmark = pytest.mark.gpu

PER, FIX = 0, 1
ROE, HAR = 0, 1
STAGED, BLOCKED, PERSISTENT = 1, 2, 3
SCHEMES = [(STAGED, None), (BLOCKED, (256, 4, 1)), (BLOCKED, (128, 8, 16)), (BLOCKED, (256, 2, 3)),
           (BLOCKED, (256, 1, 2)), (BLOCKED, (512, 4, 8)), (PERSISTENT, (128, 4, 4))]


@pytest.fixture(scope="module")
def gh():
    import gpu_helpers
    return gpu_helpers


@pytest.mark.parametrize("kernel,tiling", SCHEMES)
def test_pulse_in_a_zero_chain(gh, kernel, tiling):
    """A displaced site in a harmonic chain at rest: the front decays over hundreds of decades
    (far below the pairs' range), and the sites it has not reached stay exactly zero."""
    n, site, steps = 4001, 2000, 24
    y0 = np.zeros((n, 2))
    y0[site] = (1.0, 0.25)
    ref = oracle.rk4_integrate(y0, HAR, FIX, 0.01, steps)
    got = gh.gpu_run(y0, model=HAR, bc=FIX, nsteps=steps, kernel=kernel, tiling=tiling)
    beyond = np.abs(np.arange(n) - site) > 4 * steps
    assert np.all(got[beyond] == 0.0)
    assert np.all(np.abs(got[ref == 0.0]) < 1e-300)
    near = np.abs(ref) > 1e-250
    assert np.max(np.abs(got - ref)[near] / np.abs(ref)[near]) <= 1e-7
    assert cf.rel_inf(got, ref) <= 1e-12


@pytest.mark.parametrize("kernel,tiling", SCHEMES)
@pytest.mark.parametrize("scale", [1e-300, 1e-30, 1e-12, 1e4, 1e30, 1e200])
def test_scaled_harmonic_chain(gh, kernel, tiling, scale):
    """The harmonic chain is linear: any scale of the state is a legitimate input."""
    y0 = ci.uniform_state(3001, 2, seed=1100) * scale
    ref = oracle.rk4_integrate(y0, HAR, PER, 0.01, 40)
    got = gh.gpu_run(y0, model=HAR, bc=PER, nsteps=40, kernel=kernel, tiling=tiling)
    assert cf.rel_inf(got, ref) <= 1e-12


@pytest.mark.parametrize("kernel,tiling", SCHEMES)
def test_some_sites_out_of_range(gh, kernel, tiling):
    """Roessler sites of magnitudes the pairs do not hold among ordinary ones, at tile interiors,
    tile ends and chain ends: finite results as the FP64 form gives them."""
    n = 5003
    y0 = ci.uniform_state(n, 3, seed=1101)
    for i, v in ((0, 1e-200), (700, 3e5), (1023, -2e5), (1024, 1e-90), (2500, 1e-310), (n - 1, 7e4)):
        y0[i, 1] = v  # y enters linearly
    ref = oracle.rk4_integrate(y0, ROE, PER, 0.01, 2)
    assert np.all(np.isfinite(ref))
    got = gh.gpu_run(y0, nsteps=2, kernel=kernel, tiling=tiling)
    assert cf.rel_inf(got, ref) <= 1e-12
    far = np.r_[300:600, 1500:2300, 3000:4800]  # beyond the cones of the large sites
    assert cf.rel_inf(got[far], ref[far]) <= 1e-12


@pytest.mark.parametrize("model", [ROE, HAR])
def test_zero_and_negative_zero(gh, model):
    """Zeros of both signs, powers of two and their neighbours as state values (the corner cases
    of the conversions), every scheme bit for bit alike."""
    D = 3 if model == ROE else 2
    vals = np.array([0.0, -0.0, 1.0, -1.0, np.nextafter(1, 2), np.nextafter(1, 0), 0.5, -2.0, 2.0 ** -40, 3e-9,
                     1 + 2.0 ** -24, -(1 + 2.0 ** -24 + 2.0 ** -52), 2 - 2.0 ** -52, 8.0])
    y0 = np.resize(vals, (2003, D))
    ref = oracle.rk4_integrate(y0, model, FIX, 0.01, 30)
    st = gh.gpu_run(y0, model=model, bc=FIX, nsteps=30, kernel=STAGED)
    assert cf.rel_inf(st, ref) <= 1e-12
    for kernel, tiling in SCHEMES[1:]:
        assert np.array_equal(gh.gpu_run(y0, model=model, bc=FIX, nsteps=30, kernel=kernel, tiling=tiling), st), tiling


@pytest.mark.parametrize("model,dt,params", [
    (ROE, 0.01, dict(kappa=3.125)), (ROE, 0.01, dict(kappa=3.2)), (ROE, 0.0138, dict(c=9.0)),
    (ROE, 0.014, dict(c=9.0)), (ROE, 0.01, dict(kappa=0.0)), (ROE, 0.01, dict(a=0.0, b=0.0)),
    (ROE, 2.0 ** -21, {}), (ROE, 2.0 ** -20, {}), (ROE, 0.01, dict(kappa=-1.0)),
    (HAR, 0.01, dict(kappa=19.0, omega0=8.8)), (HAR, 0.01, dict(kappa=20.0, omega0=8.8)),
    (HAR, 0.05, dict(kappa=1.0)), (HAR, 0.01, dict(kappa=1e-70)), (HAR, 0.01, dict(omega0=0.0))])
def test_limits_of_the_rule(gh, model, dt, params):
    """Coefficients at, and just beyond, the limits under which the split form is taken."""
    D = 3 if model == ROE else 2
    y0 = ci.uniform_state(2500, D, seed=1102)
    ref = oracle.rk4_integrate(y0, model, PER, dt, 40, oracle.params(**params))
    st = gh.gpu_run(y0, model=model, dt=dt, nsteps=40, params=params, kernel=STAGED)
    assert cf.rel_inf(st, ref) <= 1e-12
    for tiling in [(256, 4, 2), (128, 2, 4)]:
        assert np.array_equal(gh.gpu_run(y0, model=model, dt=dt, nsteps=40, params=params, tiling=tiling), st), tiling


def test_batch_with_one_chain_out_of_range(gh):
    """Each chain takes its own form, in full and in packed tiles."""
    lengths = np.array([3000, 40, 7, 2100, 33], dtype=np.int64)
    kappa = np.array([1.0, 0.7, 1.9, 0.0, 1.1])
    bcs = np.array([0, 1, 0, 1, 0], dtype=np.int8)
    y0 = ci.uniform_state(int(lengths.sum()), 3, seed=1103)
    off = np.concatenate(([0], np.cumsum(lengths)))
    y0[off[1] + 3, 1] = 1e-120
    y0[off[3] + 50, 1] = 2e5
    ref = oracle.batch_rk4_integrate(y0, lengths, kappa, bcs, nsteps=2)
    for kernel, tiling in SCHEMES:
        got = gh.gpu_run(y0, nsteps=2, lengths=lengths, kappas=kappa, bcs=bcs, kernel=kernel, tiling=tiling)
        for c in range(5):
            assert cf.rel_inf(got[off[c]:off[c + 1]], ref[off[c]:off[c + 1]]) <= 1e-12, (kernel, c)


@pytest.mark.parametrize("model", [ROE, HAR])
def test_more_accurate_than_the_fp64_form(gh, model):
    """Against a long-double integration the split form's error after 1, 20 and 200 steps is no
    larger than that of the FP64 form it replaces (the weighted slopes added to the state one by
    one, rk4_device.cuh), in each component (2-norms over 20000 sites; predicted ratio: one
    rounding of the state against four, 0.5)."""
    D = 3 if model == ROE else 2
    y0 = ci.uniform_state(20000, D, seed=1104)

    def steps(dtype, count):
        dt = dtype(np.float64(0.01))
        a, c = dtype(np.float64(0.2)), dtype(9)
        y = [y0[:, d].astype(dtype) for d in range(D)]

        def f(u):
            lap = np.roll(u[0], 1) - 2 * u[0] + np.roll(u[0], -1)
            if model == ROE:
                return [lap - (u[1] + u[2]), u[0] + a * u[1], 1 + u[2] * (u[0] - c)]
            return [u[1], lap - u[0]]

        for _ in range(count):
            k1 = f(y)
            k2 = f([v + dt / 2 * k for v, k in zip(y, k1)])
            k3 = f([v + dt / 2 * k for v, k in zip(y, k2)])
            k4 = f([v + dt * k for v, k in zip(y, k3)])
            y = [v + dt / 6 * p + dt / 3 * q + dt / 3 * r + dt / 6 * s for v, p, q, r, s in zip(y, k1, k2, k3, k4)]
        return y

    for count in (1, 20, 200):
        exact = steps(np.longdouble, count)
        plain = steps(np.float64, count)
        got = gh.gpu_run(y0, model=model, nsteps=count, tiling=(256, 4, 2))
        for d in range(D):
            ours = float(np.sqrt(np.sum((got[:, d] - exact[d]) ** 2)))
            theirs = float(np.sqrt(np.sum((plain[d] - exact[d]) ** 2)))
            print(f"model {model} component {d} after {count} steps: {ours / theirs:.2f} of the FP64 form's error")
            assert ours <= theirs


# ---- generic tableaux ---------------------------------------------------------------------------

import oracle_pins as P  # noqa: E402


def gen_run(y0, A, b, *, model=ROE, bc=PER, nsteps=10, kappa2=0.0, kernel=BLOCKED, tiling=None, dt=0.01):
    import torch
    import paper_1412_0544_gb300 as rk
    h = rk.rk4_chain_create(model, rk.RK4_FP64, y0.shape[0], dt, bc, dict(kappa=1.1, omega0=0.9))
    try:
        rk.rk4_chain_set_tableau(h, A, b)
        rk.rk4_chain_set_coupling2(h, kappa2)
        rk.rk4_chain_set_kernel(h, kernel)
        if tiling:
            rk.rk4_chain_set_tiling(h, *tiling)
        st = torch.from_numpy(np.ascontiguousarray(y0)).cuda()
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        rk.rk4_chain_integrate(h, st, None, ws, nsteps)
        assert rk.rk4_chain_status(h, ws) == rk.RK4_OK
        return st.cpu().numpy()
    finally:
        rk.rk4_chain_destroy(h)


GEN = [(STAGED, None), (BLOCKED, (64, 2, 1)), (BLOCKED, (256, 2, 4)), (BLOCKED, (128, 4, 3)), (BLOCKED, (256, 4, 8))]


@pytest.mark.parametrize("kernel,tiling", GEN)
@pytest.mark.parametrize("kappa2", [0.0, 0.6])
def test_generic_pulse_and_wide_values(kernel, tiling, kappa2):
    """The generic scheme's tiles outside the pairs' range, and the sites a pulse has not reached."""
    A, b, _ = P.TABLEAUX["dopri5"]
    n, site, steps = 3001, 1500, 9
    y0 = np.zeros((n, 2))
    y0[site] = (1.0, 0.25)
    prm = oracle.params(kappa=1.1, omega0=0.9, kappa2=kappa2)
    ref = oracle.rk_integrate(y0, A, b, HAR, FIX, 0.01, steps, prm)
    got = gen_run(y0, A, b, model=HAR, bc=FIX, nsteps=steps, kappa2=kappa2, kernel=kernel, tiling=tiling)
    reach = 6 * (2 if kappa2 else 1) * steps
    assert np.all(got[np.abs(np.arange(n) - site) > reach] == 0.0)
    assert cf.rel_inf(got, ref) <= 1e-12
    y0 = ci.uniform_state(n, 3, seed=1110)
    for i, v in ((0, 1e-200), (700, 3e5), (1100, 1e-90), (n - 1, 7e4)):
        y0[i, 1] = v
    ref = oracle.rk_integrate(y0, A, b, ROE, PER, 0.01, 1, prm)
    got = gen_run(y0, A, b, nsteps=1, kappa2=kappa2, kernel=kernel, tiling=tiling)
    assert cf.rel_inf(got, ref) <= 1e-12


@pytest.mark.parametrize("name", ["dopri5", "rk4"])
def test_generic_more_accurate_than_the_fp64_form(name):
    """Against long double, runs of 20 and 100 steps are no further off than the FP64 form the split
    form replaces (k_m summed with their weights, one addition to the state): both round the
    state once per step, so the ratio is 1 up to the sampling of 60000 values (0.4 %) and the other
    roundings of either side (after a single Dormand-Prince step from a random state the split
    form's are 5 % of the total, against long double; later steps damp them)."""
    A, b, _ = P.TABLEAUX["dopri5"] if name == "dopri5" else (oracle.RK4_A, oracle.RK4_B, 4)
    A, b = np.asarray(A, dtype=float), np.asarray(b, dtype=float)
    y0 = ci.uniform_state(20000, 3, seed=1111)

    def steps(dtype, count):
        dt, kap, k2, a, c = (dtype(np.float64(v)) for v in (0.01, 1.1, 0.5, 0.2, 9.0))
        y = [y0[:, d].astype(dtype) for d in range(3)]

        def f(u):
            lap = np.roll(u[0], 1) - 2 * u[0] + np.roll(u[0], -1)
            lap2 = np.roll(u[0], 2) - 2 * u[0] + np.roll(u[0], -2)
            return [kap * lap + (k2 * lap2 - (u[1] + u[2])), u[0] + a * u[1], 1 + u[2] * (u[0] - c)]

        for _ in range(count):
            ks = []
            for j in range(len(b)):
                u = [v.copy() for v in y]
                for m in range(j):
                    if A[j, m]:
                        u = [v + (dtype(A[j, m]) * dt) * k for v, k in zip(u, ks[m])]
                ks.append(f(u))
            y = [v + sum((dtype(b[m]) * dt) * ks[m][d] for m in range(len(b)) if b[m]) for d, v in enumerate(y)]
        return y

    for count in (20, 100):
        exact, plain = steps(np.longdouble, count), steps(np.float64, count)
        got = gen_run(y0, A, b, nsteps=count, kappa2=0.5, tiling=(128, 2, 2))
        ours = np.sqrt(sum(float(np.sum((got[:, d] - exact[d]) ** 2)) for d in range(3)))
        theirs = np.sqrt(sum(float(np.sum((plain[d] - exact[d]) ** 2)) for d in range(3)))
        print(f"{name} after {count} steps: {ours / theirs:.3f} of the FP64 form's error")
        assert ours <= 1.02 * theirs


@pytest.mark.parametrize("bc", [PER, FIX])
def test_nan_spreads_as_in_the_fp64_form(gh, bc):
    """One NaN site: after m steps exactly the sites within 4 m of it are NaN; a chain that is all
    NaN stays so and reports it."""
    import torch
    import paper_1412_0544_gb300 as rk
    n, site = 6007, 2900
    for start, steps in ((site, 3), (None, 7)):
        y0 = ci.uniform_state(n, 3, seed=1120)
        y0[slice(None) if start is None else start] = np.nan
        for kernel, tiling in SCHEMES:
            h = rk.rk4_chain_create(ROE, rk.RK4_FP64, n, 0.01, bc)
            rk.rk4_chain_set_kernel(h, kernel)
            if tiling:
                rk.rk4_chain_set_tiling(h, *tiling)
            st = torch.from_numpy(y0.copy()).cuda()
            ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
            rk.rk4_chain_integrate(h, st, None, ws, steps)
            assert rk.rk4_chain_status(h, ws) == rk.RK4_ENONFINITE
            rk.rk4_chain_destroy(h)
            nan = np.isnan(st.cpu().numpy()).any(axis=1)
            want = np.ones(n, bool) if start is None else np.abs(np.arange(n) - site) <= 4 * steps
            assert np.array_equal(nan, want), (kernel, tiling, start)
