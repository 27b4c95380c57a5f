"""The split FP64 step's error against long double, component by component, over the states and
coefficients it accepts and just beyond (where the FP64 form takes over): no larger than that of the FP64
form it replaces, whose operations (rk4_device.cuh, rk4_generic.cuh) are repeated here with one rounding each.

Tolerance: the ratio of two 2-norms over 20000 sites scatters by about 0.5 % (errors of either side are
sums of a few roundings); 1.01 is asserted.  Where the library runs the FP64 form both sides are the
same numbers but for double roundings of the long-double products (one in 2^11)."""
import numpy as np
import pytest

import chain_inputs as ci

pytestmark = pytest.mark.gpu

L = np.longdouble
N = 20000


def fma(a, b, c):
    return (L(a) * b + c).astype(np.float64)


def slope(u, p, one):
    """Slopes of a periodic Roessler chain; one: long double throughout, else the FP64 operations."""
    xl, xr = np.roll(u[0], 1), np.roll(u[0], -1)
    if one:
        return [p["kappa"] * (xl - 2 * u[0] + xr) - (u[1] + u[2]), u[0] + p["a"] * u[1], p["b"] + u[2] * (u[0] - p["c"])]
    return [fma(p["kappa"], fma(-2.0, u[0], xl + xr), -(u[1] + u[2])), fma(p["a"], u[1], u[0]),
            fma(u[2], u[0], fma(-p["c"], u[2], p["b"]))]


def rk4(y, p, dt, steps):
    """The state after `steps` steps in long double and in the FP64 form."""
    exact, plain = [v.astype(L) for v in y], [v.copy() for v in y]
    lp = {k: L(v) for k, v in p.items()}
    h = L(np.float64(dt))
    for _ in range(steps):
        ks, u = [], exact
        for w in (h / 2, h / 2, h, None):
            ks.append(slope(u, lp, True))
            if w is not None:
                u = [v + w * k for v, k in zip(exact, ks[-1])]
        exact = [v + h / 6 * (a + 2 * b + 2 * c + d) for v, a, b, c, d in zip(exact, *ks)]
        acc, u = plain, plain
        for j, w in enumerate((dt / 2, dt / 2, dt, None)):
            k = slope(u, p, False)
            acc = [fma(dt / 6 if j in (0, 3) else dt / 3, q, v) for q, v in zip(k, acc)]
            if w is not None:
                u = [fma(w, q, v) for q, v in zip(k, plain)]
        plain = acc
    return exact, plain


def check(got, exact, plain, what):
    for d in range(3):
        ours = float(np.sqrt(np.sum((got[:, d] - exact[d]) ** 2)))
        theirs = float(np.sqrt(np.sum((plain[d] - exact[d]) ** 2)))
        print(f"{what}: component {d}: {ours / theirs:.3f} of the FP64 form's error")
        assert ours <= 1.01 * theirs, (what, d)


# dt, c, kappa, amplitude of a uniform state: ordinary ones, the edges of the state's range (dt |x - c| = 1/4)
# and beyond, coefficients and dt at their limits and beyond
CASES = [(0.01, 9.0, 1.0, 1.0), (0.01, 9.0, 1.0, 15.9), (0.01, 9.0, 1.0, 20.0), (0.01, 9.0, 1.0, 40.0),
         (0.01, 9.0, 1.0, 100.0), (0.01, 9.0, 1.0, 1000.0), (0.01, 9.0, 1.0, 3e4), (0.01, 5.7, 2.0, 18.0),
         (0.0138, 9.0, 2.0, 9.0), (0.0138, 9.0, 2.0, 12.0), (0.05, 2.4, 0.6, 2.5), (0.0625, 2.0, 0.5, 1.9),
         (0.0625, 2.0, 0.5, 4.0), (0.07, 1.5, 0.4, 1.0), (0.125, 1.0, 0.25, 1.0), (1e-4, 1250.0, 300.0, 1200.0)]


@pytest.mark.parametrize("dt,c,kappa,amp,steps",
                         [(*case, steps) for case in CASES for steps in (1, 3)
                          if steps == 1 or case[3] != 3e4])  # from 3e4 on the third step overflows
def test_uniform_states(dt, c, kappa, amp, steps):
    import gpu_helpers as gh
    y0 = ci.uniform_state(N, 3, seed=1250) * amp
    p = dict(a=0.2, b=1.0, c=c, kappa=kappa)
    exact, plain = rk4([y0[:, d].copy() for d in range(3)], p, dt, steps)
    for tiling in [(256, 4, 2), (128, 1, 4)]:
        check(gh.gpu_run(y0, nsteps=steps, dt=dt, params=p, tiling=tiling), exact, plain, (dt, c, amp, steps, tiling))


@pytest.mark.parametrize("dt,c", [(0.01, 9.0), (0.0138, 9.0), (0.01, 5.7)])
def test_on_the_attractor(dt, c):
    import gpu_helpers as gh
    p = dict(a=0.2, b=1.0, c=c, kappa=1.0)
    y0 = gh.gpu_run(ci.uniform_state(N, 3, seed=1251), nsteps=6000, dt=dt, params=p)
    exact, plain = rk4([y0[:, d].copy() for d in range(3)], p, dt, 1)
    check(gh.gpu_run(y0, nsteps=1, dt=dt, params=p, tiling=(256, 4, 1)), exact, plain, (dt, c))


# ---- generic tableaux ---------------------------------------------------------------------------

def generic(y, A, b, p, k2, dt, steps):
    """As rk4(), any tableau, second neighbours; the FP64 form's operations as in rk4_generic.cuh."""
    s, h = len(b), L(np.float64(dt))
    lp = {k: L(v) for k, v in p.items()}

    def f(u, one):
        l1, l2 = np.roll(u[0], 1) + np.roll(u[0], -1), np.roll(u[0], 2) + np.roll(u[0], -2)
        if one:
            return [lp["kappa"] * (l1 - 2 * u[0]) + L(k2) * (l2 - 2 * u[0]) - (u[1] + u[2]), u[0] + lp["a"] * u[1],
                    lp["b"] + u[2] * (u[0] - lp["c"])]
        inner = -(u[1] + u[2])
        if k2:
            inner = fma(k2, fma(-2.0, u[0], l2), inner)
        return [fma(p["kappa"], fma(-2.0, u[0], l1), inner), fma(p["a"], u[1], u[0]),
                fma(u[2], u[0], fma(-p["c"], u[2], p["b"]))]

    exact, plain = [v.astype(L) for v in y], [v.copy() for v in y]
    for _ in range(steps):
        for one in (True, False):
            base, ks = (exact if one else plain), []
            for j in range(s):
                u = base
                for m in range(j):
                    if A[j, m]:
                        u = [v + L(A[j, m]) * h * q for v, q in zip(u, ks[m])] if one else \
                            [fma(A[j, m] * dt, q, v) for v, q in zip(u, ks[m])]
                ks.append(f(u, one))
            inc = [np.zeros_like(v) for v in base]
            for m in range(s):
                if b[m]:
                    inc = [v + L(b[m]) * h * q for v, q in zip(inc, ks[m])] if one else \
                          [fma(b[m] * dt, q, v) for v, q in zip(inc, ks[m])]
            out = [v + i for v, i in zip(base, inc)]
            if one:
                exact = out
            else:
                plain = out
    return exact, plain


def generic_gpu(y0, A, b, p, k2, dt, steps, tiling):
    import torch
    import paper_1412_0544_gb300 as rk
    h = rk.rk4_chain_create(rk.RK4_ROESSLER, rk.RK4_FP64, y0.shape[0], dt, rk.RK4_PERIODIC, p)
    try:
        rk.rk4_chain_set_tableau(h, A, b)
        rk.rk4_chain_set_coupling2(h, k2)
        rk.rk4_chain_set_tiling(h, *tiling)
        st = torch.from_numpy(np.ascontiguousarray(y0)).cuda()
        ws = torch.empty(rk.rk4_chain_workspace_bytes(h), dtype=torch.uint8, device="cuda")
        rk.rk4_chain_integrate(h, st, None, ws, steps)
        assert rk.rk4_chain_status(h, ws) == rk.RK4_OK
        return st.cpu().numpy()
    finally:
        rk.rk4_chain_destroy(h)


@pytest.mark.parametrize("name", ["dopri5", "rk4"])
@pytest.mark.parametrize("dt,c,kappa,kappa2,amp", [
    (0.01, 9.0, 1.1, 0.5, 1.0), (0.01, 9.0, 2.0, 0.7, 1.0), (0.01, 9.0, 1.0, 0.0, 1.0), (0.01, 9.0, 2.0, 0.7, 15.0),
    (0.01, 9.0, 1.1, 0.5, 40.0), (0.0138, 9.0, 2.0, 0.25, 1.0), (0.06, 2.0, 0.5, 0.02, 0.8)])
@pytest.mark.parametrize("steps", [1, 2])
def test_generic_tableaux(name, dt, c, kappa, kappa2, amp, steps):
    """Both forms round the state once a step here; the first order of the later slopes in FP64 and the
    remainders' pairs leave the split form between 0.9 and 1."""
    import oracle
    import oracle_pins as P
    A, b = (P.TABLEAUX["dopri5"][:2] if name == "dopri5" else (oracle.RK4_A, oracle.RK4_B))
    A, b = np.asarray(A, dtype=float), np.asarray(b, dtype=float)
    y0 = ci.uniform_state(N, 3, seed=1252) * amp
    p = dict(a=0.2, b=1.0, c=c, kappa=kappa)
    exact, plain = generic([y0[:, d].copy() for d in range(3)], A, b, p, kappa2, dt, steps)
    check(generic_gpu(y0, A, b, p, kappa2, dt, steps, (128, 2, 2)), exact, plain, (name, dt, kappa, kappa2, amp, steps))


def stretched(q):
    """A four-stage tableau whose rows cancel: sums of magnitudes 1 + 2 q and 1 + 4 q."""
    A = np.zeros((4, 4))
    A[1, 0], A[2, :2], A[3, :3] = 0.5, (-q, 0.5 + q), (q, -2 * q, 1 + q)
    return A, np.array([1, 2, 2, 1]) / 6


def fehlberg():
    A = np.zeros((6, 6))
    A[1, :1], A[2, :2], A[3, :3] = [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197]
    A[4, :4], A[5, :5] = [439 / 216, -8, 3680 / 513, -845 / 4104], [-8 / 27, 2, -3544 / 2565, 1859 / 4104, -11 / 40]
    return A, np.array([16 / 135, 0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55])


@pytest.mark.parametrize("tab", [stretched(0.02), stretched(2), stretched(10), stretched(40), fehlberg()],
                         ids=["near", "beyond", "far", "farther", "fehlberg"])
@pytest.mark.parametrize("amp", [1.0, 9.0])
def test_tableaux_about_the_limit(tab, amp):
    """Tableaux that the split form takes (the first and the last) and ones whose rows would multiply its
    pairs' errors (predicted there: 1.08, 3.9 and 8.7 in z at amplitude 9)."""
    y0 = ci.uniform_state(N, 3, seed=1253) * amp
    p = dict(a=0.2, b=1.0, c=9.0, kappa=1.5)
    exact, plain = generic([y0[:, d].copy() for d in range(3)], *tab, p, 0.3, 0.0138, 1)
    check(generic_gpu(y0, *tab, p, 0.3, 0.0138, 1, (128, 2, 1)), exact, plain, (tab[1].size, amp))
