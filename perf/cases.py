"""The work that users of this library have it do, as cases that can be timed one by one.

A case is one integration through the public entry points: a chain, a batch of chains or a
decomposed chain, its initial state already on the GPU, advanced by a number of RK4 steps in
place, as the README's example does it.  Sizes and options are those of the benchmark, the tests
and the paper (Roessler parameters a = 0.2, b = 1, c = 9, kappa = 1, dt = 0.01, uniform[-1, 1)
initial states), with odd lengths among them.
"""
import math

import numpy as np
import torch

import paper_1412_0544_gb300 as rk

DT = 0.01
A, B, C = 0.2, 1.0, 9.0
# Dormand and Prince (1980) RK5(4)7M, fifth-order weights, used with a fixed step
DOPRI5_A = [
    [0, 0, 0, 0, 0, 0, 0],
    [1 / 5, 0, 0, 0, 0, 0, 0],
    [3 / 40, 9 / 40, 0, 0, 0, 0, 0],
    [44 / 45, -56 / 15, 32 / 9, 0, 0, 0, 0],
    [19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729, 0, 0, 0],
    [9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656, 0, 0],
    [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0]]
DOPRI5_B = [35 / 384, 0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84, 0]
RK4_A = [[0, 0, 0, 0], [0.5, 0, 0, 0], [0, 0.5, 0, 0], [0, 0, 1.0, 0]]
RK4_B = [1 / 6, 1 / 3, 1 / 3, 1 / 6]


def _case(name, **kw):
    c = {"kind": "chain", "model": "roessler", "fp32": False, "n": 1000, "steps": 100, "fixed": False, "kappa": 1.0,
         "tune": "default"}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # A short chain followed step by step for its dynamics: one tile, so latency and launches
        # decide.  Handle defaults.
        _case("f64_tiny", n=1000, steps=100),
        # A medium chain with fixed ends in compensated single precision, handle defaults (the
        # parity tests' size plus one).
        _case("f32_small_fixed", fp32=True, n=65537, steps=256, fixed=True),
        # The paper's own benchmark (Sec. 3.2): 2^20 sites, 50 steps; both precisions, tuned first
        # as the README shows.
        _case("f64_paper", n=1 << 20, steps=50, tune="auto"),
        _case("f32_paper", fp32=True, n=1 << 20, steps=50, tune="auto"),
        # The long chains the library exists for, far larger than L2: FP64 with fixed ends at the
        # tiling the README's results were taken with, and FP32-Kahan, tuned.
        _case("f64_long_fixed", n=(1 << 24) - 3, steps=20, fixed=True, tune="256,4,2"),
        _case("f32_long", fp32=True, n=(1 << 25) + 1, steps=64, tune="auto"),
        # 4096 independent chains of 64 .. 65536 sites (a parameter scan): handle defaults in FP64,
        # tuned in FP32-Kahan.
        _case("batch_f64", kind="batch", n=4096, steps=16),
        _case("batch_f32", kind="batch", fp32=True, n=4096, steps=64, tune="auto"),
        # The Hamiltonian model with its energy monitored after the run.
        _case("harmonic_f64_energy", model="harmonic", n=(1 << 22) + 5, steps=32),
        # Another tableau and second neighbours: Dormand-Prince 5 with next-nearest coupling.
        _case("dopri5_nnn_f64", kind="generic", n=(1 << 20) + 7, steps=20, tune="auto", kappa2=0.5),
        # A heterogeneous chain (site-dependent parameters).
        _case("het_f64_fixed", kind="het", n=(1 << 21) - 1, steps=32, fixed=True),
        # One chain kept in four parts with ghost zones (several memories), handle defaults.
        _case("domain_f32", kind="domain", fp32=True, n=1 << 24, steps=64, parts=4, ghost=64),
    ]


def draw(rng):
    """A case of the same ranges: any kind, 1000 .. 2^24 sites, odd sizes included."""
    kind = rng.choice(["chain", "chain", "chain", "batch", "generic", "het", "domain"])
    fp32 = rng.random() < 0.5
    model = "harmonic" if rng.random() < 0.25 else "roessler"
    most = (1 << 30) if fp32 else (1 << 28)  # site-steps: below the longest listed case of the precision
    if kind == "generic":
        most //= 8
    if kind == "batch":
        n = int(round(math.exp(rng.uniform(math.log(64), math.log(4096)))))
        steps = rng.randint(8, 24 if not fp32 else 96)
        steps = max(2, min(steps, most // (n * 10000)))
    else:
        lo = 20000 if kind == "domain" else 1000
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(1 << 24)))))
        steps = max(2, min(rng.randint(16, 250), most // n))
    c = _case(None, kind=kind, model=model, fp32=fp32, n=n, steps=steps, fixed=rng.random() < 0.5,
              kappa=round(rng.uniform(0.5, 2.0), 6), tune=rng.choice(["default", "auto"]))
    if kind == "generic":
        c["kappa2"] = round(rng.uniform(0.1, 0.7), 6)
        c["tableau"] = rng.choice(["dopri5", "rk4"])
    if kind == "domain":
        c["parts"] = rng.randint(2, 6)
        c["ghost"] = rng.choice([16, 32, 64])
        c["tune"] = "default"
    return c


def _dim(case):
    return 3 if case["model"] == "roessler" else 2


def _batch(case):
    """Chain lengths, couplings and boundaries of a batch: a parameter scan fixed by the case."""
    rs = np.random.RandomState(case["n"])
    m = case["n"]
    lengths = np.clip(np.rint(np.exp(rs.uniform(np.log(64), np.log(65536), m))), 64, 65536).astype(np.int64)
    return lengths, rs.uniform(0.5, 2.0, m), (rs.random_sample(m) < 0.5).astype(np.int8)


def _sites(case):
    return int(_batch(case)[0].sum()) if case["kind"] == "batch" else case["n"]


def _initial(case, seed):
    """The initial state: i.i.d. uniform[-1, 1) components from the library's generator."""
    n, d = _sites(case), _dim(case)
    st = torch.empty((n, d), dtype=torch.float32 if case["fp32"] else torch.float64, device="cuda")
    rk.rk4_fill_uniform(st, n * d, 0x14120544 + 7919 * seed, 0, rk.RK4_FP32_KAHAN if case["fp32"] else rk.RK4_FP64)
    return st


def _site_params(case, seed, dtype):
    """Per-site parameters of a heterogeneous chain, spread around the paper's values."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((case["n"], 4), generator=g, dtype=torch.float64, device="cuda")
    if case["model"] == "roessler":
        p = torch.stack([0.15 + 0.1 * u[:, 0], 0.8 + 0.4 * u[:, 1], 8.0 + 2.0 * u[:, 2], 0.5 + 1.5 * u[:, 3]], dim=1)
    else:
        p = torch.stack([0.5 + u[:, 0], 0.5 + 1.5 * u[:, 3]], dim=1)
    return p.to(dtype).contiguous()


class _Domain:
    """A decomposed chain's handle, freed with the object."""

    def __init__(self, *args, **kw):
        self.d = rk.rk4_domain_create(*args, **kw)

    def __del__(self):
        rk.rk4_domain_destroy(self.d)


def prepare(case, seed):
    model = rk.RK4_ROESSLER if case["model"] == "roessler" else rk.RK4_HARMONIC
    prec = rk.RK4_FP32_KAHAN if case["fp32"] else rk.RK4_FP64
    bc = rk.RK4_FIXED if case["fixed"] else rk.RK4_PERIODIC
    params = {"kappa": case["kappa"]}
    st = _initial(case, seed)
    cp = torch.zeros_like(st) if case["fp32"] else None
    s = {"case": case, "st": st, "cp": cp}
    if case["kind"] == "domain":
        dom = _Domain(model, prec, case["n"], DT, bc, case["parts"], case["ghost"], params=params)
        rows, d = rk.rk4_domain_shape(dom.d)
        s["dom"] = dom
        s["dst"] = torch.zeros((rows, d), dtype=st.dtype, device="cuda")
        s["dcp"] = torch.zeros_like(s["dst"]) if case["fp32"] else None
        s["ws"] = torch.empty(rk.rk4_domain_workspace_bytes(dom.d), dtype=torch.uint8, device="cuda")
        rk.rk4_domain_scatter(dom.d, st, cp, s["dst"], s["dcp"])
        return s
    if case["kind"] == "batch":
        lengths, kappas, bcs = _batch(case)
        ch = rk.Chain(lengths=lengths, kappas=kappas, bcs=bcs, model=model, precision=prec, dt=DT)
    else:
        ch = rk.Chain(case["n"], model=model, precision=prec, bc=bc, dt=DT, params=params)
    if case["kind"] == "generic":
        if case.get("tableau", "dopri5") == "dopri5":
            rk.rk4_chain_set_tableau(ch.h, DOPRI5_A, DOPRI5_B)
        rk.rk4_chain_set_coupling2(ch.h, case["kappa2"])
    if case["kind"] == "het":
        s["sp"] = _site_params(case, seed, st.dtype)
        rk.rk4_chain_set_site_params(ch.h, s["sp"])
    if case["tune"] == "auto":
        ch.autotune(st, cp)
    elif case["tune"] != "default":
        ch.set_tiling(*[int(x) for x in case["tune"].split(",")])
    s["chain"] = ch
    ch.workspace()
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "domain":
        d = s["dom"].d
        rk.rk4_domain_integrate(d, s["dst"], s["dcp"], s["ws"], case["steps"])
        rk.rk4_domain_gather(d, s["dst"], s["dcp"], s["st"], s["cp"])
        out = {"state": s["st"]}
    else:
        s["chain"].integrate(s["st"], s["cp"], case["steps"])
        out = {"state": s["st"]}
        if case["model"] == "harmonic" and case["kind"] == "chain":
            out["energy"] = s["chain"].energy(s["st"], s["cp"])
    if case["fp32"]:
        out["comp"] = s["cp"]
    return out


def work(case):
    """State (and compensation, and site parameters) read and written once; the scheme's own
    operations per site and step (an FMA counts as two)."""
    n, d, es = _sites(case), _dim(case), 4 if case["fp32"] else 8
    nbytes = 2 * n * d * es * (2 if case["fp32"] else 1)
    if case["kind"] == "het":
        nbytes += n * (4 if d == 3 else 2) * es
    slope = 13 if d == 3 else 6
    if case["kind"] == "generic":
        slope += 4
        if case.get("tableau", "dopri5") == "dopri5":
            per = 6 * slope + d * 2 * (15 + 5)
        else:
            per = 4 * slope + d * 2 * (3 + 4)
    else:
        per = 4 * slope + d * 2 * (3 + 4)
    return {"bytes": nbytes, "flops": n * case["steps"] * per}


def exact(case, seed):
    """The same integration in plain FP64 torch: Eqs. (3)-(5) stage by stage over the whole state."""
    y0 = _initial(case, seed).double()
    y = [y0[:, i].contiguous() for i in range(_dim(case))]
    n = y0.shape[0]
    if case["kind"] == "batch":
        lengths, kappas, bcs = _batch(case)
        first = torch.from_numpy(np.repeat(np.cumsum(lengths) - lengths, lengths)).cuda()
        size = torch.from_numpy(np.repeat(lengths, lengths)).cuda()
        fixed = torch.from_numpy(np.repeat(bcs, lengths)).cuda() != 0
        kappa = torch.from_numpy(np.repeat(kappas, lengths)).cuda()
        i = torch.arange(n, device="cuda") - first
        li, ri = first + (i - 1) % size, first + (i + 1) % size
        lm, rm = (~(fixed & (i == 0))).double(), (~(fixed & (i == size - 1))).double()

        def nb(x, r):
            return x[li] * lm + x[ri] * rm
    else:
        kappa = case["kappa"]

        def nb(x, r):
            s = torch.roll(x, r) + torch.roll(x, -r)
            if case["fixed"]:
                s[:r] -= torch.roll(x, r)[:r]
                s[-r:] -= torch.roll(x, -r)[-r:]
            return s
    a, b, c, w2 = A, B, C, 1.0
    if case["kind"] == "het":
        dtype = torch.float32 if case["fp32"] else torch.float64
        sp = _site_params(case, seed, dtype).double()
        if case["model"] == "roessler":
            a, b, c, kappa = (sp[:, i].contiguous() for i in range(4))
        else:
            w2, kappa = (sp[:, i].contiguous() for i in range(2))
    k2 = case.get("kappa2", 0.0)

    def slope(u):
        g = kappa * (nb(u[0], 1) - 2 * u[0])
        if k2:
            g = g + k2 * (nb(u[0], 2) - 2 * u[0])
        if case["model"] == "roessler":
            x, yy, z = u
            return [g - (yy + z), x + a * yy, b + z * (x - c)]
        return [u[1], g - w2 * u[0]]

    ta, tb = RK4_A, RK4_B
    if case["kind"] == "generic" and case.get("tableau", "dopri5") == "dopri5":
        ta, tb = DOPRI5_A, DOPRI5_B
    for _ in range(case["steps"]):
        ks = []
        for j in range(len(tb)):
            if not tb[j] and not any(row[j] for row in ta):
                continue
            u = [v.clone() for v in y]
            for m in range(j):
                if ta[j][m]:
                    for i, v in enumerate(u):
                        v.add_(ks[m][i], alpha=ta[j][m] * DT)
            ks.append(slope(u))
        for i, v in enumerate(y):
            inc = sum(tb[m] * ks[m][i] for m in range(len(ks)) if tb[m])
            v.add_(inc, alpha=DT)
    out = {"state": torch.stack(y, dim=1)}
    if case["model"] == "harmonic" and case["kind"] == "chain":
        # the energy of the state the library returns differs from this one by its rounding
        q, p = y
        dq = torch.roll(q, -1) - q
        if case["fixed"]:
            dq[-1] = -q[-1]
        e = 0.5 * (p * p + q * q).sum() + 0.5 * case["kappa"] * (dq * dq).sum()
        if case["fixed"]:
            e = e + 0.5 * case["kappa"] * q[0] * q[0]
        out["energy"] = e.reshape(1)
    if case["fp32"]:
        out["comp"] = None
    return out
