"""The work that users have this framework do, as cases to be timed.

Each case is one call (or the short sequence of calls) that a program makes
through the public binding ``paper_2305_19768_gb300.qmc``:

* ``oneshot``: a small integral evaluated once from host buffers
  (``qmc_eval_jobs``), where set-up, launches and copies count;
* ``plan``: a resident plan run on the caller's stream into a device buffer
  (``qmc_plan_run``), the form every batched and repeated evaluation takes;
* ``adaptive``: the weighted ten-integral amplitude integrated to a requested
  accuracy at a set of kinematic points (``qmc_integrate``);
* ``mlp``: the lattice-sizing network trained on a batch and applied to
  another one (``Mlp.train``, ``Mlp.forward``).

Kinematics and the seeds of the lattice shifts come from the case's seed.
``exact`` restates the subtracted, eps-expanded sector integrands and their
lattice sums in plain FP64 torch, and the network in FP64 numpy.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_2305_19768_gb300 import qmc
from paper_2305_19768_gb300.inputs import workloads
from paper_2305_19768_gb300.inputs.lattice import lattice_for, lattice_sizes

DEVICE = "cuda"
MASK64 = (1 << 64) - 1
GAMMA = 0x9E3779B97F4A7C15

# integral -> (builder, lowest order, orders, physical region)
INTEGRALS = {
    "triangle": (workloads.triangle_massive, 0, 1, False),
    "box": (workloads.box_massless, -2, 3, False),
    "box_d2": (workloads.box_massless_d2, -2, 3, False),
    "double_box": (workloads.double_box_massless, -4, 5, False),
    "box_massive": (workloads.box_massive, 0, 1, True),
    "box_physical": (functools.partial(workloads.box_massless, deform=True), -2, 3, True),
}
# integral -> most evaluations (kinematic points x sectors x shifts x lattice
# points) of a drawn case; each costs less than the largest listed case
MOST_EVALS = {"triangle": 4e8, "box": 3e8, "box_d2": 3e7, "double_box": 1.5e8, "box_massive": 2.5e8,
              "box_physical": 8e7}


def listed():
    return [
        # the smallest call: one finite integral, pilot-sized lattice, host
        # buffers in and out
        dict(name="triangle_oneshot", kind="oneshot", integral="triangle", points=1, n=1009, shifts=16, mixed=False),
        # a precise one-loop integral at one Euclidean point
        dict(name="box_1e5", kind="plan", integral="box", points=1, n=100003, shifts=32, mixed=False),
        # many Euclidean points on a pilot lattice: short lattices, ragged tiles
        dict(name="box_points_1e3", kind="plan", integral="box", points=125, n=1009, shifts=16, mixed=False),
        # the two-loop integral on the default pilot lattice
        dict(name="double_box_1e4", kind="plan", integral="double_box", points=1, n=10007, shifts=16, mixed=False),
        # and on a production lattice (the largest case)
        dict(name="double_box_1e5", kind="plan", integral="double_box", points=1, n=100003, shifts=8, mixed=False),
        # the same integral with FP32 monomial products
        dict(name="double_box_mixed", kind="plan", integral="double_box", points=1, n=20011, shifts=8, mixed=True),
        # a batch of physical points, contour-deformed, FP64
        dict(name="massive_batch", kind="plan", integral="box_massive", points=250, n=10007, shifts=16, mixed=False),
        # 1024 physical points on the smallest lattice, mixed precision, as a
        # replayed graph: the scan's first pass
        dict(name="massive_batch_mixed", kind="plan", integral="box_massive", points=1024, n=1009, shifts=16,
             mixed=True, graph=True),
        # deformed sectors with poles (subtraction on the deformed contour)
        dict(name="box_physical", kind="plan", integral="box_physical", points=60, n=4001, shifts=16, mixed=False),
        # D = 2 - 2 eps: Taylor-subtracted endpoint singularities under baker
        dict(name="box_d2_baker", kind="plan", integral="box_d2", points=1, n=10007, shifts=32, mixed=False, baker=True),
        # the amplitude at a row of grid points to 1e-4, batched, mixed precision
        dict(name="amplitude_adaptive", kind="adaptive", points=100, shifts=16, mixed=True),
        # the sizing network: 24 Adam steps on 2000 points, then 8000 predictions
        dict(name="mlp_train", kind="mlp", rows=2000, predict=8000, nout=134, steps=24),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["oneshot", "plan", "plan", "plan", "plan", "plan", "adaptive", "mlp"])
    if kind == "adaptive":
        return dict(kind=kind, points=round(_log_uniform(rng, 3, 120)), shifts=rng.choice([8, 16, 32]),
                    mixed=rng.random() < 0.6)
    if kind == "mlp":
        return dict(kind=kind, rows=round(_log_uniform(rng, 100, 4000)), predict=round(_log_uniform(rng, 10, 10000)),
                    nout=rng.randint(20, 200), steps=rng.randint(2, 30))
    name = rng.choice(sorted(INTEGRALS))
    shifts = rng.choice([7, 8, 16, 32])
    if kind == "oneshot":
        name = rng.choice(["triangle", "box", "box_massive"])
        shifts = rng.choice([7, 16])
    nsec = len(_integral(name).sectors)
    cap = (2e7 if kind == "oneshot" else MOST_EVALS[name]) / (nsec * shifts)
    sizes = [n for n in lattice_sizes() if 1009 <= n <= min(400009, cap)]
    want = _log_uniform(rng, sizes[0], sizes[-1])
    n = min(sizes, key=lambda s: abs(math.log(s / want)))
    batch = kind == "plan" and name not in ("triangle", "double_box")
    points = round(_log_uniform(rng, 1, max(1.0, min(1024.0, cap / n)))) if batch else 1
    return dict(kind=kind, integral=name, points=points, n=n, shifts=shifts,
                mixed=name not in ("triangle", "box_d2") and rng.random() < 0.3, baker=name == "box_d2")


# ---------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _integral(name):
    return INTEGRALS[name][0]()


@functools.lru_cache(maxsize=None)
def _text(name):
    return _integral(name).to_text()


def _kinematics(name, points, rng):
    if name == "triangle":
        return np.zeros((1, 0))
    if INTEGRALS[name][3]:
        s, t = rng.uniform(5.0, 20.0, points), rng.uniform(-8.0, -1.0, points)
        # keep off u = -s - t = 0, where the massless integrands are not integrable
        t = np.where(np.abs(s + t) < 0.2, t + 0.4, t)
    else:
        s, t = rng.uniform(-4.0, -2.0, points), rng.uniform(-3.0, -1.0, points)
    return np.stack([s, t], axis=1)


class _State:
    """A context with its plan or network, given back when the state goes."""

    def __init__(self, case):
        self.case, self.ctx, self.plan, self.net = case, None, None, None

    def __del__(self):
        if self.plan is not None:
            qmc.qmc_plan_destroy(self.plan)
        if self.ctx is not None:
            qmc.qmc_destroy(self.ctx)
        if self.net is not None:
            self.net.close()


def _inputs(case, seed):
    """Kinematic points and shift seed of an evaluation case."""
    rng = np.random.default_rng(seed)
    return _kinematics(case["integral"], case["points"], rng), int(rng.integers(1, 1 << 40))


def _mlp_inputs(case, seed):
    """Training rows (kinematic features, standardised targets), weights of the
    outputs, rows to predict and initial parameters."""
    rng = np.random.default_rng(seed)
    nout = case["nout"]
    x = rng.uniform(-1.0, 1.0, (case["rows"], 2)).astype(np.float32)
    p = rng.normal(size=(3, nout))
    y = np.sin(x @ p[:2] * 2.0 + p[2]) + 0.3 * rng.normal(size=(case["rows"], nout))
    wt = np.ones(nout, dtype=np.float32)
    wt[-6:] = 4.0
    xp = rng.uniform(-1.0, 1.0, (case["predict"], 2)).astype(np.float32)
    par = []
    for fan_in, rows in [(2, 256)] + [(256, 256)] * 3 + [(256, nout)]:
        par.append(rng.uniform(-1.0, 1.0, rows * fan_in) / math.sqrt(fan_in))
        par.append(np.zeros(rows))
    return x, y.astype(np.float32), wt, xp, np.concatenate(par).astype(np.float32)


def prepare(case, seed):
    st = _State(case)
    if case["kind"] == "mlp":
        st.x, st.y, st.wt, st.xp, st.par = _mlp_inputs(case, seed)
        st.net = qmc.Mlp(2, 256, 4, case["nout"])
        return st
    precision = qmc.QMC_PRECISION_MIXED if case["mixed"] else qmc.QMC_PRECISION_FP64
    if case["kind"] == "adaptive":
        rng = np.random.default_rng(seed)
        pts = _kinematics("box_physical", case["points"], rng)
        integrals = workloads.amplitude_integrals()
        coef = workloads.amplitude_coefficient_values(pts, workloads.amplitude_coefficients(len(integrals)))
        st.coef = coef.reshape(len(pts), 1, len(integrals), 1).astype(np.complex128)
        st.ctx = qmc.qmc_create(0, precision=precision, shifts=case["shifts"], seed=int(rng.integers(1, 1 << 40)),
                                target_mode=qmc.QMC_TARGET_AMPLITUDE, max_points=1000003, min_points=1009,
                                max_growth=4)
        qmc.load_lattice_table(st.ctx)
        st.ids = [qmc.qmc_load_sectors_mem(st.ctx, I.to_text()) for I in integrals]
        qmc.qmc_set_kinematics(st.ctx, pts)
        return st
    kin, shift_seed = _inputs(case, seed)
    name = case["integral"]
    _, st.lo, st.norders, _ = INTEGRALS[name]
    transform = qmc.QMC_TRANSFORM_BAKER if case.get("baker") else qmc.QMC_TRANSFORM_KOROBOV3
    st.ctx = qmc.qmc_create(0, precision=precision, transform=transform)
    qmc.load_lattice_table(st.ctx)
    iid = qmc.qmc_load_sectors_mem(st.ctx, _text(name))
    qmc.qmc_set_kinematics(st.ctx, kin)
    lam = 1.0 if INTEGRALS[name][3] else 0.0
    specs = qmc.jobs_for_integral(iid, len(_integral(name).sectors), len(kin), case["n"], case["shifts"],
                                  seed=shift_seed, lam=lam)
    st.jobs, st.njobs = qmc.make_jobs(specs)
    st.size = st.njobs * case["shifts"] * st.norders * 2
    if case["kind"] == "plan":
        st.plan = qmc.qmc_plan_create(st.ctx, st.jobs, st.njobs, st.lo, st.norders)
        qmc.qmc_plan_use_graph(st.ctx, st.plan, bool(case.get("graph")))
        st.out = torch.empty(st.size, dtype=torch.float64, device=DEVICE)
        st.stream = torch.cuda.Stream()
    return st


def run(state):
    case = state.case
    if case["kind"] == "oneshot":
        return qmc.qmc_eval_jobs(state.ctx, state.jobs, state.njobs, state.lo, state.norders, state.size)
    if case["kind"] == "plan":
        qmc.qmc_plan_run(state.ctx, state.plan, state.out.data_ptr(), state.stream.cuda_stream)
        return state.out
    if case["kind"] == "adaptive":
        value, error, _, _ = qmc.qmc_integrate(state.ctx, state.ids, coef=state.coef, epsrel=1e-4, lowest_order=-2,
                                               norders=3, npoints=case["points"], check=False, shifts=case["shifts"])
        return {"value": value, "error": error}
    state.net.set_params(state.par)
    losses = state.net.train(state.x, state.y, case["steps"], 1e-3, wt=state.wt)
    return {"losses": losses, "prediction": state.net.forward(state.xp), "params": state.net.params()}


# ---------------------------------------------------------------- work
def _sector_flops(sec, norders):
    """A floor on the arithmetic of one evaluation: the transform, one fused
    multiply-add per monomial and its factors' products, and per subtraction
    corner the integer powers and the series terms of every order (a complex
    operation counts four)."""
    cplx = 4 if sec.deform else 1
    f = 12.0 * sec.d
    mono = sum(1 + sum(1 for x in e if x) for P in (sec.U, sec.F) for e in P.terms)
    f += cplx * mono
    if sec.deform:
        f += 2.0 * mono * sec.d + 8.0 * sec.d * sec.d
    box = 1
    for a in sec.a:
        box *= 1 + max(0, -int(a))
    return f + cplx * box * (6.0 + 2.0 * norders)


def work(case):
    if case["kind"] == "mlp":
        weights = 2 * 256 + 3 * 256 * 256 + 256 * case["nout"]
        rows = 3.0 * case["rows"] * case["steps"] + case["predict"]
        out = weights + case["nout"] * case["predict"] + case["steps"]
        return {"bytes": 4.0 * (out + case["rows"] * (2 + case["nout"]) + 2 * case["predict"]),
                "flops": 2.0 * weights * rows}
    if case["kind"] == "adaptive":
        sectors = [s for I in workloads.amplitude_integrals() for s in I.sectors]
        flops = sum(_sector_flops(s, 3) for s in sectors) * case["points"] * case["shifts"] * 1009.0
        return {"bytes": case["points"] * (16.0 + 160.0 + 96.0), "flops": flops}
    secs = _integral(case["integral"]).sectors
    norders = INTEGRALS[case["integral"]][2]
    each = float(case["points"]) * case["shifts"]
    return {"bytes": each * len(secs) * norders * 16.0 + case["points"] * 16.0,
            "flops": sum(_sector_flops(s, norders) for s in secs) * each * case["n"]}


# ---------------------------------------------------------------- 64-bit values
def _splitmix_uniforms(seed, stream, count):
    state = (seed ^ (GAMMA * (stream + 1))) & MASK64
    i = np.arange(1, count + 1, dtype=np.uint64)
    z = np.uint64(state) + i * np.uint64(GAMMA)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z = z ^ (z >> np.uint64(31))
    return (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53


def _log(P):
    """Principal logarithm; negative real values from below (F - i0)."""
    if not P.is_complex():
        return torch.log(P)
    arg = torch.atan2(P.imag, P.real)
    arg = torch.where((P.imag == 0) & (P.real < 0), -math.pi, arg)
    return torch.complex(0.5 * torch.log(P.real ** 2 + P.imag ** 2), arg)


def _ipow(P, e):
    r = None
    for _ in range(abs(e)):
        r = P if r is None else r * P
    return 1.0 if r is None else (r if e > 0 else 1.0 / r)


class _Series:
    """Truncated power series: {exponents: tensor}, exponents below `caps`."""

    def __init__(self, caps, terms):
        self.caps, self.terms = caps, terms

    def __mul__(self, other):
        out = {}
        for (e, x), (g, y) in itertools.product(self.terms.items(), other.terms.items()):
            k = tuple(a + b for a, b in zip(e, g))
            if all(a < c for a, c in zip(k, self.caps)):
                out[k] = out[k] + x * y if k in out else x * y
        return _Series(self.caps, out)

    def add(self, other, scale=1.0):
        out = dict(self.terms)
        for e, x in other.terms.items():
            out[e] = out[e] + scale * x if e in out else scale * x
        return _Series(self.caps, out)


def _powers(caps):
    """The powers of a series without a constant term that do not vanish."""
    return range(1, sum(c - 1 for c in caps) + 1)


def _corner_factor(caps, P, e0, e1):
    """(P0^e0, exponent series of P^{e0 + e1 eps} / P0^e0) of one power factor;
    the last index of a series counts eps."""
    zero = (0,) * len(caps)
    P0 = P.terms[zero]
    L = _Series(caps, {})
    x = _Series(caps, {k: v / P0 for k, v in P.terms.items() if k != zero})
    xk = None
    if x.terms:
        for k in _powers(caps):
            xk = x if xk is None else xk * x
            if not xk.terms:
                break
            L = L.add(xk, (-1.0) ** (k + 1) / k)
    N = L.add(L, e0 - 1.0) if e0 else _Series(caps, {})
    if e1:
        eps = zero[:-1] + (1,)
        if caps[-1] > 1:
            full = L.add(_Series(caps, {zero: _log(P0)}))
            N = N.add(full * _Series(caps, {eps: torch.full_like(P0, e1)}))
    return _ipow(P0, int(e0)), N


def _laurent_mul(a, b, hi):
    out = {}
    for (i, x), (j, y) in itertools.product(a.items(), b.items()):
        if i + j <= hi:
            out[i + j] = out[i + j] + x * y if i + j in out else x * y
    return out


def _integrand(sec, inv, t, omt, lam, lo, norders):
    """Coefficients eps^lo.. of the subtracted integrand at t (list of tensors
    broadcastable with the invariants)."""
    d, hi = sec.d, lo + norders - 1
    sing = sec.singular
    Hm = hi + len(sing)
    one = torch.ones_like(t[0])

    def coef(c):
        return float(c[0]) + sum(float(ci) * v for ci, v in zip(c[1:], inv))

    total = {}
    for V in itertools.product((0, 1), repeat=len(sing)):
        zeroed = [j for j, v in zip(sing, V) if v]
        caps = tuple(-sec.a[j] for j in zeroed) + (max(1, hi + len(zeroed) + 1),)

        def poly(P, x, power):
            terms = {}
            for e, c in P.terms.items():
                k = tuple(e[j] for j in zeroed) + (0,)
                if any(a >= m for a, m in zip(k, caps)):
                    continue
                v = coef(c) * one
                for j in range(d):
                    if j not in zeroed and e[j]:
                        v = v * power[j][e[j]]
                terms[k] = terms[k] + v if k in terms else v
            return _Series(caps, terms)

        factors = []
        lead = one
        if lam is None:
            x = t
        else:
            tc = [torch.zeros_like(t[j]) if j in zeroed else t[j] for j in range(d)]
            oc = [torch.ones_like(t[j]) if j in zeroed else omt[j] for j in range(d)]
            dF = [one * 0.0 for _ in range(d)]
            H = [[one * 0.0 for _ in range(d)] for _ in range(d)]
            for e, c in sec.F.terms.items():
                for j in range(d):
                    if not e[j]:
                        continue
                    dF[j] = dF[j] + coef(c) * e[j] * math.prod(
                        (tc[i] ** (e[i] - (i == j)) for i in range(d) if e[i] - (i == j)), start=one)
                    for k in range(d):
                        ek = e[k] - (j == k)
                        if ek > 0:
                            H[j][k] = H[j][k] + coef(c) * e[j] * ek * math.prod(
                                (tc[i] ** (e[i] - (i == j) - (i == k)) for i in range(d)
                                 if e[i] - (i == j) - (i == k)), start=one)
            rho = [torch.complex(one, -lam * oc[j] * dF[j]) for j in range(d)]
            x = [tc[j] * rho[j] for j in range(d)]
            J = [[torch.complex(one if j == k else one * 0.0,
                                -lam * (tc[j] * oc[j] * H[j][k] + ((oc[j] - tc[j]) * dF[j] if j == k else 0.0)))
                  for k in range(d)] for j in range(d)]
            if d == 2:
                det = J[0][0] * J[1][1] - J[0][1] * J[1][0]
            else:
                det = (J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1])
                       - J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0])
                       + J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]))
            lead = det
            zero = (0,) * len(caps)
            for j in sing:
                factors.append((_Series(caps, {zero: rho[j]}), sec.a[j], float(sec.b[j])))
        power = [{1: x[j]} for j in range(d)]
        for j in range(d):
            for e in range(2, 5):
                power[j][e] = power[j][e - 1] * x[j]
        zero = (0,) * len(caps)
        for j in range(d):
            if j not in sing and (sec.a[j] or sec.b[j]):
                factors.append((_Series(caps, {zero: x[j]}), sec.a[j], float(sec.b[j])))
        factors.append((poly(sec.U, x, power), float(sec.u0), float(sec.u1)))
        factors.append((poly(sec.F, x, power), float(sec.f0), float(sec.f1)))
        N = _Series(caps, {})
        for P, e0, e1 in factors:
            p, n = _corner_factor(caps, P, e0, e1)
            lead = lead * p
            N = N.add(n)
        G, term = _Series(caps, {zero: one}), _Series(caps, {zero: one})
        # the exponent's constant terms in eps alone and its terms in t are nilpotent
        for k in _powers(caps):
            term = term * N
            if not term.terms:
                break
            term = _Series(caps, {e: v / k for e, v in term.terms.items()})
            G = G.add(term)
        base = {0: lead}
        phis = {}
        for q, (j, v) in enumerate(zip(sing, V)):
            p, b = -sec.a[j], float(sec.b[j])
            bl = b * torch.log(t[j])
            expo, e = {}, one
            for i in range(Hm + 1):
                expo[i] = e
                e = e * bl / (i + 1)
            if not v:
                base = _laurent_mul(base, {i: y * t[j] ** (-p) for i, y in expo.items()}, Hm)
                continue
            for k in range(p):
                phi = {i: -y * t[j] ** (k - p) for i, y in expo.items()}
                m = k - p + 1
                if m == 0:
                    phi[-1] = one / b
                else:
                    c = 1.0 / m
                    for i in range(Hm + 1):
                        phi[i] = phi[i] + c
                        c *= -b / m
                phis[j, k] = phi
        acc = {}
        for e, v in G.terms.items():
            part = {e[-1]: v}
            for j, k in zip(zeroed, e):
                part = _laurent_mul(part, phis[j, k], Hm)
            for i, y in part.items():
                acc[i] = acc[i] + y if i in acc else y
        for i, y in _laurent_mul(base, acc, hi).items():
            total[i] = total[i] + y if i in total else y
    return [total.get(lo + o) for o in range(norders)]


def _exact_sums(case, seed):
    kin, shift_seed = _inputs(case, seed)
    name = case["integral"]
    I = _integral(name)
    _, lo, norders, physical = INTEGRALS[name]
    m, n, nsec = case["shifts"], case["n"], len(I.sectors)
    out = np.zeros((len(kin), nsec, m, norders, 2))
    k = torch.arange(n, dtype=torch.int64, device=DEVICE)
    chunk = max(1, int(4e6 / (m * n)))          # kinematic points at a time
    for s, sec in enumerate(I.sectors):
        _, z = lattice_for(n, sec.d)
        frac = [((k * int(z[j])) % n).double() / n for j in range(sec.d)]
        for p0 in range(0, len(kin), chunk):
            pts = range(p0, min(len(kin), p0 + chunk))
            delta = torch.tensor(np.stack([_splitmix_uniforms(shift_seed, p * nsec + s, m * sec.d).reshape(m, sec.d)
                                           for p in pts]), device=DEVICE)
            inv = [torch.tensor(kin[list(pts), i], device=DEVICE)[:, None, None] for i in range(kin.shape[1])]
            t, omt, w = [], [], float(sec.weight)
            for j in range(sec.d):
                u = frac[j] + delta[:, :, j, None]
                u = torch.where(u >= 1.0, u - 1.0, u)
                if case.get("baker"):
                    t.append(torch.where(u < 0.5, 2.0 * u, 2.0 * (1.0 - u)))
                    omt.append(torch.where(u < 0.5, 1.0 - 2.0 * u, 2.0 * u - 1.0))
                else:
                    v = 1.0 - u
                    phi = [x ** 4 * (35.0 - x * (84.0 - x * (70.0 - 20.0 * x))) for x in (u, v)]
                    lower = u < 0.5          # the small one of t, 1 - t without cancellation
                    t.append(torch.where(lower, phi[0], 1.0 - phi[1]))
                    omt.append(torch.where(lower, 1.0 - phi[0], phi[1]))
                    w = w * 140.0 * (u * v) ** 3
            use = functools.reduce(torch.logical_and, [x > 0 for x in t])
            t = [torch.where(use, x, 0.5) for x in t]
            res = _integrand(sec, inv, t, omt, 1.0 if physical else None, lo, norders)
            for o, f in enumerate(res):
                if f is None:
                    continue
                f = torch.where(use, f * w, 0.0).sum(dim=-1) / n
                out[p0:p0 + len(pts), s, :, o, 0] = f.real.cpu().numpy() if f.is_complex() else f.cpu().numpy()
                if f.is_complex():
                    out[p0:p0 + len(pts), s, :, o, 1] = f.imag.cpu().numpy()
    return out.reshape(-1)


def _exact_mlp(case, seed):
    x, y, wt, xp, par = (a.astype(np.float64) for a in _mlp_inputs(case, seed))
    shapes = [(256, 2)] + [(256, 256)] * 3 + [(case["nout"], 256)]

    def views(flat):
        out, off = [], 0
        for r, c in shapes:
            out.append((flat[off:off + r * c].reshape(r, c), flat[off + r * c:off + r * c + r]))
            off += r * c + r
        return out

    layers, grad = views(par), np.zeros_like(par)
    gviews = views(grad)

    def forward(h):
        acts = [h]
        for i, (W, b) in enumerate(layers):
            h = h @ W.T + b
            if i < 4:
                h = np.tanh(h)
            acts.append(h)
        return acts

    m, v = np.zeros_like(par), np.zeros_like(par)
    losses = []
    for step in range(1, case["steps"] + 1):
        acts = forward(x)
        r = acts[-1] - y
        losses.append(float((wt * r * r).sum() / len(x)))
        dz = 2.0 * wt * r / len(x)
        for i in range(4, -1, -1):
            gviews[i][0][:] = dz.T @ acts[i]
            gviews[i][1][:] = dz.sum(axis=0)
            if i:
                dz = (dz @ layers[i][0]) * (1.0 - acts[i] ** 2)
        m = 0.9 * m + 0.1 * grad
        v = 0.999 * v + 0.001 * grad * grad
        par -= 1e-3 * (m / (1.0 - 0.9 ** step)) / (np.sqrt(v / (1.0 - 0.999 ** step)) + 1e-8)
    return {"losses": np.array(losses, dtype=np.float64), "prediction": forward(xp)[-1], "params": par}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    if case["kind"] == "adaptive":
        return None      # an estimate whose lattices the driver chooses: no value of its own
    evals = case["points"] * len(_integral(case["integral"]).sectors) * case["shifts"] * case["n"]
    if evals > (6e7 if case["integral"] == "double_box" else 2e8):
        return None      # over about 20 seconds
    return _exact_sums(case, seed)
