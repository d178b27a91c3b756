"""Measured cases of the Magnus library: what its users have it do, through its public calls.

A case is one pass of a program that keeps a context and a plan (operators resident on the
GPU) and calls with new data: an evolution takes new drive samples (`mg_set_controls`, the
package's update_control_sigs) and evolves; a step-level call takes a batch of matrices.
The models are the library's circuit-QED and spin-chain families; their parameters and
drives are drawn from the seed.  `exact` gives the same outputs from plain torch in FP64.
"""
import math

import numpy as np
import torch

from paper_2411_09982_gb300 import magnus as M

TWO_PI = 2.0 * math.pi
DEV = "cuda"

FP64, SPLIT = "fp64", "split"


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a strongly driven qubit in its rotating frame, evolved again
        # and again in a pulse search; latency of the call and its launches
        dict(name="qubit_d2_state_fp64", kind="evolve", family="qubit", N=50, P=16, out="state", prec=FP64, slices=6),
        # transmon and resonator, one drive: the ordinary small system, FP64 state
        dict(name="tr_d30_state_fp64", kind="evolve", family="tr", nt=3, nr=10, N=1000, P=16, out="state", prec=FP64,
             slices=6),
        # the same family with the second-order term and every stroboscopic state
        dict(name="tr_d84_order2_traj_fp64", kind="evolve", family="tr", nt=4, nr=21, N=300, P=16, out="trajectory",
             prec=FP64, slices=6, order=2),
        # the paper's spin chain (8 spins, 200 intervals, complex controls), the default precision
        dict(name="spin_d256_state_fp64", kind="evolve", family="spin", n=8, N=200, P=16, out="state", prec=FP64,
             slices=6),
        # full propagator of the six-transmon chain at the default precision
        dict(name="chain_d729_prop_fp64", kind="evolve", family="chain", levels=3, sites=6, N=20, P=16,
             out="propagator", prec=FP64, slices=6),
        # the same chain on the tensor cores: the throughput workload
        dict(name="chain_d729_prop_split", kind="evolve", family="chain", levels=3, sites=6, N=200, P=16,
             out="propagator", prec=SPLIT, slices=6),
        # the largest dimension: four eight-level transmons, all-to-all coupling, two tones
        dict(name="all_d4096_prop_split", kind="evolve", family="all", levels=8, sites=4, N=3, P=8, out="propagator",
             prec=SPLIT, slices=7),
        # a run resumed from a propagator and re-orthonormalised on the way
        dict(name="chain_d243_resume_split", kind="evolve", family="chain", levels=3, sites=5, N=200, P=16,
             out="propagator", prec=SPLIT, slices=6, resume=True, reorth=64),
        # independent jobs of uneven size in one call, split precision
        dict(name="batch32_state_split", kind="batch", jobs=32, dmin=16, dmax=256, Nmin=50, Nmax=400, mix=1, prec=SPLIT,
             slices=6, action=False),
        # the same kind of batch on the sparse action path (FP64)
        dict(name="batch64_state_action", kind="batch", jobs=64, dmin=16, dmax=256, Nmin=200, Nmax=2000, mix=2,
             prec=FP64, slices=6, action=True),
        # a batch of exponentials of arbitrary Hermitian matrices, step-level call
        dict(name="expm_d81_fp64", kind="expm", d=81, batch=64, prec=FP64, slices=6),
        # a batch of general complex products, step-level call, ragged size
        dict(name="cgemm_d487_split", kind="cgemm", d=487, batch=16, prec=SPLIT, slices=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_CHAINS = [(2, 5), (3, 3), (2, 6), (3, 4), (5, 3), (2, 7), (6, 3), (3, 5), (4, 4), (7, 3), (8, 3), (5, 4), (3, 6),
           (9, 3), (10, 3), (11, 3), (6, 4)]


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["evolve", "evolve", "evolve", "evolve", "evolve", "evolve", "batch", "expm", "cgemm"])
    prec = rng.choice([FP64, SPLIT])
    slices = 6
    if kind == "batch":
        dmin = rng.randint(16, 64)
        action = rng.random() < 0.5
        return dict(kind="batch", jobs=rng.randint(3, 32), dmin=dmin, dmax=rng.randint(dmin + 32, 256), Nmin=50,
                    Nmax=rng.randint(100, 400), mix=rng.randrange(1 << 20), prec=FP64 if action else SPLIT, slices=6,
                    action=action)
    if kind in ("expm", "cgemm"):
        d = _log_int(rng, 3, 400 if prec == FP64 else 1000)
        cap = 3e10 if prec == FP64 else 1e12
        batch = max(1, min(_log_int(rng, 1, 200), int(cap / (8.0 * d ** 3))))
        return dict(kind=kind, d=d, batch=batch, prec=prec, slices=6)
    family = rng.choice(["qubit", "tr", "tr", "spin", "chain", "chain"])
    case = dict(kind="evolve", family=family, P=rng.choice([4, 8, 16]), prec=prec, slices=slices)
    if family == "qubit":
        d = 2
    elif family == "tr":
        case.update(nt=rng.randint(2, 8), nr=rng.randint(4, 32))
        d = case["nt"] * case["nr"]
    elif family == "spin":
        case.update(n=rng.randint(3, 8 if prec == FP64 else 9))
        d = 2 ** case["n"]
    else:
        levels, sites = rng.choice([c for c in _CHAINS if c[0] ** c[1] <= (729 if prec == FP64 else 1331)])
        case.update(levels=levels, sites=sites, dt=rng.choice([0.025, 0.05, 0.1, 0.25]))
        d = levels ** sites
    # FP64: at most about half a second of native products; split: the 200 intervals of the
    # paper's evolutions
    cap = 4e11 / (96.0 * d ** 3) if prec == FP64 else 1e13 / (96.0 * d ** 3)
    case["N"] = max(2, min(_log_int(rng, 10, 1000 if prec == FP64 else 200), int(cap)))
    case["out"] = rng.choice(["state", "propagator"]) if d <= 729 else "propagator"
    if case["out"] == "propagator" and rng.random() < 0.25:
        case.update(resume=True, reorth=rng.choice([0, 8, 64]))
    return case


# ----------------------------------------------------------------------------
# models: operators (float64 or complex128 on the GPU), drives (numpy callables)
# ----------------------------------------------------------------------------
def _lower(n):
    return torch.diag(torch.sqrt(torch.arange(1, n, dtype=torch.float64, device=DEV)), 1)


def _kron(ops):
    out = ops[0]
    for o in ops[1:]:
        out = torch.kron(out.contiguous(), o.contiguous())
    return out


def _at(dims, placed, dtype=torch.float64):
    """Tensor product with placed[site] on the named sites and the identity elsewhere."""
    return _kron([placed.get(j, torch.eye(n, dtype=dtype, device=DEV)) for j, n in enumerate(dims)])


class _Tones:
    """u_k(t) = Gaussian envelope x sum_j a cos(w t + phi)."""

    def __init__(self, amp, freq, phase, T, sigma):
        self.amp, self.freq, self.phase, self.tc, self.sigma = amp, freq, phase, T / 2, sigma

    def __call__(self, t):
        t = np.asarray(t)
        env = np.exp(-((t - self.tc) ** 2) / (2.0 * self.sigma ** 2))
        return env[..., None] * (self.amp * np.cos(self.freq * t[..., None, None] + self.phase)).sum(-1)


def _model(case, rng):
    """(H0, [H_k], drive, T): real operators stay float64."""
    fam = case["family"]
    if fam == "qubit":
        T, w = 10.0, TWO_PI * rng.uniform(4.5, 5.5)
        om = rng.uniform(0.1, 0.4) * w
        sx = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128, device=DEV)
        sy = torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128, device=DEV)

        def drive(t):
            q = 0.25 * om * np.exp(-((t - T / 2) ** 2) / (2.0 * (T / 5) ** 2))
            return np.stack([q, q * np.cos(2 * w * t), -q * np.sin(2 * w * t)], axis=-1)

        return torch.zeros(2, 2, dtype=torch.complex128, device=DEV), [sx, sx, sy], drive, T
    if fam == "tr":
        dims, T = [case["nt"], case["nr"]], 50.0
        b, a = _lower(dims[0]), _lower(dims[1])
        wq, al = rng.uniform(4.8, 5.2), rng.uniform(-0.3, -0.2)
        wr, g, om = rng.uniform(6.5, 7.5), rng.uniform(0.05, 0.15), 0.05 * (1.0 - rng.uniform())
        nq = torch.arange(dims[0], dtype=torch.float64, device=DEV)
        na = torch.arange(dims[1], dtype=torch.float64, device=DEV)
        H0 = _at(dims, {0: torch.diag(wq * nq + 0.5 * al * nq * (nq - 1))}) + _at(dims, {1: torch.diag(wr * na)})
        x = _kron([b.T, a])
        H0 = TWO_PI * (H0 + g * (x + x.T))
        drive = _Tones(np.array([[TWO_PI * om]]), np.array([[TWO_PI * wq]]), np.array([[rng.uniform(0, TWO_PI)]]), T,
                       10.0)
        return H0, [_at(dims, {0: b + b.T})], drive, T
    if fam == "spin":
        n = case["n"]
        dims, T = [2] * n, 25.0
        s = torch.arange(2 ** n, device=DEV)
        z = [1.0 - 2.0 * ((s >> (n - 1 - j)) & 1).to(torch.float64) for j in range(n)]
        diag = sum(0.5 * TWO_PI * z[j] - TWO_PI * 0.5 * z[j] * z[(j + 1) % n] - TWO_PI * 0.1 * z[j] * z[(j + 2) % n]
                   for j in range(n))
        sx = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128, device=DEV)
        sy = torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128, device=DEV)
        Hk = [sum(_at(dims, {j: m}, torch.complex128) for j in range(n)) for m in (sx, sy)]
        drive = _Tones(TWO_PI * 0.05 * np.ones((2, 1)), TWO_PI * rng.uniform(0, 10, (2, 1)),
                       rng.uniform(0, TWO_PI, (2, 1)), T, T / 5)
        return torch.diag(diag).to(torch.complex128), Hk, drive, T
    # transmon chain (nearest neighbours) or all-to-all graph with two-tone drives
    dims, T = [case["levels"]] * case["sites"], 50.0
    lv, ns = case["levels"], case["sites"]
    b = _lower(lv)
    n1 = torch.arange(lv, dtype=torch.float64, device=DEV)
    w, al = rng.uniform(4.8, 5.2, ns), rng.uniform(-0.3, -0.2, ns)
    H0 = torch.zeros(lv ** ns, lv ** ns, dtype=torch.float64, device=DEV)
    for j in range(ns):
        H0 += _at(dims, {j: torch.diag(w[j] * n1 + 0.5 * al[j] * n1 * (n1 - 1))})
    for i in range(ns):
        for j in range(i + 1, ns):
            if fam == "all" or j == i + 1:
                x = _at(dims, {i: b.T, j: b})
                H0 += (rng.uniform(0.0, 0.02) if fam == "all" else 0.01) * (x + x.T)
    tones = 2 if fam == "all" else 1
    freq = TWO_PI * np.stack([w, w + al], axis=1)[:, :tones]
    drive = _Tones(TWO_PI * 0.05 * (1.0 - rng.uniform(0, 1, (ns, tones))), freq,
                   rng.uniform(0, TWO_PI, (ns, tones)), T, 10.0)
    return TWO_PI * H0, [_at(dims, {j: b + b.T}) for j in range(ns)], drive, T


def _dim(case):
    fam = case["family"]
    return {"qubit": lambda: 2, "tr": lambda: case["nt"] * case["nr"], "spin": lambda: 2 ** case["n"]}.get(
        fam, lambda: case["levels"] ** case["sites"])()


def _state(d, rng):
    v = rng.standard_normal(d) + 1j * rng.standard_normal(d)
    return torch.from_numpy(v / np.linalg.norm(v)).to(DEV)


def _inputs(case, rng):
    """One evolution's data: operators, samples at the quadrature nodes, input, grid."""
    H0, Hk, drive, T = _model(case, rng)
    N, P = case["N"], case["P"]
    x, w = np.polynomial.legendre.leggauss(P)
    # the chains' workloads take 2000 and 500 intervals of 50 ns: a stretch of N of them
    dt = case.get("dt", {"chain": 0.025, "all": 0.1}.get(case["family"], T / N))
    t0 = 0.5 * T - 0.5 * N * dt   # short runs sit where the drive is on
    t = t0 + dt * np.arange(N)[:, None] + (1.0 + x[None, :]) * (0.5 * dt)
    d = H0.shape[0]
    if case["out"] != "propagator":
        inp = _state(d, rng)
    elif case.get("resume"):
        # an earlier stretch's propagator: a random unitary
        g = torch.from_numpy(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))).to(DEV)
        inp = torch.linalg.qr(g)[0].contiguous()
    else:
        inp = None
    return dict(H0=H0, Hk=Hk, drive=drive, N=N, P=P, t0=t0, dt=dt, w=w,
                samples=np.ascontiguousarray(drive(t)), inp=inp, d=d)


def _batch_cases(case):
    """The jobs' sizes belong to the case, their parameters and drives to the seed."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["jobs"]):
        while True:
            nt, nr = int(rng.integers(2, 9)), int(rng.integers(8, 33))
            if case["dmin"] <= nt * nr <= case["dmax"]:
                break
        out.append(dict(family="tr", nt=nt, nr=nr, N=int(rng.integers(case["Nmin"], case["Nmax"] + 1)), P=16,
                        out="state"))
    return out


def _matrices(case, seed):
    """Step-level operands: Hermitian exponents of norms from 0.1 to 20, or general matrices."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    d, n = case["d"], case["batch"]

    def normal():
        return torch.randn(n, d, d, dtype=torch.complex128, device=DEV, generator=g)

    A = normal()
    if case["kind"] == "cgemm":
        return A, normal()
    A = 0.5 * (A + A.mH) / math.sqrt(d)   # spectrum within about +-1.5
    scale = torch.exp(torch.rand(n, 1, 1, dtype=torch.float64, device=DEV, generator=g) * math.log(200.0)) * 0.1
    return (scale * A).contiguous(), None


# ----------------------------------------------------------------------------
# a pass
# ----------------------------------------------------------------------------
def _plan(ctx, case, x):
    H0 = x["H0"].to(torch.complex128).contiguous()
    Hk = torch.stack([h.to(torch.complex128) for h in x["Hk"]]).contiguous()
    plan = M.Plan(ctx, H0, Hk, M.MG_PREC_SPLIT if case["prec"] == SPLIT else M.MG_PREC_FP64, case["slices"],
                  M.MG_FLAG_STATE_ACTION if case.get("action") else 0)
    if case.get("order", 1) != 1:
        plan.set_magnus_order(case["order"])
    return plan


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    ctx = M.Context(0)
    prec = M.MG_PREC_SPLIT if case["prec"] == SPLIT else M.MG_PREC_FP64
    st = dict(kind=case["kind"], ctx=ctx, prec=prec, slices=case["slices"])
    if case["kind"] in ("expm", "cgemm"):
        st["A"], st["B"] = _matrices(case, seed)
        st["out"] = torch.empty_like(st["A"])
        return st
    if case["kind"] == "batch":
        xs = [_inputs(c, rng) for c in _batch_cases(case)]
        st["plans"] = [_plan(ctx, case, x) for x in xs]
        st["controls"] = [(x["N"], x["P"], x["t0"], x["dt"], x["w"], torch.from_numpy(x["samples"]).to(DEV))
                          for x in xs]
        st["inputs"] = [x["inp"] for x in xs]
        # the final states end to end in one buffer
        st["psi"] = torch.empty(sum(x["d"] for x in xs), dtype=torch.complex128, device=DEV)
        st["outs"] = list(torch.split(st["psi"], [x["d"] for x in xs]))
        torch.cuda.synchronize()
        return st
    x = _inputs(case, rng)
    d, N = x["d"], x["N"]
    st["plan"] = _plan(ctx, case, x)
    st["controls"] = (N, x["P"], x["t0"], x["dt"], x["w"], torch.from_numpy(x["samples"]).to(DEV))
    st["output"] = dict(state=M.MG_OUT_STATE, propagator=M.MG_OUT_PROPAGATOR,
                        trajectory=M.MG_OUT_TRAJECTORY)[case["out"]]
    st["reorth"] = case.get("reorth", 0)
    st["inp"] = x["inp"]
    shape = dict(state=(d,), propagator=(d, d), trajectory=(N + 1, d))[case["out"]]
    st["out"] = torch.empty(shape, dtype=torch.complex128, device=DEV)
    torch.cuda.synchronize()
    return st


def run(st):
    """New controls, then the evolution (with its report, as the binding does by default); or the step-level call."""
    if st["kind"] == "expm":
        M.mg_expm(st["ctx"], st["A"].shape[0], st["A"].shape[1], st["A"], st["out"], st["prec"], st["slices"])
        return st["out"]
    if st["kind"] == "cgemm":
        M.mg_cgemm(st["ctx"], st["A"].shape[0], st["A"].shape[1], st["A"], st["B"], st["out"], st["prec"],
                   st["slices"])
        return st["out"]
    if st["kind"] == "batch":
        for plan, c in zip(st["plans"], st["controls"]):
            plan.set_controls(*c)
        status = M.mg_evolve_batch(st["ctx"], st["plans"], [M.MG_OUT_STATE] * len(st["plans"]), st["inputs"],
                                   st["outs"])
        return dict(psi=st["psi"], status=np.array(status, dtype=np.int32))
    st["plan"].set_controls(*st["controls"])
    st["plan"].evolve(st["output"], st["inp"], st["out"], st["reorth"])
    return st["out"]


def work(case):
    """Bytes: operators, samples and input read once, result written once.  Flops: a dense
    exponential takes at least five complex products (degree 18) and one more folds it in;
    with real operators its polynomial in i H needs real products only.  The action path
    applies the operators' nonzeros to the state a few dozen times per interval."""
    if case["kind"] == "cgemm":
        d, n = case["d"], case["batch"]
        return dict(bytes=48 * d * d * n, flops=8 * d ** 3 * n)
    if case["kind"] == "expm":
        d, n = case["d"], case["batch"]
        return dict(bytes=32 * d * d * n, flops=5 * 8 * d ** 3 * n)
    if case["kind"] == "batch":
        # the mean job
        d, N, n = 0.5 * (case["dmin"] + case["dmax"]), 0.5 * (case["Nmin"] + case["Nmax"]), case["jobs"]
        per = 8 * 7 * d * 30 if case["action"] else 5 * 2 * d ** 3 + 8 * d * d
        return dict(bytes=n * (32 * d * d + N * 16 * 8), flops=n * N * per)
    d, N, P = _dim(case), case["N"], case["P"]
    K = dict(qubit=3, tr=1, spin=2).get(case["family"], case.get("sites", 1))
    real = case["family"] in ("tr", "chain", "all") and case.get("order", 1) == 1
    fold = 8 * d ** 3 if case["out"] == "propagator" else 8 * d * d
    rows = dict(state=2, propagator=d * (2 if case.get("resume") else 1), trajectory=N + 2)[case["out"]]
    return dict(bytes=16 * d * d * (1 + K) + 8 * N * P * K + 16 * d * rows,
                flops=N * (5 * (2 if real else 8) * d ** 3 + fold))


# ----------------------------------------------------------------------------
# the same outputs in plain FP64
# ----------------------------------------------------------------------------
def _coefs(x):
    """c_{k,n} = (dt/2) sum_p w_p u_k(t_{n,p})"""
    return 0.5 * x["dt"] * np.einsum("p,npk->nk", x["w"], x["samples"])


def _second_order(x, ops):
    """(operators, coefficients) of -(i/2) int int_{t2 <= t1} [H(t1), H(t2)] by nested quadrature."""
    xs, ws = np.polynomial.legendre.leggauss(16)
    s, w = 0.5 * (1.0 + xs), 0.5 * ws
    dt = x["dt"]
    t = x["t0"] + dt * np.arange(x["N"])[:, None]

    def u(tt):
        v = x["drive"](tt)
        return np.concatenate([np.ones(v.shape[:-1] + (1,)), v], axis=-1)

    u1 = u(t + dt * s[None, :])                                    # N x P x (1 + K)
    u2 = u(t[:, :, None] + dt * (s[:, None] * s[None, :])[None])   # N x P x Q x (1 + K)
    inner = np.einsum("q,npqb->npb", w, u2) * (dt * s)[None, :, None]
    I = dt * np.einsum("p,npa,npb->nab", w, u1, inner)
    out_ops, cs = [], []
    for a in range(len(ops)):
        for b in range(a + 1, len(ops)):
            A, B = ops[a].to(torch.complex128), ops[b].to(torch.complex128)
            out_ops.append(-0.5j * (A @ B - B @ A))
            cs.append(I[:, a, b] - I[:, b, a])
    return out_ops, np.stack(cs, axis=1)


def _bessel(r):
    """J_k(r), k = 0.. until negligible (Miller's downward recurrence)."""
    n = int(1.5 * r) + 60
    j = np.zeros(n + 2)
    j[n] = 1e-280
    for k in range(n, 0, -1):
        j[k - 1] = 2.0 * k / max(r, 1e-12) * j[k] - j[k + 1]
        if abs(j[k - 1]) > 1e250:
            j *= 1e-250
    j /= j[0] + 2.0 * j[2::2].sum()
    keep = int(np.nonzero(np.abs(j) > 1e-19)[0].max()) + 1
    return j[:keep]


def _exact_states(xs, orders, trajectory=False):
    """psi(T) of several jobs (padded to one dimension): Chebyshev series of every interval."""
    dm, n = max(x["d"] for x in xs), len(xs)
    nops = max(len(x["Hk"]) for x in xs) + 1
    full = []
    for x, order in zip(xs, orders):
        ops, c = [x["H0"]] + x["Hk"], _coefs(x)
        c = np.concatenate([np.full((x["N"], 1), x["dt"]), c], axis=1)
        if order == 2:
            o2, c2 = _second_order(x, ops)
            ops, c = ops + o2, np.concatenate([c, c2], axis=1)
            nops = max(nops, len(ops))
        full.append((ops, c))
    O = torch.zeros(n, nops, dm, dm, dtype=torch.complex128, device=DEV)
    N = max(x["N"] for x in xs)
    C = np.zeros((N, n, nops))
    psi = torch.zeros(n, dm, 1, dtype=torch.complex128, device=DEV)
    for i, ((ops, c), x) in enumerate(zip(full, xs)):
        for k, o in enumerate(ops):
            O[i, k, :x["d"], :x["d"]] = o
        C[:x["N"], i, :c.shape[1]] = c
        psi[i, :x["d"], 0] = x["inp"]
    # one spectral interval per job: Gershgorin with the largest coefficients
    cmax = torch.from_numpy(np.abs(C).max(axis=0)).to(DEV)
    diag = torch.diagonal(O[:, 0], dim1=-2, dim2=-1).real * cmax[:, :1]
    rest = torch.zeros(n, dm, dtype=torch.float64, device=DEV)
    for k in range(nops):
        a = O[:, k].abs()
        if k == 0:
            a = a - torch.diag_embed(torch.diagonal(a, dim1=-2, dim2=-1))
        rest += a.sum(-1) * cmax[:, k:k + 1]
    lo, hi = (diag - rest).min(-1).values, (diag + rest).max(-1).values
    mid, rad = 0.5 * (lo + hi), (0.5 * (hi - lo)).clamp_min(1e-3)
    js = [_bessel(float(r)) for r in rad]
    terms = max(len(j) for j in js)
    co = np.zeros((terms, n), dtype=np.complex128)
    for i, j in enumerate(js):
        co[:len(j), i] = np.array([1.0 if k == 0 else 2.0 for k in range(len(j))]) * j * (-1j) ** np.arange(len(j))
    co *= np.exp(-1j * mid.cpu().numpy())[None]
    co = torch.from_numpy(co).to(DEV).view(terms, n, 1, 1)
    Cd = torch.from_numpy(C).to(DEV)
    last = torch.tensor([x["N"] for x in xs], device=DEV).view(n, 1, 1)
    eye = torch.eye(dm, dtype=torch.complex128, device=DEV)
    rows = [psi.clone()]
    flat = O.view(n, nops, dm * dm)
    for s in range(N):
        H = torch.bmm(Cd[s].to(torch.complex128).view(n, 1, nops), flat).view(n, dm, dm)
        H = (H - mid.view(n, 1, 1) * eye) / rad.view(n, 1, 1)
        t0, t1 = psi, torch.bmm(H, psi)
        acc = co[0] * t0 + (co[1] * t1 if terms > 1 else 0)
        for k in range(2, terms):
            t0, t1 = t1, 2.0 * torch.bmm(H, t1) - t0
            acc = acc + co[k] * t1
        psi = torch.where(s < last, acc, psi)
        if trajectory:
            rows.append(psi)
    if trajectory:
        return torch.stack([r[0, :, 0] for r in rows])
    return [psi[i, :x["d"], 0].contiguous() for i, x in enumerate(xs)]


def _expm(A):
    """exp(-i A) of a batch of Hermitian (complex128) or real symmetric (float64) matrices."""
    nrm = A.abs().sum(-2).max().item()
    s = max(0, math.ceil(math.log2(max(nrm, 1e-300) / 0.5)))
    A = A * 2.0 ** -s
    d = A.shape[-1]
    eye = torch.eye(d, dtype=A.dtype, device=A.device)
    if not A.is_complex():
        # cosine and sine as polynomials in A^2 (degrees 16 and 17)
        Y = A @ A
        c = eye / math.factorial(16)
        q = eye / math.factorial(17)
        for k in range(7, -1, -1):
            c = eye / math.factorial(2 * k) - Y @ c
            q = eye / math.factorial(2 * k + 1) - Y @ q
        c, q = c + 0.0, A @ q
        for _ in range(s):
            c, q = (c + q) @ (c - q), 2.0 * (c @ q)
        return torch.complex(c, -q)
    X = -1j * A
    T = eye / math.factorial(18) + 0 * X
    for k in range(17, -1, -1):
        T = eye / math.factorial(k) + X @ T
    for _ in range(s):
        T = T @ T
    return T


def exact(case, seed):
    if case["kind"] in ("expm", "cgemm"):
        A, B = _matrices(case, seed)
        if case["kind"] == "cgemm":
            return torch.stack([a @ b for a, b in zip(A, B)])
        out = []
        for a in A:
            lam, V = torch.linalg.eigh(a)
            out.append((V * torch.exp(-1j * lam)) @ V.mH)
        return torch.stack(out)
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        xs = [_inputs(c, rng) for c in _batch_cases(case)]
        return dict(psi=torch.cat(_exact_states(xs, [1] * len(xs))), status=None)
    x = _inputs(case, rng)
    if case["out"] == "state":
        return _exact_states([x], [case.get("order", 1)])[0]
    if case["out"] == "trajectory":
        return _exact_states([x], [case.get("order", 1)], trajectory=True)
    c = _coefs(x)
    U = x["inp"] if x["inp"] is not None else torch.eye(x["d"], dtype=torch.complex128, device=DEV)
    for n in range(x["N"]):
        H = x["dt"] * x["H0"]
        for k, h in enumerate(x["Hk"]):
            H = H + float(c[n, k]) * h
        tau = torch.diagonal(H).real.mean().item()
        U = (_expm(H - tau * torch.eye(x["d"], dtype=H.dtype, device=DEV)) * complex(math.cos(tau), -math.sin(tau))) @ U
    return U
