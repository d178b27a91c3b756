"""Weak entries in MG_PREC_FP64: products of arbitrary operands (mg_propagate, mg_expm, a resumed
run's running product) hold FP64's error entry by entry, |error| <= c u |A| |B|, whatever the
range of a row's entries; and so does every product under Context.set_fp64_entrywise(True)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


def enough(d):
    """A batch whose products run from digits at dimension d."""
    return 8000000 // (-(-d // 16) * 16) ** 3 + 1


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("d", [33, 64, 129, 209])
def test_shear_squared(d):
    """[[1, e], [0, 1]] squared is [[1, 2 e], [0, 1]] exactly, also amid dense rows."""
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        for e in (1e-10, 1e-14, 1e-18, 1e-20, 1e-120, 1e-250):
            n = enough(d)
            U = torch.eye(d, dtype=torch.complex128, device="cuda").repeat(2 * n, 1, 1)
            S = np.eye(d, dtype=np.complex128)
            S[0, 1] = e
            S[2:, 2:] = np.linalg.qr(rng.normal(size=(d - 2, d - 2)) + 1j * rng.normal(size=(d - 2, d - 2)))[0]
            S[d - 1, 0] = e
            U[0] = U[1] = cuda(S)
            out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
            M.mg_propagate(ctx, 2 * n, d, U, M.MG_OUT_PROPAGATOR, None, out, 0, M.MG_PREC_FP64)
            got = out.cpu().numpy()
            assert got[0, 1] == 2 * e
            # column 0 of the dense rows: e (Q[:, last] + 1 at the last row), each a sum of one or two terms
            ref = e * S[2:, d - 1]
            ref[-1] += e
            assert np.abs(got[2:, 0] - ref).max() <= 4 * 2.0 ** -53 * e
            assert got[1, 0] == 0 and got[0, 2] == 0
    finally:
        ctx.close()


@pytest.mark.parametrize("width", [0.5, 2.0, 6.0, 20.0, 1e9])
@pytest.mark.parametrize("d", [33, 65, 129, 300])
def test_graded_operands_hold_the_bound(d, width):
    """Entries falling by 2^-(distance from the diagonal / width): tiles on either side of the
    check's line.  FP64 arithmetic keeps (2 d + 2) u M, M = |A| |B|; tiles from digits pass the
    check with a standard error below d u M, taken eightfold."""
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        fall = 2.0 ** -(np.abs(np.subtract.outer(np.arange(d), np.arange(d))) / width)
        A, B = ((rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))) * fall for _ in range(2))
        n = enough(d)
        U = torch.eye(d, dtype=torch.complex128, device="cuda").repeat(2 * n, 1, 1)
        U[0], U[1] = cuda(B), cuda(A)
        out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
        M.mg_propagate(ctx, 2 * n, d, U, M.MG_OUT_PROPAGATOR, None, out, 0, M.MG_PREC_FP64)
        C = out.cpu().numpy()
        rows = np.unique(np.linspace(0, d - 1, 40).astype(int))
        Ar, Ai, Br, Bi = (x.astype(np.longdouble) for x in (A.real[rows], A.imag[rows], B.real, B.imag))
        bound = 8 * d * 2.0 ** -53 * (np.abs(A[rows]) @ np.abs(B))
        assert np.all(np.abs((C.real[rows] - (Ar @ Br - Ai @ Bi)).astype(np.float64)) <= bound)
        assert np.all(np.abs((C.imag[rows] - (Ar @ Bi + Ai @ Br)).astype(np.float64)) <= bound)
    finally:
        ctx.close()


def expm_dense(T):
    """exp(T) by scaling and squaring of the Taylor series, entries of one size."""
    s = max(0, int(np.ceil(np.log2(np.abs(T).sum(0).max()))) + 3)
    X, R = T / 2 ** s, np.eye(len(T), dtype=T.dtype)
    term = R
    for k in range(1, 20):
        term = term @ X / k
        R = R + term
    for _ in range(s):
        R = R @ R
    return R


def weakly_coupled(rng, d, e, real):
    """Two dense blocks with couplings e V, and e times the off-diagonal block of exp(-i A) to
    first order in e (the next term is e^3)."""
    h = d // 2
    g = lambda m, n: rng.normal(size=(m, n)) + (0 if real else 1j * rng.normal(size=(m, n)))  # noqa: E731
    A1, A2, V = g(h, h), g(d - h, d - h), g(h, d - h)
    A1, A2 = (A1 + A1.conj().T) / np.sqrt(4 * h), (A2 + A2.conj().T) / np.sqrt(4 * h)
    A = np.zeros((d, d), dtype=np.complex128)
    A[:h, :h], A[h:, h:], A[:h, h:], A[h:, :h] = A1, A2, e * V, e * V.conj().T
    T = np.zeros((d, d), dtype=np.complex128)
    T[:h, :h], T[h:, h:], T[:h, h:] = A1, A2, V
    return A, e * expm_dense(-1j * T)[:h, h:]


@pytest.mark.parametrize("e", [2.0 ** -40, 2.0 ** -60])
@pytest.mark.parametrize("d", [20, 40, 130])
def test_expm_of_weakly_coupled_blocks(d, e):
    rng = np.random.default_rng(d)
    n = enough(d) if d > 32 else 3
    ctx = M.Context(0)
    try:
        A, ref = weakly_coupled(rng, d, e, False)
        U = torch.empty((n, d, d), dtype=torch.complex128, device="cuda")
        M.mg_expm(ctx, n, d, cuda(np.broadcast_to(A, (n, d, d))), U, M.MG_PREC_FP64)
        got = U.cpu().numpy()
        # ~15 products of d-term sums on either side, doubled by the squarings
        assert np.abs(got[:, :d // 2, d // 2:] - ref).max() <= 2.0 ** -53 * 200 * d * np.abs(ref).max()
    finally:
        ctx.close()


@pytest.mark.parametrize("call", ["evolve", "batch"])
def test_resumed_running_product(call):
    """U(T) in with a diagonal U and weak entries in `in`: one product term per entry."""
    rng = np.random.default_rng(5)
    d, e = 209, 1e-15
    h = rng.normal(size=d)
    inp = np.eye(d, dtype=np.complex128)
    inp[0, 1:] = e * rng.normal(size=d - 1)
    ctx = M.Context(0)
    try:
        plan = M.Plan(ctx, cuda(np.diag(h).astype(np.complex128)), None, M.MG_PREC_FP64)
        plan.set_controls(1, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((1, 1, 0), dtype=torch.float64))
        out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
        if call == "evolve":
            plan.evolve(M.MG_OUT_PROPAGATOR, cuda(inp), out)
        else:
            assert M.mg_evolve_batch(ctx, [plan], [M.MG_OUT_PROPAGATOR], [cuda(inp)], [out]) == [0]
        got = out.cpu().numpy()
        assert np.abs(got[0, 1:] - got[0, 0] * inp[0, 1:]).max() <= 8 * 2.0 ** -53 * np.abs(inp[0, 1:]).max()
        plan.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("d", [20, 40, 130, 209])
def test_every_product_when_asked_for(d, real):
    """set_fp64_entrywise: evolutions keep weak amplitudes (exponentials, tree and running products)."""
    rng = np.random.default_rng(d)
    e = 2.0 ** -50
    N = 2 * enough(d) if d > 32 else 8
    ctx = M.Context(0)
    try:
        A, ref = weakly_coupled(rng, d, e, real)
        ctx.set_fp64_entrywise(True)
        plan = M.Plan(ctx, cuda(A), None, M.MG_PREC_FP64)
        plan.set_controls(N, 1, 0.0, 1.0 / N, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
        for output in (M.MG_OUT_PROPAGATOR, M.MG_OUT_STATE):
            if output == M.MG_OUT_PROPAGATOR:
                out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
                plan.evolve(output, None, out)
                got, want = out.cpu().numpy()[:d // 2, d // 2:], ref
            else:
                psi = np.zeros(d, dtype=np.complex128)
                psi[d - 1] = 1.0
                out = torch.empty(d, dtype=torch.complex128, device="cuda")
                plan.evolve(output, cuda(psi), out)
                got, want = out.cpu().numpy()[:d // 2], ref[:, -1]
            # N intervals of ~10 products of d-term sums
            assert np.abs(got - want).max() <= 2.0 ** -53 * 200 * d * np.abs(ref).max()
        plan.close()
    finally:
        ctx.close()
