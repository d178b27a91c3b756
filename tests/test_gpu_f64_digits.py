"""FP64 products from digits on the tensor cores (csrc/gemm_f64_digits.cu).

A propagator product U_1 U_0 (mg_propagate) is one such product where the batch is large
enough; the tests below fill it up with identities.  It is held, against extended precision, to the bound of 56-bit operands (every entry
of a row or column rounded to 2^-56 of the power of two above its largest entry, digit
products of level 9 and up dropped, the last level rounded to its own unit, the result
rounded to FP64); the eight base-256 digits hold 63.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


def enough(d):
    """A batch that takes the digits at dimension d."""
    return 8000000 // (-(-d // 16) * 16) ** 3 + 1


def product(ctx, A, B):
    """A B by mg_propagate: the first of enough(d) pairs, the others identities (exact)."""
    d = A.shape[0]
    U = torch.eye(d, dtype=torch.complex128, device="cuda").repeat(2 * enough(d), 1, 1)
    U[0], U[1] = torch.from_numpy(B).cuda(), torch.from_numpy(A).cuda()
    out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
    M.mg_propagate(ctx, U.shape[0], d, U, M.MG_OUT_PROPAGATOR, None, out, 0, M.MG_PREC_FP64)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def on_the_pipe(ctx, A, B):
    d = A.shape[0]
    out = torch.empty((1, d, d), dtype=torch.complex128, device="cuda")
    M.mg_cgemm(ctx, 1, d, torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda(), out, M.MG_PREC_FP64)
    torch.cuda.synchronize()
    return out.cpu().numpy()[0]


def matrices(kind, d, rng):
    g = lambda: rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))  # noqa: E731
    if kind == "gauss":
        return g(), g()
    if kind == "near_identity":
        return np.eye(d) + 1e-3 * g(), np.eye(d) + 1e-3 * g()
    if kind == "largest_digits":   # every digit of every entry at its largest: the exactness bound's worst case
        x = (127 / 128) * (1 - 2.0 ** -53)
        return np.full((d, d), x * (1 + 1j)), np.full((d, d), x * (1 - 1j))
    if kind == "largest_bytes":    # the same in base 256: 63, 127, 127, ... in units of 2^-6
        x = (63 + 127 / 255) / 64
        return np.full((d, d), x * (1 + 1j)), np.full((d, d), x * (1 - 1j))
    if kind == "scaled":           # rows of A and columns of B 2^-120 .. 2^120
        s = 2.0 ** rng.integers(-120, 121, size=d)
        return s[:, None] * g(), g() * s[None, :]
    z = g() * (rng.random((d, d)) < 0.05)   # sparse, with a zero row and a zero column
    z[d // 2] = 0.0
    w = g() * (rng.random((d, d)) < 0.05)
    w[:, d // 3] = 0.0
    return z, w


@pytest.mark.parametrize("kind", ["gauss", "near_identity", "largest_digits", "largest_bytes", "scaled", "sparse"])
@pytest.mark.parametrize("d", [33, 64, 65, 127, 129, 200, 600])
def test_product_within_its_bound(d, kind):
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        A, B = matrices(kind, d, rng)
        C = product(ctx, A, B)
        rows = np.unique([0, 1, d // 2, d - 2, d - 1])
        Ar, Ai, Br, Bi = (x.astype(np.longdouble) for x in (A.real[rows], A.imag[rows], B.real, B.imag))
        re, im = Ar @ Br - Ai @ Bi, Ar @ Bi + Ai @ Br
        ea = 2.0 ** np.ceil(np.log2(np.maximum(np.abs(A.real), np.abs(A.imag)).max(1) + 1e-300))[rows]
        eb = 2.0 ** np.ceil(np.log2(np.maximum(np.abs(B.real), np.abs(B.imag)).max(0) + 1e-300))
        sa = (np.abs(A.real) + np.abs(A.imag)).sum(1)[rows]
        sb = (np.abs(B.real) + np.abs(B.imag)).sum(0)
        # 2 ea, 2 eb: a largest entry that is itself a power of two is bounded by the next one
        bound = 2.0 ** -56 * (2 * ea[:, None] * sb[None, :] + 2 * eb[None, :] * sa[:, None])
        bound = bound + 4 * np.outer(ea, eb) * (2 * d) * 7 * 2.0 ** -63 + 4 * np.outer(ea, eb) * 2.0 ** -61
        for ref, got in ((re, C.real[rows]), (im, C.imag[rows])):
            assert np.all(np.abs((got - ref).astype(np.float64)) <= bound + 2.0 ** -53 * np.abs(ref))
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [209, 260])
@pytest.mark.parametrize("case", ["nan_a", "inf_b", "out_of_range"])
def test_operands_outside_the_digits_take_the_fp64_pipe(d, case):
    """NaN, infinities and exponents beyond 2^400 give what the FP64-pipe product gives, bit for bit."""
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        A, B = matrices("gauss", d, rng)
        if case == "nan_a":
            A[3, 5] = np.nan
        elif case == "inf_b":
            B[1, 2] = np.inf
        else:
            A, B = A * 2.0 ** 450, B * 2.0 ** -460
        got, ref = product(ctx, A, B), on_the_pipe(ctx, A, B)
        assert np.array_equal(got.view(np.float64), ref.view(np.float64), equal_nan=True)
    finally:
        ctx.close()


def test_bounded_wait_runs_out_and_context_recovers():
    """The stall test's waits give up, the call reports MG_ETIMEOUT and the outputs are not
    left looking like a result; the context then works."""
    rng = np.random.default_rng(1)
    d = 150
    H = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
    H = torch.from_numpy((H + H.conj().T) / np.sqrt(d)).cuda()
    ctx = M.Context(0)
    try:
        plan = M.Plan(ctx, H, None, M.MG_PREC_FP64)
        plan.set_controls(4, 2, 0.0, 0.25, np.ones(2), torch.zeros((4, 2, 0), dtype=torch.float64))
        out = torch.zeros((d, d), dtype=torch.complex128, device="cuda")
        ctx.set_wait_limit(0.002, stall_test=True)
        with pytest.raises(M.MagnusError) as e:
            plan.evolve(M.MG_OUT_PROPAGATOR, None, out)
        assert e.value.code == M.MG_ETIMEOUT
        assert not torch.isfinite(torch.view_as_real(out)).all()
        ctx.set_wait_limit(4.0, stall_test=False)
        plan.evolve(M.MG_OUT_PROPAGATOR, None, out)
        lam, V = np.linalg.eigh(H.cpu().numpy())
        ref = (V * np.exp(-1j * lam)) @ V.conj().T
        assert np.abs(out.cpu().numpy() - ref).max() <= 1e-11
        plan.close()
    finally:
        ctx.close()


def symmetric(rng, d, norm):
    A = rng.normal(size=(d, d))
    A = A + A.T
    A *= norm / np.abs(A - np.trace(A) / d * np.eye(d)).sum(0).max()
    return A.astype(np.complex128)


def exact_exp(A):
    lam, V = np.linalg.eigh(A.real)
    return (V * np.exp(-1j * lam)) @ V.T


@pytest.mark.parametrize("d", [33, 64, 97, 128, 129, 257, 400])
def test_real_symmetric_exponentials(d):
    """Cosine and sine form over every Taylor degree (norms 1e-9 .. 30: degrees 2 to 16, squarings)."""
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        for norm in (1e-9, 1e-5, 1e-2, 0.08, 0.3, 0.7, 3.0, 30.0):
            A = symmetric(rng, d, norm)
            N = enough(d)
            plan = M.Plan(ctx, torch.from_numpy(A).cuda(), None, M.MG_PREC_FP64)
            plan.set_controls(N, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
            out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
            rep = plan.evolve(M.MG_OUT_PROPAGATOR, None, out)
            # ~20 products of d-term sums, their errors doubled by every squaring (2^s <= 4 norm),
            # in each of the N equal intervals
            tol = N * 2.0 ** -53 * 20 * d * (1 + 4 * norm)
            assert np.abs(out.cpu().numpy() - exact_exp(N * A)).max() <= tol, (norm, rep)
            plan.close()
    finally:
        ctx.close()


def test_batch_of_real_exponents_with_uneven_squarings():
    rng = np.random.default_rng(3)
    ctx = M.Context(0)
    try:
        As = [symmetric(rng, d, norm) for d, norm in ((40, 0.1), (45, 40.0), (48, 2.0), (70, 5.0), (33, 1e-3))]
        plans, outs = [], []
        for A in As:
            p = M.Plan(ctx, torch.from_numpy(A).cuda(), None, M.MG_PREC_FP64)
            p.set_controls(90, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((90, 1, 0), dtype=torch.float64))
            plans.append(p)
            outs.append(torch.empty(A.shape, dtype=torch.complex128, device="cuda"))
        assert M.mg_evolve_batch(ctx, plans, [M.MG_OUT_PROPAGATOR] * 5, [None] * 5, outs) == [0] * 5
        torch.cuda.synchronize()
        for A, o in zip(As, outs):
            norm = np.abs(A - np.trace(A) / len(A) * np.eye(len(A))).sum(0).max()
            assert np.abs(o.cpu().numpy() - exact_exp(90 * A)).max() <= 90 * 2.0 ** -53 * 20 * 80 * (1 + 4 * norm)
    finally:
        ctx.close()
