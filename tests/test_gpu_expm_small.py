"""FP64 exponentials of d <= 32 in one launch (csrc/expm_small.cu) against the
eigendecomposition, over every Taylor degree (norms from 1e-9 up) and the size edges:
real symmetric exponents (cosine and sine) through a plan, complex Hermitian ones through
mg_expm, batches with per-interval squaring counts through mg_evolve_batch."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402

NORMS = [0.0, 1e-9, 1e-5, 1e-2, 0.08, 0.3, 0.7, 3.0, 60.0]


def tol(d, norm):
    # ~20 products of d-term sums, their errors doubled by every squaring (2^s <= 4 norm)
    return 2.0 ** -53 * 20 * d * (1.0 + 4.0 * norm)


def hermitian(rng, d, norm, real):
    A = rng.normal(size=(d, d)) + (0 if real else 1j * rng.normal(size=(d, d)))
    A = (A + A.conj().T).astype(np.complex128)
    n1 = np.abs(A - np.trace(A) / d * np.eye(d)).sum(0).max()
    return A * (norm / n1 if n1 > 0 else norm)


def exact(A):
    lam, V = np.linalg.eigh(A)
    return (V * np.exp(-1j * lam)) @ V.conj().T


@pytest.mark.parametrize("d", [1, 2, 5, 16, 31, 32])
def test_real_symmetric_plan(d):
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        for norm in NORMS:
            A = hermitian(rng, d, norm, True)
            plan = M.Plan(ctx, torch.from_numpy(A).cuda(), None, M.MG_PREC_FP64)
            plan.set_controls(1, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((1, 1, 0), dtype=torch.float64))
            out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
            rep = plan.evolve(M.MG_OUT_PROPAGATOR, None, out)
            assert np.abs(out.cpu().numpy() - exact(A)).max() <= tol(d, norm), (norm, rep)
            plan.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [1, 2, 5, 16, 31, 32])
def test_complex_hermitian_batch(d):
    rng = np.random.default_rng(100 + d)
    ctx = M.Context(0)
    try:
        for norm in NORMS:
            A = np.stack([hermitian(rng, d, norm, False) for _ in range(3)])
            U = torch.empty((3, d, d), dtype=torch.complex128, device="cuda")
            M.mg_expm(ctx, 3, d, torch.from_numpy(A).cuda(), U, M.MG_PREC_FP64)
            torch.cuda.synchronize()
            for a, u in zip(A, U.cpu().numpy()):
                assert np.abs(u - exact(a)).max() <= tol(d, norm), norm
    finally:
        ctx.close()


@pytest.mark.parametrize("real", [True, False])
def test_batch_with_uneven_squarings(real):
    rng = np.random.default_rng(7)
    ctx = M.Context(0)
    try:
        As = [hermitian(rng, d, norm, real) for d, norm in ((17, 0.1), (20, 40.0), (32, 2.0), (30, 1e-3))]
        plans, outs = [], []
        for A in As:
            p = M.Plan(ctx, torch.from_numpy(A).cuda(), None, M.MG_PREC_FP64)
            p.set_controls(2, 1, 0.0, 0.5, np.array([2.0]), torch.zeros((2, 1, 0), dtype=torch.float64))
            plans.append(p)
            outs.append(torch.empty(A.shape, dtype=torch.complex128, device="cuda"))
        st = M.mg_evolve_batch(ctx, plans, [M.MG_OUT_PROPAGATOR] * 4, [None] * 4, outs)
        torch.cuda.synchronize()
        assert st == [0] * 4
        for A, o in zip(As, outs):
            norm = np.abs(A - np.trace(A) / len(A) * np.eye(len(A))).sum(0).max()
            assert np.abs(o.cpu().numpy() - exact(A)).max() <= tol(32, norm)
    finally:
        ctx.close()
