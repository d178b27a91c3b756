"""FP64 products from digits (csrc/gemm_f64_digits.cu) with marked items -- operands outside the
digits' range, whose products run in FP64 arithmetic -- among unmarked ones.

mg_expm takes batches whose first items are 2^-450 times a matrix: their first powers are
marked, and exp(-i A) is the identity to 1e-130."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


def hermitian(rng, n, d, norm):
    A = rng.normal(size=(n, d, d)) + 1j * rng.normal(size=(n, d, d))
    A = A + A.conj().transpose(0, 2, 1)
    return A * (norm / np.abs(A).sum(1).max())


def exact(A):
    lam, V = np.linalg.eigh(A)
    return (V * np.exp(-1j * lam)[..., None, :]) @ V.conj().swapaxes(-1, -2)


def expm(ctx, A):
    U = torch.empty(A.shape, dtype=torch.complex128, device="cuda")
    M.mg_expm(ctx, A.shape[0], A.shape[1], torch.from_numpy(A).cuda(), U, M.MG_PREC_FP64)
    torch.cuda.synchronize()
    return U.cpu().numpy()


def test_unfinished_marked_items_do_not_keep_older_values():
    """The stall test's waits give up in every CTA: a marked item's entries are then right or
    NaN, never what an earlier call left in the workspace."""
    rng = np.random.default_rng(0)
    n, d = 60, 150
    A = hermitian(rng, n, d, 2.0)
    ctx = M.Context(0)
    try:
        expm(ctx, A)   # finite values in every buffer
        B = 4e-9 * A   # norms of 8e-9: degree 2, I + X + X X / 2, one product
        B[1::2] *= 2.0 ** -450
        ctx.set_wait_limit(0.002, stall_test=True)
        U = expm(ctx, B)
        ctx.set_wait_limit(4.0, stall_test=False)
        assert not np.isfinite(U[0::2]).all()
        marked = U[1::2]
        stale = np.isfinite(marked) & (np.abs(marked - np.eye(d)) > 1e-7)
        assert not stale.any(), int(stale.sum())
    finally:
        ctx.close()


def test_marked_items_do_not_run_out_the_waits_of_the_others():
    """A limit of 3 ms, no stall: marked items take their time on the FP64 pipe, and the other
    items' products finish (their waits are for loads and products of their own)."""
    rng = np.random.default_rng(1)
    n, d = 6, 700
    A = hermitian(rng, n, d, 1.5)
    A[:2] *= 2.0 ** -450
    ctx = M.Context(0)
    try:
        ctx.set_wait_limit(0.003)
        U = expm(ctx, A)
        assert np.abs(U[:2] - np.eye(d)).max() <= 1e-14
        # ~10 products of d-term sums
        assert np.abs(U[2:] - exact(A[2:])).max() <= 2.0 ** -53 * 20 * d
    finally:
        ctx.close()


def test_subnormal_rows_and_columns_take_fp64_arithmetic():
    """A row of A (a column of B) with nothing but subnormal entries is not a zero one."""
    rng = np.random.default_rng(2)
    d = 64
    n = 8000000 // d ** 3 + 1
    ctx = M.Context(0)
    try:
        for side in (0, 1):
            A, B = (rng.normal(size=(2, d, d)) + 1j * rng.normal(size=(2, d, d)))
            if side == 0:
                A[5] *= 2.0 ** -1060
                B *= 2.0 ** 300
            else:
                B[:, 5] *= 2.0 ** -1060
                A *= 2.0 ** 300
            U = torch.eye(d, dtype=torch.complex128, device="cuda").repeat(2 * n, 1, 1)
            U[0], U[1] = torch.from_numpy(B).cuda(), torch.from_numpy(A).cuda()
            out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
            M.mg_propagate(ctx, 2 * n, d, U, M.MG_OUT_PROPAGATOR, None, out, 0, M.MG_PREC_FP64)
            ref = torch.empty((1, d, d), dtype=torch.complex128, device="cuda")
            M.mg_cgemm(ctx, 1, d, U[1:2].contiguous(), U[0:1].contiguous(), ref, M.MG_PREC_FP64)
            torch.cuda.synchronize()
            assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref[0]))
            assert (ref[0].abs() > 0).all()
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [33, 130])
def test_tiny_real_symmetric_exponents_keep_their_bits(d):
    """exp(-i A) of a real symmetric A of 2^-450: entry by entry I - i A."""
    rng = np.random.default_rng(3)
    n = 8000000 // (-(-d // 16) * 16) ** 3 + 1
    A = rng.normal(size=(d, d))
    A = (A + A.T) * 2.0 ** -450
    ctx = M.Context(0)
    try:
        plan = M.Plan(ctx, torch.from_numpy(A.astype(np.complex128)).cuda(), None, M.MG_PREC_FP64)
        plan.set_controls(n, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((n, 1, 0), dtype=torch.float64))
        psi = np.zeros(d, dtype=np.complex128)
        psi[3] = 1.0
        traj = torch.empty((n + 1, d), dtype=torch.complex128, device="cuda")
        plan.evolve(M.MG_OUT_TRAJECTORY, torch.from_numpy(psi).cuda(), traj)
        got = traj[1].cpu().numpy()
        off = np.arange(d) != 3
        assert np.abs(got[off].imag + A[off, 3]).max() <= 1e-14 * np.abs(A).max()
        plan.close()
    finally:
        ctx.close()
