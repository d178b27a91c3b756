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
