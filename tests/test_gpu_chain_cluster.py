"""The state chain on thread-block clusters (d <= 256, csrc/propagate.cu) against plain
matrix-vector steps: one CTA and every cluster size's edges, trajectories, renormalisation."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


@pytest.mark.parametrize("reorth", [0, 3])
@pytest.mark.parametrize("d", [1, 2, 7, 31, 32, 33, 48, 49, 64, 65, 96, 97, 129, 193, 255, 256])
def test_chain_matches_matrix_vector_steps(d, reorth):
    rng = np.random.default_rng(d)
    N = 7
    U = np.stack([np.linalg.qr(rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d)))[0] for _ in range(N)])
    U *= 1.01   # the renormalisation has something to do
    psi = rng.normal(size=d) + 1j * rng.normal(size=d)
    psi /= np.linalg.norm(psi)
    ref = psi
    for n in range(N):
        ref = U[n] @ ref
        if reorth and (n + 1) % reorth == 0:
            ref = ref / np.linalg.norm(ref)
    ctx = M.Context(0)
    try:
        out = torch.empty(d, dtype=torch.complex128, device="cuda")
        M.mg_propagate(ctx, N, d, torch.from_numpy(U).cuda(), M.MG_OUT_STATE, torch.from_numpy(psi).cuda(), out, reorth)
        torch.cuda.synchronize()
        # N steps of d-term FP64 sums on vectors of norm ~1
        assert np.abs(out.cpu().numpy() - ref).max() <= 4 * N * d * 2.0 ** -53
    finally:
        ctx.close()
