"""The state chain (csrc/propagate.cu): runs longer than the intervals read ahead, the length at
which the tree takes over, trajectories through a plan, and batches of so many states that each
gets fewer CTAs (several rounds of rows per CTA) or one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def unitary(rng, n, d):
    return np.stack([np.linalg.qr(rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d)))[0] for _ in range(n)])


@pytest.mark.parametrize("reorth", [0, 5])
@pytest.mark.parametrize("N", [1, 7, 8, 9, 17, 32, 33, 70])
@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8, 9, 32])
def test_lengths(d, N, reorth):
    rng = np.random.default_rng(100 * d + N)
    U = 1.01 * unitary(rng, N, d)
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
        M.mg_propagate(ctx, N, d, cuda(U), M.MG_OUT_STATE, cuda(psi), out, reorth)
        # N steps of d-term FP64 sums on vectors of norm ~1.01^N, through products of up to 3 intervals
        assert np.abs(out.cpu().numpy() - ref).max() <= 16 * N * (d + 2) * 2.0 ** -53 * 1.01 ** N
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [2, 30, 96, 256])
def test_trajectory_through_a_plan(d):
    rng = np.random.default_rng(d)
    N = 19
    H = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
    H = (H + H.conj().T) / np.sqrt(d)
    psi = rng.normal(size=d) + 1j * rng.normal(size=d)
    psi /= np.linalg.norm(psi)
    lam, V = np.linalg.eigh(H)
    ctx = M.Context(0)
    try:
        plan = M.Plan(ctx, cuda(H), None, M.MG_PREC_FP64)
        plan.set_controls(N, 1, 0.0, 0.1, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
        traj = torch.empty((N + 1, d), dtype=torch.complex128, device="cuda")
        plan.evolve(M.MG_OUT_TRAJECTORY, cuda(psi), traj)
        got = traj.cpu().numpy()
        for n in range(N + 1):
            ref = V @ (np.exp(-0.1j * n * lam) * (V.conj().T @ psi))
            assert np.abs(got[n] - ref).max() <= 1e-12, n
        plan.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("d,jobs", [(256, 40), (256, 200), (100, 60), (64, 180)])
def test_many_states_get_fewer_ctas_each(d, jobs):
    """Renormalised chains keep their length (no tree); clusters of 16 do not fit this often."""
    rng = np.random.default_rng(d + jobs)
    N = 6
    ctx = M.Context(0)
    try:
        base = rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d))
        base = (base + base.conj().T) / np.sqrt(d)
        lam, V = np.linalg.eigh(base)
        plans, ins, outs, refs = [], [], [], []
        for q in range(jobs):
            c = 0.2 + 0.8 * q / jobs
            p = M.Plan(ctx, cuda(c * base), None, M.MG_PREC_FP64)
            p.set_controls(N, 1, 0.0, 0.05, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
            psi = rng.normal(size=d) + 1j * rng.normal(size=d)
            psi /= np.linalg.norm(psi)
            plans.append(p)
            ins.append(cuda(psi))
            outs.append(torch.empty(d, dtype=torch.complex128, device="cuda"))
            refs.append(V @ (np.exp(-1j * c * 0.05 * N * lam) * (V.conj().T @ psi)))
        assert M.mg_evolve_batch(ctx, plans, [M.MG_OUT_STATE] * jobs, ins, outs, 4) == [0] * jobs
        for o, r in zip(outs, refs):
            assert np.abs(o.cpu().numpy() - r).max() <= 1e-12
    finally:
        ctx.close()
