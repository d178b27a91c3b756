"""The action path's kernel for real operators (action_rows_kernel): one CTA and clusters, rows
of up to 8, 16 and 24 nonzeros, uneven jobs sharing a launch, against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import workloads as W  # noqa: E402
from paper_2411_09982_gb300 import magnus as M  # noqa: E402

JOBS = {
    "d1": lambda: W.transmon_resonator(nt=1, nr=1, N=5, T=0.5, sigma=0.2),
    "d30_one_cta": lambda: W.transmon_resonator(N=12, T=0.6, sigma=0.2),
    "d65_two_ctas": lambda: W.transmon_resonator(nt=5, nr=13, N=9, T=0.9, sigma=0.2),
    "d129": lambda: W.transmon_resonator(nt=3, nr=43, N=6, T=0.3, sigma=0.2),
    "d243_rows16": lambda: W.transmon_chain(n_sites=5, N=6, T=0.3, sigma=0.2, unitary=False),
    "d512_all_to_all": lambda: W.transmon_chain(n_sites=3, levels=8, N=4, T=0.2, sigma=0.2, all_to_all=True,
                                                two_tone=True, unitary=False),
    "d729_rows24": lambda: W.transmon_chain(n_sites=6, N=4, T=0.1, sigma=0.2, unitary=False),
}


@pytest.mark.parametrize("name", list(JOBS))
def test_rows_kernel_matches_oracle(name):
    wl = JOBS[name]()
    ctx = M.Context(0)
    try:
        ref = oracle.evolve_workload(wl)
        psi, rep = M.evolve_workload(ctx, wl, M.MG_PREC_FP64, flags=M.MG_FLAG_STATE_ACTION)
        assert np.abs(psi.cpu().numpy() - ref).max() <= 1e-11
        traj, _ = M.evolve_workload(ctx, wl, M.MG_PREC_FP64, flags=M.MG_FLAG_STATE_ACTION, trajectory=True)
        assert torch.equal(traj[-1], psi) and np.array_equal(traj[0].cpu().numpy(), wl.psi0)
    finally:
        ctx.close()


def test_uneven_jobs_share_a_launch():
    wls = [JOBS[n]() for n in JOBS]
    ctx = M.Context(0)
    try:
        plans, ins, outs = [], [], []
        for wl in wls:
            smp, w = M.node_samples(wl)
            p = M.Plan(ctx, torch.from_numpy(wl.H0).cuda(), torch.from_numpy(wl.Hk).cuda(), M.MG_PREC_FP64, 6,
                       M.MG_FLAG_STATE_ACTION)
            p.set_controls(wl.N, wl.P, wl.t0, wl.dt, w, torch.from_numpy(smp).cuda())
            plans.append(p)
            ins.append(torch.from_numpy(wl.psi0).cuda())
            outs.append(torch.empty_like(ins[-1]))
        assert M.mg_evolve_batch(ctx, plans, [M.MG_OUT_STATE] * len(plans), ins, outs) == [0] * len(plans)
        torch.cuda.synchronize()
        for wl, o in zip(wls, outs):
            assert np.abs(o.cpu().numpy() - oracle.evolve_workload(wl)).max() <= 1e-11
    finally:
        ctx.close()
