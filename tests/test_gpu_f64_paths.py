"""MG_PREC_FP64 beside its results: the structure option, the counted work, the error of a product
from digits at the 63 bits it holds, and per-interval squaring counts of complex operators."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09982_gb300 import magnus as M  # noqa: E402


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def enough(d):
    return 8000000 // (-(-d // 16) * 16) ** 3 + 1


def hermitian(rng, d, norm, real):
    A = rng.normal(size=(d, d)) + (0 if real else 1j * rng.normal(size=(d, d)))
    A = (A + A.conj().T).astype(np.complex128)
    return A * (norm / np.abs(A - np.trace(A) / d * np.eye(d)).sum(0).max())


def exact(A):
    lam, V = np.linalg.eigh(A)
    return (V * np.exp(-1j * lam)) @ V.conj().T


def one_plan(ctx, A, N, prec=M.MG_PREC_FP64):
    plan = M.Plan(ctx, cuda(A), None, prec)
    plan.set_controls(N, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
    return plan


@pytest.mark.parametrize("d", [33, 64, 129, 300])
def test_product_holds_63_bits(d):
    """A product of Gaussian matrices against extended precision.  Rounding each entry to 2^-63 of
    its row's or column's scale 2^E and leaving out the digit pairs s + t >= 8 (7 of them at
    s + t = 8, digits of RMS 74) are random: sigma = sqrt(d) 2^-61 2^(Ea + Eb) for the sum over
    2 d terms.  Eight of them (some 1e4 entries) beside the rounding of the result; without the
    last digit the error would be 150 times sigma."""
    rng = np.random.default_rng(d)
    ctx = M.Context(0)
    try:
        A, B = (rng.normal(size=(d, d)) + 1j * rng.normal(size=(d, d)) for _ in range(2))
        U = torch.eye(d, dtype=torch.complex128, device="cuda").repeat(2 * enough(d), 1, 1)
        U[0], U[1] = cuda(B), cuda(A)
        out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
        M.mg_propagate(ctx, U.shape[0], d, U, M.MG_OUT_PROPAGATOR, None, out, 0, M.MG_PREC_FP64)
        C = out.cpu().numpy()
        rows = np.unique(np.linspace(0, d - 1, 30).astype(int))
        Ar, Ai, Br, Bi = (x.astype(np.longdouble) for x in (A.real[rows], A.imag[rows], B.real, B.imag))
        re, im = Ar @ Br - Ai @ Bi, Ar @ Bi + Ai @ Br
        scale = lambda x, axis: 2.0 ** (np.floor(np.log2(np.maximum(abs(x.real), abs(x.imag)).max(axis))) + 1)  # noqa: E731
        sigma = np.sqrt(d) * 2.0 ** -61 * np.outer(scale(A, 1)[rows], scale(B, 0))
        for ref, got in ((re, C.real[rows]), (im, C.imag[rows])):
            assert np.all(np.abs((got - ref).astype(np.float64)) <= 2.0 ** -53 * np.abs(ref) + 8 * sigma)
    finally:
        ctx.close()


def test_batch_of_complex_exponents_with_uneven_squarings():
    """Per-interval squaring counts, complex products from digits (d > 32)."""
    rng = np.random.default_rng(11)
    N = 90
    ctx = M.Context(0)
    try:
        As = [hermitian(rng, d, norm, False) for d, norm in ((40, 0.1), (45, 40.0), (48, 2.0), (70, 5.0), (33, 1e-3))]
        plans = [one_plan(ctx, A, N) for A in As]
        outs = [torch.empty(A.shape, dtype=torch.complex128, device="cuda") for A in As]
        assert M.mg_evolve_batch(ctx, plans, [M.MG_OUT_PROPAGATOR] * 5, [None] * 5, outs) == [0] * 5
        for A, o in zip(As, outs):
            norm = np.abs(A - np.trace(A) / len(A) * np.eye(len(A))).sum(0).max()
            # N intervals of ~20 products of d-term sums, doubled by every squaring
            assert np.abs(o.cpu().numpy() - exact(N * A)).max() <= N * 2.0 ** -53 * 20 * 80 * (1 + 4 * norm)
    finally:
        ctx.close()


@pytest.mark.parametrize("d", [20, 40, 130])
def test_structure_option_issues_products_in_full(d):
    """Structure 0: complex products of 8 d^3 each; 3: the real symmetric form, fewer; the same U."""
    rng = np.random.default_rng(d)
    N = enough(d) if d > 32 else 4
    A = hermitian(rng, d, 3.0, True)
    ctx = M.Context(0)
    try:
        outs, flops = [], []
        for mode in (0, 1, 2, 3):
            ctx.set_structure(mode)
            ctx.enable_gemm_timing(True)
            ctx.gemm_stats(reset=True)
            plan = one_plan(ctx, A, N)
            psi = np.eye(d)[0].astype(np.complex128)
            traj = torch.empty((N + 1, d), dtype=torch.complex128, device="cuda")   # a trajectory takes no products beside the exponentials'
            rep = plan.evolve(M.MG_OUT_TRAJECTORY, cuda(psi), traj)
            flops.append(ctx.gemm_stats()["flops"] / (8.0 * d ** 3 * rep["matrix_products"]))
            outs.append(traj[1].cpu().numpy())
            plan.close()
        assert abs(flops[0] - 1) <= 1e-12 and abs(flops[1] - 1) <= 1e-12 and flops[2] < 0.6 and flops[3] == flops[2]
        for o in outs:
            assert np.abs(o - exact(A)[:, 0]).max() <= 2.0 ** -53 * 20 * d * 13
        assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[2], outs[3])
    finally:
        ctx.close()


@pytest.mark.parametrize("prec", ["fp64", "split"])
@pytest.mark.parametrize("real", [True, False])
@pytest.mark.parametrize("d", [32, 48])   # a batch pads d to a multiple of 16
def test_batch_counts_the_work_that_an_evolution_counts(d, real, prec):
    """The squarings of a batch are counted on the device, those of mg_evolve on the host."""
    rng = np.random.default_rng(d)
    N = 2 * enough(d) if d > 32 else 8
    A = hermitian(rng, d, 5.0, real)
    ctx = M.Context(0)
    try:
        ctx.enable_gemm_timing(True)
        plan = one_plan(ctx, A, N, M.MG_PREC_FP64 if prec == "fp64" else M.MG_PREC_SPLIT)
        flops = []
        for batch in (False, True):
            ctx.gemm_stats(reset=True)
            out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
            if batch:
                assert M.mg_evolve_batch(ctx, [plan], [M.MG_OUT_PROPAGATOR], [None], [out]) == [0]
            else:
                plan.evolve(M.MG_OUT_PROPAGATOR, None, out, report=False)
            flops.append(ctx.gemm_stats()["flops"])
        assert abs(flops[1] / flops[0] - 1) <= 1e-12
        plan.close()
    finally:
        ctx.close()


@pytest.mark.parametrize("case", ["reorth", "report"])
def test_workspace_stays_within_its_limit(case):
    """Split precision with two slices: the FP64 digits of re-orthonormalisation and of the
    report's product are four times its own operands'.  The context's pool (device memory taken
    during the call) holds no more than the limit and 2 MiB of rounding per buffer."""
    rng = np.random.default_rng(0)
    d, N = 1024, 24 if case == "reorth" else 2
    md = 16 * d * d
    limit = 260 * md if case == "reorth" else 25 * md
    A = hermitian(rng, d, 1.0, False)

    def taken(N, reorth, limit):
        ctx = M.Context(0, workspace_limit=limit)
        plan = M.Plan(ctx, cuda(A), None, M.MG_PREC_SPLIT, 2)
        plan.set_controls(N, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
        out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        plan.evolve(M.MG_OUT_PROPAGATOR, None, out, reorth)
        used = before - torch.cuda.mem_get_info()[0]
        plan.close()
        ctx.close()
        return used

    taken(2, 2, limit)   # loads every kernel of the path
    assert taken(N, 2 if case == "reorth" else 0, limit) <= limit + 20 * (2 << 20)


def test_fp64_chunks_without_digits_are_not_cut_for_them():
    """64 products of d = 40 run on the FP64 pipe: a limit that fits 64 intervals without digits
    runs them in one chunk, as any larger one."""
    rng = np.random.default_rng(0)
    d, N = 40, 64
    A = hermitian(rng, d, 1.0, False)
    launches = []
    for limit in (1 << 30, N * 10 * 16 * d * d):
        ctx = M.Context(0, workspace_limit=limit)
        plan = one_plan(ctx, A, N)
        out = torch.empty((d, d), dtype=torch.complex128, device="cuda")
        before = M.mg_kernel_launch_count()
        plan.evolve(M.MG_OUT_PROPAGATOR, None, out)
        launches.append(M.mg_kernel_launch_count() - before)
        plan.close()
        ctx.close()
    assert launches[0] == launches[1]


def test_captured_batch_takes_the_products_of_the_run_before_it():
    """Re-orthonormalised propagators of d = 64 beside states of d = 128, two slices: by the time
    of the capture the second group has grown the operand slots, which must not change the first
    group's FP64 products (how many at a time, and so whether from digits)."""
    rng = np.random.default_rng(4)
    ctx = M.Context(0, stream=torch.cuda.Stream())   # the default stream cannot be captured
    try:
        plans, outs, ins, kinds = [], [], [], []
        for d, N, kind in ((64, 70, M.MG_OUT_PROPAGATOR), (128, 200, M.MG_OUT_STATE)):
            p = M.Plan(ctx, cuda(hermitian(rng, d, 0.5, False)), None, M.MG_PREC_SPLIT, 2)
            p.set_controls(N, 1, 0.0, 1.0, np.array([2.0]), torch.zeros((N, 1, 0), dtype=torch.float64))
            plans.append(p)
            kinds.append(kind)
            shape = (d, d) if kind == M.MG_OUT_PROPAGATOR else (d,)
            outs.append(torch.empty(shape, dtype=torch.complex128, device="cuda"))
            ins.append(None if kind == M.MG_OUT_PROPAGATOR else cuda(np.eye(d)[0].astype(np.complex128)))
        torch.cuda.synchronize()
        g = M.BatchGraph(ctx, plans, kinds, ins, outs, 2)
        g.launch()
        torch.cuda.synchronize()
        got = [o.clone() for o in outs]
        g.close()
        assert M.mg_evolve_batch(ctx, plans, kinds, ins, outs, 2) == [0, 0]
        torch.cuda.synchronize()
        for a, b in zip(got, outs):
            assert torch.equal(a, b)
    finally:
        ctx.close()
