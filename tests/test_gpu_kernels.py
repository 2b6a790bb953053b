"""Kernels at the sizes where their tiling can go wrong, against the FP64 oracle.

Tolerances (relative, coefficient 2-norm) follow tests/test_gpu_parity.py:
FP64 and double-float components 1e-12 (sums of at most some thousand terms
in another order, double-float carrying 48 bits), FP32 1e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.index_set import IndexSet as OIndex  # noqa: E402
from oracle.krylov import krylov_expv  # noqa: E402
from oracle.operator import (DIRICHLET0, PERIODIC, cross_blocks_1d, sipg_1d,  # noqa: E402
                             sparse_matvec, sparse_matvec_general)
from oracle.reaction import Reaction  # noqa: E402
from paper_1810_11111_gb300 import sgkiif, workloads  # noqa: E402
from paper_1810_11111_gb300.runner import Problem  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


def dev(x, dtype=torch.float64):
    return torch.as_tensor(np.asarray(x), dtype=dtype, device="cuda").contiguous()


@pytest.fixture(scope="module", params=[sgkiif.SGK_FP64, sgkiif.SGK_MIXED], ids=["fp64", "mixed"])
def ctx(request):
    c = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, request.param)
    yield c
    c.close()


@pytest.mark.parametrize("d,n,k,pairs,bc", [
    (2, 0, 2, [(0, 1)], PERIODIC),            # one tuple
    (2, 1, 3, [(0, 1)], DIRICHLET0),
    (3, 5, 1, [(0, 2)], PERIODIC),            # a direction between the pair
    (3, 4, 3, [(1, 2)], DIRICHLET0),          # a direction before the pair
    (4, 3, 2, [(0, 1), (1, 3)], PERIODIC),    # directions after and between
    (5, 2, 1, [(0, 4), (2, 3)], DIRICHLET0),
])
def test_mixed_derivative_rows(ctx, d, n, k, pairs, bc):
    K = np.diag(np.linspace(1.0, 0.6, d))
    for i, j in pairs:
        K[i, j] = K[j, i] = 0.2 + 0.05 * j
    idx = sgkiif.IndexSet(ctx, d, n, k)
    op = sgkiif.Operator(ctx, idx, K, bc)
    P, E = cross_blocks_1d(n, k, bc)
    dtype, tol = ((torch.float64, 1e-12) if ctx.precision == sgkiif.SGK_FP64 else (torch.float32, 1e-5))
    xd = dev(np.random.default_rng(d + n).standard_normal(idx.dof), dtype)
    yd = torch.empty_like(xd)
    op.matvec(xd.data_ptr(), yd.data_ptr(), ctx.precision)
    torch.cuda.synchronize()
    want = sparse_matvec_general(OIndex(d, n, k), sipg_1d(n, k, bc), P, E, K, xd.double().cpu().numpy())
    assert rel(yd.double().cpu().numpy(), want) <= tol
    op.close()
    idx.close()


CUBIC = [[(-2.0, (3,)), (0.7, (2,)), (-0.3, (0,))]]
QUADRATIC = [[(1.5, (2,)), (-0.4, (1,))]]
PAIR = [[(0.1, (0, 0)), (-1.0, (1, 0)), (1.0, (2, 1)), (0.4, (0, 3))],
        [(0.9, (0, 0)), (-1.0, (2, 1)), (0.6, (1, 2)), (-0.2, (0, 1))]]
# every shape of the fused last-direction pass (d, k, reaction) with levels at
# which its stages differ: one split only, partial and full subtrees, several
# pencils and several stages per CTA, levels whose cells outnumber the threads
FUSED = [(2, 1, CUBIC, (1, 2, 5, 9)), (2, 2, CUBIC, (1, 3, 6)), (2, 3, CUBIC, (1, 2, 4, 8)),
         (2, 1, PAIR, (1, 4)), (2, 2, PAIR, (1, 3, 8)), (2, 3, PAIR, (1, 2, 5)),
         (2, 1, QUADRATIC, (1, 6)), (2, 2, QUADRATIC, (1, 4, 7)), (2, 3, QUADRATIC, (2, 5)),
         (3, 1, CUBIC, (1, 2, 5)), (3, 2, CUBIC, (1, 2, 3, 5)), (3, 3, CUBIC, (1, 3, 4)),
         (3, 1, PAIR, (1, 4)), (3, 2, PAIR, (1, 2, 4)), (3, 3, PAIR, (1, 3)),
         (3, 1, QUADRATIC, (1, 3)), (3, 2, QUADRATIC, (2, 4)),
         (4, 1, CUBIC, (1, 2, 4)), (4, 2, CUBIC, (1, 3)), (4, 1, PAIR, (1, 3))]


@pytest.mark.parametrize("d,k,rx,n", [(d, k, rx, n) for d, k, rx, levels in FUSED for n in levels])
def test_fused_reaction_shapes(ctx, d, k, rx, n):
    S = len(rx)
    idx = sgkiif.IndexSet(ctx, d, n, k)
    ops = [sgkiif.Operator(ctx, idx, [1.0] * d) for _ in range(S)]
    sol = sgkiif.Solver(ctx, ops, rx, 5, 0.01)
    rng = np.random.default_rng(n)
    U = [0.5 * (np.arange(idx.dof) == 0) + 0.3 * rng.standard_normal(idx.dof) / np.sqrt(idx.dof) for _ in range(S)]
    W = [rng.standard_normal(idx.dof) for _ in range(S)]
    Ud, Wd = dev(np.concatenate(U)), dev(np.concatenate(W))
    Fd, Jd = torch.empty_like(Ud), torch.empty_like(Ud)
    sol.reaction_eval(Ud.data_ptr(), Fd.data_ptr())
    sol.jacobian_apply(Ud.data_ptr(), Wd.data_ptr(), Jd.data_ptr())
    torch.cuda.synchronize()
    R = Reaction(OIndex(d, n, k), rx)
    assert rel(Fd.cpu().numpy(), np.concatenate(R.F(U))) <= 1e-12
    assert rel(Jd.cpu().numpy(), np.concatenate(R.J(U, W))) <= (1e-12 if ctx.precision == sgkiif.SGK_FP64 else 1e-5)
    sol.close()
    for o in ops:
        o.close()
    idx.close()


@pytest.mark.parametrize("d,n,k,M,skip", [
    (2, 0, 2, 12, 0),   # one tuple of 9 coefficients: the projection ends in a breakdown
    (2, 1, 2, 20, 1),   # 27 coefficients, the vector 8 bytes off a 16-byte boundary
    (2, 3, 1, 31, 0), (2, 3, 1, 32, 1), (2, 4, 1, 33, 0),   # the columns of one warp, one more
    (3, 3, 2, 70, 0),   # columns read in two rounds
    (2, 9, 3, 3, 0),    # few columns on long slices
])
def test_krylov_projection_edges(ctx, d, n, k, M, skip):
    # exp(dt A) v with dt small enough for the projection to be converged,
    # where it does not depend on how the basis was rounded: 1e-10 as for the
    # other exponentials, 1e-9 with the double-float matvec
    idx = sgkiif.IndexSet(ctx, d, n, k)
    kap = [1.0, 0.5, 0.1][:d]
    op = sgkiif.Operator(ctx, idx, kap)
    dt = 1e-9 if M < 10 else 1e-4
    sol = sgkiif.Solver(ctx, [op], [[]], M, dt)
    v = np.random.default_rng(M).standard_normal(idx.dof)
    held = dev(np.concatenate([np.zeros(skip), v]))
    vd = held[skip:]
    wd = torch.empty(idx.dof, dtype=torch.float64, device="cuda")
    sol.krylov_expv(0, vd.data_ptr(), wd.data_ptr())
    ref, S = OIndex(d, n, k), sipg_1d(n, k)
    want, _ = krylov_expv(lambda x: sparse_matvec(ref, S, kap, x), v, dt, M)
    assert rel(wd.cpu().numpy(), want) <= (1e-10 if ctx.precision == sgkiif.SGK_FP64 else 1e-9)
    sol.close()
    op.close()
    idx.close()


@pytest.mark.parametrize("d,n,k,M,bc", [(2, 1, 1, 9, PERIODIC), (2, 6, 2, 12, DIRICHLET0), (3, 4, 2, 35, PERIODIC),
                                        (4, 2, 1, 20, DIRICHLET0)])
def test_krylov_projection_mixed_derivatives(ctx, d, n, k, M, bc, monkeypatch):
    # one list of all entries per output in the persistent kernel, against the
    # sequence of launches (the same sums in another order) and the oracle;
    # FP64 matvecs in both modes
    K = np.diag(np.linspace(1.0, 0.6, d)) + 0.1 * (np.eye(d, k=1) + np.eye(d, k=-1))
    idx = sgkiif.IndexSet(ctx, d, n, k)
    op = sgkiif.Operator(ctx, idx, K, bc)
    v = np.random.default_rng(n).standard_normal(idx.dof)
    vd = dev(v)
    dt, got = 1e-5, []
    for off in (False, True):
        if off:
            monkeypatch.setenv("SGK_NO_PERSISTENT", "1")
        sol = sgkiif.Solver(ctx, [op], [[]], M, dt)
        wd = torch.empty_like(vd)
        sol.krylov_expv(0, vd.data_ptr(), wd.data_ptr())
        got.append(wd.cpu().numpy())
        sol.close()
    P, E = cross_blocks_1d(n, k, bc)
    ref, S = OIndex(d, n, k), sipg_1d(n, k, bc)
    want, _ = krylov_expv(lambda x: sparse_matvec_general(ref, S, P, E, K, x), v, dt, M)
    assert rel(got[0], want) <= 1e-10 and rel(got[1], want) <= 1e-10
    assert rel(got[0], got[1]) <= 1e-12
    op.close()
    idx.close()


@pytest.mark.parametrize("n,k", [(0, 2), (1, 2), (3, 1), (3, 2)])  # n = 0: 27 values, an odd count
@pytest.mark.parametrize("scheme", [sgkiif.SGK_IIF2, sgkiif.SGK_IIF3], ids=["graph", "host"])
def test_mixed_corrections_use_the_current_state(n, k, scheme):
    # the FP32 copy of the transformed state behind a mixed correction: a
    # stale one only costs corrections.  Both modes stop at 1e-12 of the
    # stage's scale; against FP64 the FP32 first residual may cost one
    # correction a step and the inner tolerance of 1e-6 one more.
    cfg = dict(workloads.cubic3d(n=n, k=k), scheme=scheme)
    steps, out, its = 3, {}, {}
    for prec in (sgkiif.SGK_FP64, sgkiif.SGK_MIXED):
        prob = Problem(cfg, prec)
        prob.reset()
        U0 = np.random.default_rng(5).standard_normal(prob.U0[0].numel())
        prob.solver.set_state(0, U0 / np.linalg.norm(U0))
        prob.solver.step(steps)
        out[prec] = prob.state()[0]
        its[prec] = prob.solver.stats()["newton_iters"]
        prob.close()
    assert rel(out[sgkiif.SGK_MIXED], out[sgkiif.SGK_FP64]) <= 1e-10
    assert its[sgkiif.SGK_MIXED] <= its[sgkiif.SGK_FP64] + 2 * steps


# Three heat steps whose unconverged projections amplify a rounding: the
# largest coefficients, recorded before the sums of the persistent Arnoldi
# kernel were first rearranged.  Another order of one of its sums moves them by
# 1e-8 to 1e-5, so 1e-9 holds the order (slices, and so sums, go by the number
# of SMs).
WAVES = np.array([[1, 2, 1], [2, 1, 3], [3, 3, 2], [1, 1, 2]], np.int32)
KINDS = np.array([[0, 1, 0], [1, 0, 0], [0, 0, 1], [1, 1, 0]], np.int32)
AMPLIFIED = [
    (3, 3, 3, 20, 0.005, sgkiif.SGK_MIXED, slice(0, 4),
     {41: -0.003271583982073906, 43: -0.0030994131983151717, 105: 0.006966140093553048,
      529: 0.003479553274309175, 531: -0.0027540474380408127, 537: -0.0019932718917509726,
      561: -0.0027540474380408383, 563: 0.0021529999571539616}),
    (3, 3, 3, 20, 0.005, sgkiif.SGK_MIXED, slice(1, 2),
     {37: -5.764616895548291e-06, 1285: -1.2965191226569354e-05, 1287: 7.323860043138634e-06,
      1293: 1.1716066326707738e-05, 1295: -7.157901932217996e-06, 1317: 7.684680082379417e-06,
      1319: -4.149563333670409e-06, 1325: -6.65949686508748e-06}),
    (3, 5, 1, 40, 0.0025, sgkiif.SGK_FP64, slice(0, 4),
     {1025: -0.01369145403862061, 1033: -0.023429195143054637, 1041: 0.011077942307921348,
      1043: 0.011077942307921416, 1056: -0.00899816104998158, 1058: 0.008978195831283849,
      1060: -0.0089781958312839, 1062: 0.008998161049981633})]


@pytest.mark.parametrize("d,n,k,M,dt,prec,modes,want", AMPLIFIED, ids=["mixed", "mixed_one_mode", "fp64"])
def test_order_of_sums_of_the_projection(d, n, k, M, dt, prec, modes, want):
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded on 152 SMs")
    with_amp = np.array([0.7, -0.4, 0.5, 0.9])[modes]
    ctx = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, prec)
    idx = sgkiif.IndexSet(ctx, d, n, k)
    op = sgkiif.Operator(ctx, idx, [1.0] * d)
    sol = sgkiif.Solver(ctx, [op], [[]], M, dt)
    U = torch.empty(idx.dof, dtype=torch.float64, device="cuda")
    idx.project_separable(with_amp, WAVES[modes].copy(), KINDS[modes].copy(), 0.0, U.data_ptr())
    sol.set_state(0, dev_ptr=U.data_ptr())
    sol.step(3)
    got = sol.get_state(0)[list(want)]
    assert rel(got, list(want.values())) <= 1e-9
    sol.close()
    op.close()
    idx.close()
    ctx.close()


@pytest.mark.parametrize("d,n,k", [(2, 5, 3), (2, 9, 3), (3, 4, 3), (3, 7, 2), (3, 7, 3), (4, 4, 2), (4, 4, 3), (4, 6, 2)])
def test_matvec_lanes_per_output(ctx, d, n, k):
    # eight, four and two lanes per output in every dimension
    idx = sgkiif.IndexSet(ctx, d, n, k)
    kap = [1.0, 0.5, 0.1, 0.7][:d]
    op = sgkiif.Operator(ctx, idx, kap)
    dtype, tol = ((torch.float64, 1e-12) if ctx.precision == sgkiif.SGK_FP64 else (torch.float32, 1e-5))
    xd = dev(np.random.default_rng(n).standard_normal(idx.dof), dtype)
    yd = torch.empty_like(xd)
    op.matvec(xd.data_ptr(), yd.data_ptr(), ctx.precision)
    torch.cuda.synchronize()
    want = sparse_matvec(OIndex(d, n, k), sipg_1d(n, k), kap, xd.double().cpu().numpy())
    assert rel(yd.double().cpu().numpy(), want) <= tol
    op.close()
    idx.close()


@pytest.mark.parametrize("full", [(True, False), (False, True)], ids=["full_diagonal", "diagonal_full"])
@pytest.mark.parametrize("d,n,k,M", [(2, 4, 2, 20), (3, 3, 1, 12)])
def test_full_and_diagonal_tensor_in_one_system(ctx, d, n, k, M, full, monkeypatch):
    # the species share the slices of the persistent kernel, one with a merged
    # list per output, one with gather entries in shared memory
    kap = np.linspace(1.0, 0.6, d)
    K = np.diag(kap) + 0.1 * (np.eye(d, k=1) + np.eye(d, k=-1))
    idx = sgkiif.IndexSet(ctx, d, n, k)
    ops = [sgkiif.Operator(ctx, idx, K if f else list(kap)) for f in full]
    P, E = cross_blocks_1d(n, k, PERIODIC)
    ref, S = OIndex(d, n, k), sipg_1d(n, k)
    V = np.random.default_rng(d).standard_normal((2, idx.dof))
    dt, launches, states = 1e-5, [], []
    for off in (False, True):
        if off:
            monkeypatch.setenv("SGK_NO_PERSISTENT", "1")
        sol = sgkiif.Solver(ctx, ops, [[(-1.0, (1, 0))], [(0.5, (1, 1))]], M, dt)
        for s, f in enumerate(full):
            vd, wd = dev(V[s]), torch.empty(idx.dof, dtype=torch.float64, device="cuda")
            before = ctx.launches
            sol.krylov_expv(s, vd.data_ptr(), wd.data_ptr())
            launches.append(ctx.launches - before)
            want, _ = krylov_expv(lambda x: sparse_matvec_general(ref, S, P, E, K, x) if f else
                                  sparse_matvec(ref, S, kap, x), V[s], dt, M)
            assert rel(wd.cpu().numpy(), want) <= (1e-10 if f or ctx.precision == sgkiif.SGK_FP64 else 1e-9)
        for s in range(2):
            sol.set_state(s, 0.1 * V[s])
        sol.step(2)
        states.append(np.concatenate([sol.get_state(s) for s in range(2)]))
        sol.close()
    # one launch for the process and a few around it, against several a step
    assert max(launches[:2]) < M < min(launches[2:])
    assert rel(states[0], states[1]) <= 1e-9
    for o in ops:
        o.close()
    idx.close()


@pytest.mark.parametrize("d,n,k", [(2, 4, 1), (2, 5, 2), (3, 4, 2)])
def test_projection_with_the_most_columns(ctx, d, n, k):
    # 128 columns and the norm: two lanes a column instead of four.  Converged
    # for this dt: 1e-10, with the double-float matvec 1e-9
    idx = sgkiif.IndexSet(ctx, d, n, k)
    kap = [1.0, 0.5, 0.1][:d]
    op = sgkiif.Operator(ctx, idx, kap)
    M, dt = 128, 1e-4
    sol = sgkiif.Solver(ctx, [op], [[]], M, dt)
    v = np.random.default_rng(n).standard_normal(idx.dof)
    vd, wd = dev(v), torch.empty(idx.dof, dtype=torch.float64, device="cuda")
    sol.krylov_expv(0, vd.data_ptr(), wd.data_ptr())
    ref, S = OIndex(d, n, k), sipg_1d(n, k)
    want, _ = krylov_expv(lambda x: sparse_matvec(ref, S, kap, x), v, dt, M)
    assert rel(wd.cpu().numpy(), want) <= (1e-10 if ctx.precision == sgkiif.SGK_FP64 else 1e-9)
    sol.close()
    op.close()
    idx.close()
