"""Tables that an operator does without when the device has no memory for them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.index_set import IndexSet as OIndex  # noqa: E402
from oracle.krylov import krylov_expv  # noqa: E402
from oracle.operator import cross_blocks_1d, sipg_1d, sparse_matvec_general  # noqa: E402
from paper_1810_11111_gb300 import sgkiif  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("prec", [sgkiif.SGK_FP64, sgkiif.SGK_MIXED], ids=["fp64", "mixed"])
def test_full_tensor_without_tables(prec, monkeypatch):
    # (failure injected on the host) assembly, matvec and projection go the way
    # of operators whose tables would be too large: 1e-12, FP32 1e-5, 1e-10
    monkeypatch.setenv("SGK_TEST_NO_TABLE_MEMORY", "1")
    d, n, k, M, dt = 3, 3, 2, 15, 1e-5
    K = np.diag([1.0, 0.8, 0.6]) + 0.1 * (np.eye(d, k=1) + np.eye(d, k=-1))
    ctx = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, prec)
    idx = sgkiif.IndexSet(ctx, d, n, k)
    op = sgkiif.Operator(ctx, idx, K)
    P, E = cross_blocks_1d(n, k)
    ref, S = OIndex(d, n, k), sipg_1d(n, k)
    v = np.random.default_rng(1).standard_normal(idx.dof)
    dtype, tol = (torch.float64, 1e-12) if prec == sgkiif.SGK_FP64 else (torch.float32, 1e-5)
    xd = torch.as_tensor(v, dtype=dtype, device="cuda")
    yd = torch.empty_like(xd)
    op.matvec(xd.data_ptr(), yd.data_ptr(), prec)
    torch.cuda.synchronize()
    want = sparse_matvec_general(ref, S, P, E, K, xd.double().cpu().numpy())
    assert rel(yd.double().cpu().numpy(), want) <= tol
    sol = sgkiif.Solver(ctx, [op], [[]], M, dt)
    vd = torch.as_tensor(v, device="cuda")
    wd = torch.empty_like(vd)
    before = ctx.launches
    sol.krylov_expv(0, vd.data_ptr(), wd.data_ptr())
    assert ctx.launches - before > M  # the sequence of launches
    want, _ = krylov_expv(lambda x: sparse_matvec_general(ref, S, P, E, K, x), v, dt, M)
    assert rel(wd.cpu().numpy(), want) <= 1e-10
    sol.close()
    op.close()
    idx.close()
    ctx.close()
