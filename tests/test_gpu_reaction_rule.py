"""Which reaction passes a solver takes: sizes and coefficients at which a pass
does not serve, against the general passes and closed values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1810_11111_gb300 import sgkiif  # noqa: E402

pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

CUBIC = [[(-2.0, (3,)), (0.7, (2,)), (-0.3, (0,))]]
PAIR = [[(0.1, (0, 0)), (-1.0, (1, 0)), (1.0, (2, 1))], [(0.9, (0, 0)), (-1.0, (2, 1))]]


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-300))


def passes(ctx, d, n, k, rx, U, W):
    """F(U) and J_F(U) W of a fresh solver."""
    idx = sgkiif.IndexSet(ctx, d, n, k)
    ops = [sgkiif.Operator(ctx, idx, [1.0] * d) for _ in rx]
    sol = sgkiif.Solver(ctx, ops, rx, 2, 0.01)
    Ud, Wd = (torch.from_numpy(x).cuda() for x in (U, W))
    Fd, Jd = torch.empty_like(Ud), torch.empty_like(Ud)
    sol.reaction_eval(Ud.data_ptr(), Fd.data_ptr())
    sol.jacobian_apply(Ud.data_ptr(), Wd.data_ptr(), Jd.data_ptr())
    torch.cuda.synchronize()
    out = Fd.cpu().numpy(), Jd.cpu().numpy()
    sol.close()
    for o in ops:
        o.close()
    idx.close()
    return out


@pytest.fixture(scope="module", params=[sgkiif.SGK_FP64, sgkiif.SGK_MIXED], ids=["fp64", "mixed"])
def ctx(request):
    c = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, request.param)
    yield c
    c.close()


@pytest.mark.parametrize("n,k,rx", [(10, 2, PAIR), (11, 1, CUBIC), (11, 2, CUBIC)])
def test_lines_beyond_shared_memory(ctx, n, k, rx, monkeypatch):
    # 2D lines of which not every pass fits a CTA's shared memory: the general
    # passes serve them.  Sums of at most some thousand terms in another
    # order: 1e-12, FP32 Jacobian 1e-5
    S, dof = len(rx), sgkiif.dof_of(2, n, k)
    rng = np.random.default_rng(n)
    U = 0.3 * rng.standard_normal(S * dof) / np.sqrt(dof)
    U[::dof] += 0.5
    W = rng.standard_normal(S * dof)
    F, J = passes(ctx, 2, n, k, rx, U, W)
    monkeypatch.setenv("SGK_NO_FUSED", "1")
    F1, J1 = passes(ctx, 2, n, k, rx, U, W)
    assert rel(F, F1) <= 1e-12
    assert rel(J, J1) <= (1e-12 if ctx.precision == sgkiif.SGK_FP64 else 1e-5)


@pytest.mark.parametrize("c,u", [(1e-300, 1e110), (-1e-220, 1e105), (1e200, 1e-110)])
@pytest.mark.parametrize("low", [0.0, 0.5])
def test_coefficients_near_the_ends_of_the_range(c, u, low):
    # FP64, f(u) = c u^3 + low c u^2 u_0 with u_0 the state's size: c u^3 is
    # finite where u^3 is not.  F scales like c u^3, J like c u^2
    fp64 = sgkiif.Context(0, torch.cuda.current_stream().cuda_stream, sgkiif.SGK_FP64)
    d, n, k = 3, 3, 2
    rng = np.random.default_rng(3)
    U = 0.1 * rng.standard_normal(sgkiif.dof_of(d, n, k))
    U[0] = 1.0
    W = rng.standard_normal(U.size)

    def terms(c, u0):
        return [[(c, (3,))] + ([(low * c * u0, (2,))] if low else [])]

    # the oracle scales by powers of two, which are exact
    su = 2.0 ** round(np.log2(u))
    F1, J1 = passes(fp64, d, n, k, terms(1.0, 1.0), U, W)
    F, J = passes(fp64, d, n, k, terms(c, su), su * U, W)
    assert rel(F / (c * su) / su / su, F1) <= 1e-12
    assert rel(J / (c * su) / su, J1) <= 1e-12
    fp64.close()


@pytest.mark.parametrize("d,n,k", [(2, 6, 2), (3, 5, 2), (4, 3, 1)])
def test_large_coefficients_of_a_small_state(ctx, d, n, k):
    # 1e32 u^3 at u = 1e-11: within FP32's range in the orthonormal basis, not
    # in the pass's scaled one.  F to 1e-12 in both modes, an FP32 J to 1e-5
    c, u = 2.0 ** 106, 2.0 ** -36
    rng = np.random.default_rng(n)
    U = 0.1 * rng.standard_normal(sgkiif.dof_of(d, n, k)) / (1 + np.arange(sgkiif.dof_of(d, n, k)))
    U[0] = 1.0
    W = rng.standard_normal(U.size)
    F1, J1 = passes(ctx, d, n, k, [[(1.0, (3,))]], U, W)
    F, J = passes(ctx, d, n, k, [[(c, (3,))]], u * U, W)
    assert rel(F / c / u ** 3, F1) <= 1e-12
    assert rel(J / c / u ** 2, J1) <= (1e-12 if ctx.precision == sgkiif.SGK_FP64 else 1e-5)
