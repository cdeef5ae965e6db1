"""The one-launch Gram-Schmidt step with chunks of more than 512 rows per CTA,
where its update works in three and in two parts of the columns, and with two
CTAs per SM.

GMRES against one written here on the same preconditioner and product, with
modified Gram-Schmidt applied twice: the residual estimates of both are exact to
rounding, so the iteration counts to 1e-9 are the same (a residual within 1e-6
relative of the tolerance aside, which is checked), and the solutions agree to
the tolerance times the condition number of the preconditioned operator (below
100 here): 1e-7."""
import numpy as np
import pytest

from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu

RTOL = 1e-9


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


def _gmres(P, pc, b, steps):
    """Solution and relative residuals after each step (right preconditioned)."""
    n = b.numel()
    V = torch.zeros((steps + 1, n), dtype=torch.float64, device="cuda")
    Z = torch.zeros((steps, n), dtype=torch.float64, device="cuda")
    H = np.zeros((steps + 1, steps))
    beta = float(b.norm())
    V[0] = b / beta
    w = torch.empty_like(b)
    res, y = [], None
    for j in range(steps):
        pc.apply(V[j], Z[j])
        P.spmv(Z[j], w)
        for _ in range(2):
            for i in range(j + 1):
                h = float(V[i] @ w)
                H[i, j] += h
                w -= h * V[i]
        H[j + 1, j] = float(w.norm())
        V[j + 1] = w / H[j + 1, j]
        e = np.zeros(j + 2)
        e[0] = beta
        y, *_ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
        res.append(float(np.linalg.norm(H[:j + 2, :j + 1] @ y - e)) / beta)
        if res[-1] <= RTOL:
            break
    k = len(res)
    return torch.as_tensor(y, device="cuda") @ Z[:k], res


# unknowns 3 (nx + 1)(ny + 1) nz and rows per CTA: 101k, 672 (three parts);
# 139k, 928 (two); 158k in two CTAs per SM, 544 (three); 286k, 960 (two)
@pytest.mark.parametrize("n,parts", [((40, 40, 20), (4, 4, 2)), ((46, 46, 21), (4, 4, 2)), ((48, 48, 22), (4, 4, 4)),
                                     ((62, 62, 24), (8, 8, 2))])
def test_gmres_with_long_chunks(n, parts):
    prob = slab_problem(*n, order=1, lengths=tuple(0.1 * k for k in n), parts=parts, primal="VE")
    P = pkg.Problem(prob)
    assert P.n_free == 3 * (n[0] + 1) * (n[1] + 1) * n[2]
    P.assemble_tangent(torch.zeros(P.n_free, dtype=torch.float64, device="cuda"), 0.5)
    pc = pkg.BDDC(P, precision=pkg.FP32, primal="VE").setup()
    b = torch.as_tensor(np.random.default_rng(9).standard_normal(P.n_free), device="cuda")
    x = torch.empty_like(b)
    rep = pc.gmres(b, x, restart=120, max_iters=120, rtol=RTOL)
    assert rep["converged"]
    ref, res = _gmres(P, pc, b, 120)
    assert all(abs(r / RTOL - 1.0) > 1e-6 for r in res)
    assert rep["iterations"] == len(res)
    assert float((x - ref).norm()) <= 1e-7 * float(ref.norm())
