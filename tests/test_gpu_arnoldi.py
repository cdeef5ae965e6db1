"""The one-launch Gram-Schmidt step where its work division changes: vectors
shorter than a warp, than a CTA's chunk, chunks with one to four column parts
of the update, and bases that end inside a group of eight columns.

GMRES to 1e-12 in FP64 (two subdomains, so that it takes more than one
iteration) against a dense solve: the solution is off by at most the condition
number (below 5e3 on these slabs) times the residual tolerance, 5e-9; the
bound is 1e-8."""
import numpy as np
import pytest

from oracle.assembly import FEProblem
from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


# unknowns: 3 (nx + 1)(ny + 1) nz = 18, 36, 216, 1344, 2592
@pytest.mark.parametrize("n", [(2, 1, 1), (2, 1, 2), (5, 3, 3), (7, 7, 7), (11, 8, 8)])
@pytest.mark.parametrize("restart", [100, 7])
def test_gmres_against_dense_solve(n, restart):
    prob = slab_problem(*n, order=1, lengths=tuple(0.2 * k for k in n), parts=(2, 1, 1), jitter=0.1, primal="VEF")
    fe = FEProblem(prob)
    X = fe.coords[fe.free_nodes]
    d = (0.02 * X[:, 2:3] * np.sin(X + 1.0)).reshape(-1)
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.as_tensor(d, device="cuda"), 0.6)
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="VEF").setup()
    b = np.random.default_rng(7).standard_normal(fe.n_free)
    x = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    rep = pc.gmres(torch.as_tensor(b, device="cuda"), x, restart=restart, max_iters=2000, rtol=1e-12)
    assert rep["converged"] and rep["iterations"] >= 2
    ref = np.linalg.solve(fe.tangent(d, 0.6)[0].toarray(), b)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-8 * np.linalg.norm(ref)
    # the same call again gives the same bits
    y = torch.empty_like(x)
    pc.gmres(torch.as_tensor(b, device="cuda"), y, restart=restart, max_iters=2000, rtol=1e-12)
    assert torch.equal(x, y)


@pytest.mark.parametrize("n,m", [((5, 3, 3), 200), ((11, 8, 8), 200), ((7, 7, 7), 257), ((11, 8, 8), 300)])
def test_basis_past_the_chunked_step(n, m):
    # m vectors whatever the residual: the steps past 128 take the tiled
    # kernel, those past 256 modified Gram-Schmidt (here most of its CTAs own no
    # row), and the least squares solution must stay the converged one
    prob = slab_problem(*n, order=1, lengths=tuple(0.2 * k for k in n), parts=(2, 1, 1), jitter=0.1, primal="VEF")
    fe = FEProblem(prob)
    d = np.zeros(fe.n_free)
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.as_tensor(d, device="cuda"), 0.6)
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="VEF").setup()
    b = np.random.default_rng(11).standard_normal(fe.n_free)
    x = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    rep = pc.gmres(torch.as_tensor(b, device="cuda"), x, restart=m, max_iters=m, rtol=1e-300)
    assert rep["iterations"] == m and not rep["converged"]
    ref = np.linalg.solve(fe.tangent(d, 0.6)[0].toarray(), b)
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 1e-8 * np.linalg.norm(ref)
