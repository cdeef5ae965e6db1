"""The warp-per-element Q2 tangent kernel against the oracle, at element counts
around its five elements per CTA, with both fibre fields, and with inertia and
Robin faces.  Both sides integrate with the same rule in FP64; every entry is a
sum of 27 x 9 products whose largest partial sums stay within a hundred times
the largest entry, so rounding is below 243 x 100 x 2^-53 = 3e-12 of it in the
worst case and far below on average: 1e-12 of the largest entry."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle.assembly import FEProblem
from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [(1, 1, 1), (4, 1, 1), (5, 1, 1), (3, 2, 1), (3, 2, 2)])
@pytest.mark.parametrize("fibers", ["slab_helix", "nodal"])
@pytest.mark.parametrize("timed", [False, True])
def test_q2_tangent(n, fibers, timed):
    prob = slab_problem(*n, order=2, lengths=(0.3 * n[0], 0.25 * n[1], 0.2 * n[2]), parts=(1, 1, 1), jitter=0.1)
    rng = np.random.default_rng(4)
    if fibers == "nodal":
        f = np.array([1.0, 0.2, 0.1]) + 0.1 * rng.standard_normal((len(prob["coords"]), 3))
        s = np.array([0.1, -0.1, 1.0]) + 0.1 * rng.standard_normal((len(prob["coords"]), 3))
        prob["fibers"] = {"kind": "nodal", "f": f, "n": s}
    if timed:
        prob["rho"] = 1000.0
        prob["robin_faces"] = np.array([[0, 0, 0], [0, 2, 1]])
        prob["robin"] = [dict(k_perp=2e5, k_par=2e4, c_perp=1e4, c_par=2e3),
                         dict(k_perp=1e5, k_par=1e4, c_perp=5e3, c_par=1e3)]
    fe = FEProblem(prob)
    X = fe.coords[fe.free_nodes]
    d = (0.05 * X[:, 2:3] * np.sin(3 * X + 1.0)).reshape(-1)
    P = pkg.Problem(prob)
    if timed:
        d1, d2 = 0.9 * d, 0.7 * d
        fe.set_time_state(0.01, d1, d2)
        P.set_time_state(0.01, _dev(d1), _dev(d2))
    r = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    P.assemble_tangent(_dev(d), 0.7, r)
    vals, row_ptr, col = P.tangent_to_host()
    K = sp.bsr_matrix((vals, col, row_ptr), shape=(fe.n_free, fe.n_free)).toarray()
    ref = fe.tangent(d, 0.7)[0].toarray()
    assert np.abs(K - ref).max() <= 1e-12 * np.abs(ref).max()
    rr = fe.residual(d, 0.7)
    assert np.linalg.norm(r.cpu().numpy() - rr) <= 1e-12 * np.linalg.norm(rr)
