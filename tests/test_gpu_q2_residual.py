"""The warp-per-element Q2 residual kernel against the oracle, at element
counts around its four elements per CTA, with both fibre fields, and with
inertia and Robin faces.  Both sides integrate with the same rule in FP64, so
they differ by rounding of sums of at most a few hundred terms: 1e-12."""
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


def _dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 1, 1), (2, 2, 1), (5, 1, 1), (3, 2, 2)])
@pytest.mark.parametrize("fibers", ["slab_helix", "nodal"])
@pytest.mark.parametrize("timed", [False, True])
def test_q2_residual(n, fibers, timed):
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
    out = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    P.residual(_dev(d), 0.7, out)
    ref = fe.residual(d, 0.7)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)


def test_q2_inverted_element_is_reported():
    prob = slab_problem(3, 1, 1, order=2, parts=(1, 1, 1))
    P = pkg.Problem(prob)
    X = np.asarray(prob["coords"])
    free = np.setdiff1d(np.arange(len(X)), prob["dirichlet_nodes"])
    d = np.zeros((len(free), 3))
    d[X[free][:, 2] > 0.9, 2] = -2.0  # the top face is pushed through the bottom
    out = torch.empty(3 * len(free), dtype=torch.float64, device="cuda")
    with pytest.raises(pkg.CBDDCError) as ei:
        P.residual(_dev(d.reshape(-1)), 0.5, out)
    assert ei.value.code == pkg.EINVERTED
