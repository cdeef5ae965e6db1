"""The FP64 dense products of the BDDC setup (integer slices on the tensor
cores) at the sizes where their tiles end: output tiles of 128 x 64, K blocks
of 64, pivot blocks of 64.

With one subdomain and no interface the BDDC apply is the inverse of the
tangent, formed by the sweep alone, so a dense solve is the reference.
Tolerance: a backward-stable inverse of these matrices (condition numbers up
to 2e4 on these slabs) is off by at most a small multiple of cond x 2^-53 =
2e-12; 1e-10 leaves a factor of 50."""
import numpy as np
import pytest

from oracle.assembly import FEProblem
from oracle.bddc import BDDC as OracleBDDC
from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


def _state(prob, seed=3):
    fe = FEProblem(prob)
    X = fe.coords[fe.free_nodes]
    rng = np.random.default_rng(seed)
    d = (0.02 * X[:, 2:3] * np.sin(X + rng.uniform(0, 3, 3))).reshape(-1)
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.as_tensor(d, device="cuda"), 0.6)
    return fe, d, P


# unknowns: 3 (nx + 1)(ny + 1) nz = 12, 54, 63, 66, 126, 129, 192, 195, 375, 600
@pytest.mark.parametrize("n", [(1, 1, 1), (2, 2, 2), (2, 6, 1), (1, 10, 1), (6, 2, 2), (42, 0, 1), (3, 3, 4),
                               (4, 12, 1), (4, 4, 5), (4, 4, 8)])
def test_single_subdomain_is_the_inverse(n):
    nx, ny, nz = n[0], max(n[1], 1), n[2]
    prob = slab_problem(nx, ny, nz, order=1, lengths=(0.25 * nx, 0.25 * ny, 0.25 * nz), parts=(1, 1, 1),
                        jitter=0.1, primal="V")
    fe, d, P = _state(prob)
    K = fe.tangent(d, 0.6)[0].toarray()
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="V").setup()
    r = np.random.default_rng(5).standard_normal(fe.n_free)
    z = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    pc.apply(torch.as_tensor(r, device="cuda"), z)
    ref = np.linalg.solve(K, r)
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("kw", [dict(), dict(scaling="deluxe"), dict(coarse="petrov")])
def test_ragged_subdomains_against_the_oracle(kw):
    """Every kind of product (E, S, constraint, coarse-basis, deluxe, left
    basis) on subdomains of 12 to 300 unknowns."""
    prob = slab_problem(9, 5, 4, order=1, lengths=(0.9, 0.5, 0.4), parts=(3, 2, 2), jitter=0.15, primal="VEF")
    fe, d, P = _state(prob)
    _, (Ke, Kf) = fe.tangent(d, 0.6)
    ref = OracleBDDC(fe, Ke, Kf, "VEF", **kw)
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="VEF", **kw).setup()
    r = np.random.default_rng(6).standard_normal(fe.n_free)
    z = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    pc.apply(torch.as_tensor(r, device="cuda"), z)
    zr = ref.apply(r)
    assert np.linalg.norm(z.cpu().numpy() - zr) <= 1e-9 * np.linalg.norm(zr)


def test_overflowed_tangent_is_refused():
    """An infinite entry anywhere in a local matrix (the exponential energy
    overflows in the top element layer) reaches a pivot through the products
    and is reported, in a subdomain whose interior pivots are finite too."""
    prob = slab_problem(4, 4, 4, order=1, parts=(2, 2, 1), primal="VE")
    P = pkg.Problem(prob)
    X = np.asarray(prob["coords"])
    free = np.setdiff1d(np.arange(len(X)), prob["dirichlet_nodes"])
    d = np.where(X[free][:, 2:3] > 0.99, np.array([[0.0, 0.0, 10.0]]), 0.0).reshape(-1)
    P.assemble_tangent(torch.as_tensor(np.ascontiguousarray(d), device="cuda"), 0.5)
    with pytest.raises(pkg.CBDDCError) as ei:
        pkg.BDDC(P, precision=pkg.FP64, primal="VE").setup()
    assert ei.value.code == pkg.EPIVOT
