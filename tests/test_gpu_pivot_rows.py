"""The sweeps of FP64 operators around 4096 columns, from where the pivot rows
are multiplied by the pivot block's inverse as products of their own: a single
matrix below and above the line (with a partial last pivot block), where the
apply is the inverse, and subdomains of several sizes in one list.

Single matrices: condition numbers up to 1e5 times 2^-53 make 1e-11; 1e-9
leaves a factor of 100.  Against the oracle's BDDC both sides carry that error:
the same bound."""
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


# unknowns: 3 (nx + 1)(ny + 1) nz = 4095 and 4200
@pytest.mark.parametrize("n", [(20, 12, 5), (24, 13, 4)])
def test_single_matrix(n):
    prob = slab_problem(*n, order=1, lengths=(0.25 * n[0], 0.25 * n[1], 0.25 * n[2]), parts=(1, 1, 1), jitter=0.1,
                        primal="V")
    fe, d, P = _state(prob)
    K = fe.tangent(d, 0.6)[0].toarray()
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="V").setup()
    r = np.random.default_rng(5).standard_normal(fe.n_free)
    z = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    pc.apply(torch.as_tensor(r, device="cuda"), z)
    ref = np.linalg.solve(K, r)
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 1e-9 * np.linalg.norm(ref)


@pytest.mark.parametrize("kw", [dict(), dict(scaling="deluxe"), dict(coarse="petrov")])
def test_ragged_list(kw):
    prob = slab_problem(22, 19, 5, order=1, lengths=(2.2, 1.9, 0.5), parts=(4, 4, 1), jitter=0.15, primal="VEF")
    fe, d, P = _state(prob)
    _, (Ke, Kf) = fe.tangent(d, 0.6)
    ref = OracleBDDC(fe, Ke, Kf, "VEF", **kw)
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="VEF", **kw).setup()
    r = np.random.default_rng(6).standard_normal(fe.n_free)
    z = torch.empty(fe.n_free, dtype=torch.float64, device="cuda")
    pc.apply(torch.as_tensor(r, device="cuda"), z)
    zr = ref.apply(r)
    assert np.linalg.norm(z.cpu().numpy() - zr) <= 1e-9 * np.linalg.norm(zr)
