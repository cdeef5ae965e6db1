"""The block product on both sides of the line between its kernels (40 blocks
per row on average), with rows of every remainder modulo three blocks.

Against the same matrix on the host: each entry of the product is a sum of at
most 3 x 125 terms in either order, so the two differ by at most 2 x 375 x 2^-53
times the sum of the terms' magnitudes."""
import numpy as np
import pytest
import scipy.sparse as sp

from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


@pytest.mark.parametrize("n,order,long_rows", [((1, 1, 1), 2, False), ((2, 2, 1), 2, False), ((3, 3, 3), 2, True),
                                               ((5, 4, 2), 2, True), ((6, 5, 4), 2, True), ((6, 5, 4), 1, False)])
def test_block_product(n, order, long_rows):
    prob = slab_problem(*n, order=order, lengths=(0.3 * n[0], 0.25 * n[1], 0.2 * n[2]), parts=(1, 1, 1), jitter=0.1)
    P = pkg.Problem(prob)
    rng = np.random.default_rng(3)
    d = 0.01 * rng.standard_normal(P.n_free)
    P.assemble_tangent(torch.as_tensor(d, device="cuda"), 0.5)
    vals, row_ptr, col = P.tangent_to_host()
    K = sp.bsr_matrix((vals, col, row_ptr), shape=(P.n_free, P.n_free)).tocsr()
    blocks = len(col) / (P.n_free / 3)
    assert (blocks >= 40) == long_rows, blocks
    x = rng.standard_normal(P.n_free)
    y = torch.empty(P.n_free, dtype=torch.float64, device="cuda")
    P.spmv(torch.as_tensor(x, device="cuda"), y)
    bound = 2 * 375 * 2.0**-53 * (abs(K) @ np.abs(x))
    assert np.all(np.abs(y.cpu().numpy() - K @ x) <= bound)
