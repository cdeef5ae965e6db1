"""What the launch timer says of GMRES and of the parts of an apply.

GMRES launches one step before the last residual is known; the Gram-Schmidt
kernels skip the step that was not needed, and the timer does not count it.
The coarse correction runs beside the local solves, but while its own time is
recorded it is a part of the apply's, with the same result."""
import numpy as np
import pytest

from workloads import slab_problem
from workloads.slab import box_groups

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


def _setup(parts, **kw):
    prob = slab_problem(8, 8, 4, order=1, parts=parts, jitter=0.1, primal="VEF")
    P = pkg.Problem(prob)
    d = torch.zeros(P.n_free, dtype=torch.float64, device="cuda")
    P.assemble_tangent(d, 0.5)
    b = torch.as_tensor(np.random.default_rng(3).standard_normal(P.n_free), device="cuda")
    return P, pkg.BDDC(P, primal="VEF", **kw).setup(), b


# one subdomain: the preconditioner is the inverse, the first step reduces the
# residual by far more than the factor that a step is launched ahead on
@pytest.mark.parametrize("parts,rtol,max_iters", [((1, 1, 1), 1e-8, 100), ((2, 2, 1), 1e-8, 100),
                                                  ((2, 2, 1), 1e-1, 100), ((2, 2, 1), 1e-12, 3)])
def test_one_orthogonalisation_per_iteration(parts, rtol, max_iters):
    P, pc, b = _setup(parts, precision=pkg.FP64)
    x, y = torch.empty_like(b), torch.empty_like(b)
    plain = pc.gmres(b, x, restart=50, max_iters=max_iters, rtol=rtol)
    pkg.timer_start(pkg.TIMER_ORTH)
    rep = pc.gmres(b, y, restart=50, max_iters=max_iters, rtol=rtol)
    t = pkg.timer_stop()
    assert rep["iterations"] == plain["iterations"] and torch.equal(x, y)
    assert t["launches"] == rep["iterations"]
    # flops of steps 0 .. its - 1: 4 (j + 1) n each
    its = rep["iterations"]
    assert t["flops"] == pytest.approx(2.0 * its * (its + 1) * P.n_free, rel=1e-12)


@pytest.mark.parametrize("precision", [pkg.FP64, pkg.FP32])
@pytest.mark.parametrize("levels", [2, 3])
def test_coarse_correction_is_a_part_of_the_apply(precision, levels):
    kw = {}
    if levels == 3:
        part2, n2 = box_groups((4, 4, 2), (2, 2, 1))
        kw = dict(levels=3, part2=part2, n_parts2=n2)
    P, pc, r = _setup((4, 4, 2), precision=precision, **kw)
    z, t0 = torch.empty_like(r), torch.empty_like(r)
    pc.apply(r, z)
    pkg.timer_start(pkg.TIMER_APPLY)
    pkg.timer_enable(pkg.TIMER_LEVEL2_APPLY)
    pkg.timer_enable(pkg.TIMER_COARSE_APPLY)
    for _ in range(5):
        pc.apply(r, t0)
    level2, coarse = pkg.timer_result(pkg.TIMER_LEVEL2_APPLY), pkg.timer_result(pkg.TIMER_COARSE_APPLY)
    apply = pkg.timer_stop()
    assert torch.equal(z, t0)
    assert apply["launches"] == coarse["launches"] == 5
    assert level2["launches"] == (5 if levels == 3 else 0)
    assert 0.0 < coarse["ms"] < apply["ms"]
    assert levels == 2 or coarse["ms"] < level2["ms"] < apply["ms"]
