"""The apply forks its coarse correction onto a second stream and joins it
again.  On streams other than the default one, with inputs and outputs that are
written and read on that stream alone, without synchronisation between the
calls, on two handles at once and replayed from a captured graph, it gives the
bits of the first call."""
import numpy as np
import pytest

from workloads import slab_problem
from workloads.slab import box_groups

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu

CALLS = 12


@pytest.fixture(scope="module", autouse=True)
def _lib():
    pkg.build()
    pkg.load_library()


def _context(precision, levels):
    prob = slab_problem(12, 8, 4, order=1, parts=(4, 4, 2), jitter=0.1, primal="VE")
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.zeros(P.n_free, dtype=torch.float64, device="cuda"), 0.5)
    kw = {}
    if levels == 3:
        part2, n2 = box_groups((4, 4, 2), (2, 2, 1))
        kw = dict(levels=3, part2=part2, n_parts2=n2)
    return P, pkg.BDDC(P, precision=precision, primal="VE", **kw).setup()


@pytest.mark.parametrize("precision", [pkg.FP64, pkg.FP32])
@pytest.mark.parametrize("levels", [2, 3])
def test_apply_on_other_streams(precision, levels):
    handles = [_context(precision, levels) for _ in range(2)]
    n = handles[0][0].n_free
    rng = np.random.default_rng(4)
    rs = torch.as_tensor(rng.standard_normal((CALLS, n)), device="cuda")
    ref = torch.empty_like(rs)
    for q in range(CALLS):
        handles[0][1].apply(rs[q], ref[q])
    torch.cuda.synchronize()
    outs = []
    for P, pc in handles:     # one stream per handle, their work overlapping
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            r, z, out = torch.empty_like(rs[0]), torch.empty_like(rs[0]), torch.zeros_like(rs)
            for q in range(CALLS):
                r.copy_(rs[q])           # overwrites the last call's input
                pc.apply(r, z)
                out[q].copy_(z)
                z.zero_()
        outs.append((s, r, z, out))
    torch.cuda.synchronize()
    for _, _, _, out in outs:
        assert torch.equal(out, ref)


@pytest.mark.parametrize("precision", [pkg.FP64, pkg.FP32])
def test_captured_apply(precision):
    P, pc = _context(precision, 2)
    r = torch.as_tensor(np.random.default_rng(5).standard_normal(P.n_free), device="cuda")
    ref, z = torch.empty_like(r), torch.zeros_like(r)
    pc.apply(r, ref)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        pc.apply(r, z)
    for _ in range(3):
        z.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(z, ref)
