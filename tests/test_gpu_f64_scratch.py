"""With little device memory free, an FP64 context takes a smaller buffer for
the digits of its products, and gives the same bits."""
import numpy as np
import pytest

from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu


def test_smaller_buffer_when_memory_is_short():
    # 8 subdomains of up to 2.5k unknowns: the products E take 440 MB of digits,
    # a sixteenth of 3 GB is less than half of that
    prob = slab_problem(24, 24, 8, order=1, lengths=(3.0, 3.0, 1.0), parts=(2, 2, 2), primal="VE")
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.zeros(P.n_free, dtype=torch.float64, device="cuda"), 0.5)
    r = torch.as_tensor(np.random.default_rng(2).standard_normal(P.n_free), device="cuda")
    z = [torch.empty_like(r) for _ in range(2)]
    pc = pkg.BDDC(P, precision=pkg.FP64, primal="VE").setup()
    pc.apply(r, z[0])
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(max(torch.cuda.mem_get_info()[0] - (3 << 30), 1), dtype=torch.uint8, device="cuda")
    try:
        short = pkg.BDDC(P, precision=pkg.FP64, primal="VE").setup()
        short.apply(r, z[1])
        torch.cuda.synchronize()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert torch.equal(z[0], z[1])
    assert short.info()["device_bytes"] < pc.info()["device_bytes"] - (20 << 20)
