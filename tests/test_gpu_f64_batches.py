"""The digits of the FP64 slice products live in one buffer of bounded size, in
which long lists go through batch by batch and large products block by block,
and which the context's memory figure counts."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from workloads import slab_problem

torch = pytest.importorskip("torch")
import paper_2208_06191_gb300 as pkg  # noqa: E402

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "dense.cuh"
namespace cbddc {
void count_launch() {}
void timer_begin(int, cudaStream_t) {}
void timer_end(int, cudaStream_t, double, double) {}
bool tensor_cores_for(bool) { return true; }
bool tc_sweep_ks1() { return true; }
bool tc_other_ks1() { return false; }
}
using namespace cbddc;
// problems: np x {M, N, K, lda, ldb, ldc, a, b, c}; C is the whole product list's
// result with digits of at most cap bytes per batch.  info: batches, bytes.
extern "C" int products(int np, const long long* prob, long long na, double* A, long long nb, double* B, long long nc,
                        double* C, int ta, int tb, int order, long long cap, long long* info) {
  try {
    std::vector<GemmProb> v;
    for (int i = 0; i < np; ++i, prob += 9)
      v.push_back(GemmProb{(int)prob[0], (int)prob[1], (int)prob[2], (int)prob[3], (int)prob[4], (int)prob[5],
                           prob[6], prob[7], prob[8]});
    DVec<double> dA, dB, dC;
    DVec<int> status;
    dA.upload(std::vector<double>(A, A + na));
    dB.upload(std::vector<double>(B, B + nb));
    dC.upload(std::vector<double>(C, C + nc));
    status.upload(std::vector<int>(4, 0));
    GemmList g;
    g.set(v, 8, ta != 0, order, tb != 0);
    if (cap > 0) g.plan_oz(cap);
    info[0] = (long long)g.oz_batches.size();
    info[1] = g.oz_bytes();
    DVec<unsigned char> s;
    s.alloc((size_t)g.oz_bytes());
    g.bind_oz(s.p, status.p);
    if (ta && tb) launch_list<double, true, true>(g, dA.p, dB.p, dC.p, -1.0, 1.0, 0);
    else if (ta) launch_list<double, true, false>(g, dA.p, dB.p, dC.p, -1.0, 1.0, 0);
    else launch_list<double, false, false>(g, dA.p, dB.p, dC.p, -1.0, 1.0, 0);
    int st = 0;
    CB_CUDA(cudaMemcpy(C, dC.p, nc * sizeof(double), cudaMemcpyDeviceToHost));
    CB_CUDA(cudaMemcpy(&st, status.p, sizeof st, cudaMemcpyDeviceToHost));
    return st;
  } catch (const Error& e) {
    fprintf(stderr, "%s\n", e.msg.c_str());
    return -2;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    if not os.path.exists(nvcc):
        nvcc = shutil.which("nvcc")
    if nvcc is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("batches")
    src = d / "batches.cu"
    src.write_text(SOURCE)
    so = d / "libbatches.so"
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode=arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2208_06191_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


# (a tile row, a tile column and K = 200 take 690 KB of digits)
SIZES = [(300, 200, 200), (1, 700, 65), (500, 1, 64), (0, 5, 3), (129, 65, 1), (640, 600, 130)]


@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("cap", [1, 1 << 20, 3 << 20])
def test_batches_and_blocks_give_the_same_bits(lib, ta, tb, order, cap):
    rng = np.random.default_rng(1)
    prob, As, Bs, Cs = [], [], [], []
    for M, N, K in SIZES:
        row = [M, N, K]
        offs = []
        for shape, lst in (((K, M) if ta else (M, K), As), ((N, K) if tb else (K, N), Bs), ((M, N), Cs)):
            ld = max(-(-shape[1] // 4) * 4, 4)
            row.append(ld)
            offs.append(sum(x.size for x in lst))
            lst.append(rng.standard_normal(shape[0] * ld))
        prob.append(row + offs)
    prob = np.array(prob, np.int64)
    a, b, c0 = (np.concatenate(x) for x in (As, Bs, Cs))
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    ll = ctypes.c_longlong
    out = []
    for limit in (0, cap):
        c, info = c0.copy(), np.zeros(2, np.int64)
        assert lib.products(len(SIZES), ptr(prob), ll(a.size), ptr(a), ll(b.size), ptr(b), ll(c.size), ptr(c), ta, tb,
                            order, ll(limit), ptr(info)) == 0
        out.append(c)
        assert (info[0] == 1) if limit == 0 else (info[0] > 1)
        # rounding of the parts to 256 bytes, and one tile row and column at least
        assert limit == 0 or info[1] <= max(cap, (128 + 64) * (256 * 14 + 8)) + 1024
    assert np.array_equal(out[0], out[1])
    assert not np.array_equal(out[0], c0)


@pytest.mark.parametrize("kw", [dict(precision=pkg.FP64), dict(precision=pkg.FP32),
                                dict(precision=pkg.FP64, scaling="deluxe", coarse="petrov")])
def test_context_memory_is_counted(kw):
    """What a context reports is what the device loses, but for the allocator's
    rounding (512 bytes for each of a few hundred arrays, 2 MB for what does not
    share a block)."""
    prob = slab_problem(24, 24, 8, order=1, lengths=(3.0, 3.0, 1.0), parts=(2, 2, 2), primal="VE")
    P = pkg.Problem(prob)
    n = P.n_free
    d = torch.zeros(n, dtype=torch.float64, device="cuda")
    b, x = torch.ones_like(d), torch.empty_like(d)
    P.assemble_tangent(d, 0.5)
    warm = pkg.BDDC(P, primal="VE", **kw).setup()     # loads the kernels
    warm.gmres(b, x, restart=20, max_iters=20, rtol=1e-3)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    pc = pkg.BDDC(P, primal="VE", **kw).setup()
    pc.gmres(b, x, restart=20, max_iters=20, rtol=1e-3)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    told = pc.info()["device_bytes"]
    assert told <= held + (1 << 20)
    assert held <= told + (64 << 20)
    del warm
