"""FP64 dense products whose operands are scaled against each other along K.

FMAs do not see a diagonal scaling between the operands, and the setup of a
graded problem has it in every product: a Gauss-Jordan sweep multiplies columns
of size d_i d_k by rows of size d_j / d_k, with d the square roots of the diagonal.
Two kinds of test:

* single products of csrc/dense.cuh against extended precision, with the
  exponents of the scaling given.  Bound of entry (i, j): the final rounding and
  addition, 2^-52 (|C| + |A B|), and for K terms held as seven digits of nine
  bits relative to the largest of the scaled row and column, 2^-57 K max_k |a_ik|
  2^s_k max_k |b_kj| 2^-s_k (the operands' quantisation is 2^-62 of it per term, the
  dropped digit products 2^-60.4, the truncated order sums 2^-60, and a power of
  two above the largest entry is up to twice it, in both operands);
* the whole setup on meshes that are graded by layers: with one subdomain the
  apply is the inverse of the tangent, and in the norm of the Jacobi-scaled
  unknowns an FP64 sweep is off by a small multiple of the scaled matrix's
  condition number (below 1e4, asserted) times 2^-53: 1e-12 leaves a factor of
  ten to 100.  With more subdomains the oracle is the reference."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle.assembly import FEProblem
from oracle.bddc import BDDC as OracleBDDC
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
template <bool TA, bool TB>
static void go(const GemmList& g, const double* A, const double* B, double* C, int add) {
  launch_list<double, TA, TB>(g, A, B, C, add ? -1.0 : 1.0, add ? 1.0 : 0.0, 0);
}
// problems: np x {M, N, K, lda, ldb, ldc, a, b, c, ks, ke}; A, B, C, kexp: host arrays
extern "C" int products(int np, const long long* prob, long long na, double* A, long long nb, double* B, long long nc,
                        double* C, long long nk, int* kexp, int ta, int tb, int add, long long* scratch) {
  try {
    std::vector<GemmProb> v;
    for (int i = 0; i < np; ++i, prob += 11)
      v.push_back(GemmProb{(int)prob[0], (int)prob[1], (int)prob[2], (int)prob[3], (int)prob[4], (int)prob[5],
                           prob[6], prob[7], prob[8], (int)prob[9], prob[10]});
    DVec<double> dA, dB, dC;
    DVec<int> dk, status;
    dA.upload(std::vector<double>(A, A + na));
    dB.upload(std::vector<double>(B, B + nb));
    dC.upload(std::vector<double>(C, C + nc));
    dk.upload(std::vector<int>(kexp, kexp + nk));
    status.upload(std::vector<int>(4, 0));
    GemmList g;
    g.set(v, 8, ta != 0, 0);
    DVec<unsigned char> s;
    s.alloc((size_t)g.oz_bytes());
    *scratch = g.oz_bytes();
    g.bind_oz(s.p, status.p, dk.p);
    if (ta && tb) go<true, true>(g, dA.p, dB.p, dC.p, add);
    else if (ta) go<true, false>(g, dA.p, dB.p, dC.p, add);
    else if (tb) go<false, true>(g, dA.p, dB.p, dC.p, add);
    else go<false, false>(g, dA.p, dB.p, dC.p, add);
    int st = 0;
    CB_CUDA(cudaMemcpy(C, dC.p, nc * sizeof(double), cudaMemcpyDeviceToHost));
    CB_CUDA(cudaMemcpy(&st, status.p, sizeof st, cudaMemcpyDeviceToHost));
    return st == 0 ? (int)g.oz_batches.size() : -1;
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
    d = tmp_path_factory.mktemp("products")
    src = d / "products.cu"
    src.write_text(SOURCE)
    so = d / "libproducts.so"
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode=arch=compute_103a,code=sm_103a", "--expt-relaxed-constexpr",
                    "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2208_06191_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so))


def _run(lib, sizes, ta=0, tb=0, add=0, grade=0, fill=None, pad=0, seed=0):
    """The products of random operands with the given sizes (M, N, K), entries of
    op(A)(:, k) of size 2^g_k and of op(B)(k, :) of size 2^-g_k with |g_k| <= grade,
    rows and columns of sizes 2^-20 to 2^20; returns per product C, its exact
    value and the bound."""
    rng = np.random.default_rng(seed)
    prob, As, Bs, Cs, ks, ops = [], [], [], [], [], []
    for M, N, K in sizes:
        g = rng.integers(-grade, grade + 1, K)
        A = rng.standard_normal((M, K)) * 2.0 ** (g + rng.integers(-20, 21, (M, 1)))
        B = rng.standard_normal((K, N)) * 2.0 ** (rng.integers(-20, 21, (1, N)) - g[:, None])
        if fill:
            fill(A, B)
        C = rng.standard_normal((M, N))
        sa, sb = (A.T if ta else A), (B.T if tb else B)
        lay = []
        for X, lst in ((sa, As), (sb, Bs), (C, Cs)):
            ld = -(-X.shape[1] // 4) * 4 + pad
            buf = np.zeros((X.shape[0], ld))
            buf[:, :X.shape[1]] = X
            off = sum(x.size for x in lst)
            lst.append(np.concatenate([buf.ravel(), np.zeros(-buf.size % 4)]))
            lay.append((ld, off))
        prob.append([M, N, K, lay[0][0], lay[1][0], lay[2][0], lay[0][1], lay[1][1], lay[2][1], -1 if grade else 0,
                     sum(x.size for x in ks)])
        ks.append(g)
        ops.append((A, B, C, -g if grade else 0 * g, lay[2]))
    prob = np.array(prob, np.int64)
    a, b, c = (np.concatenate(x) for x in (As, Bs, Cs))
    k = np.concatenate(ks).astype(np.int32)
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    ll = ctypes.c_longlong
    scratch = ll(0)
    nb = lib.products(len(sizes), ptr(prob), ll(a.size), ptr(a), ll(b.size), ptr(b), ll(c.size), ptr(c), ll(k.size),
                      ptr(k), ta, tb, add, ctypes.byref(scratch))
    assert nb >= 1
    out = []
    for (M, N, K), (A, B, C, s, (ld, off)) in zip(sizes, ops):
        got = c[off:off + M * ld].reshape(M, ld)[:, :N]
        with np.errstate(all="ignore"):
            AB = A.astype(np.longdouble) @ B.astype(np.longdouble)
            ref = C - AB if add else AB
            big = np.abs(A) * 2.0 ** s
            bound = 2.0 ** -52 * (np.abs(ref) + np.abs(AB)) + K * 2.0 ** -57 * np.outer(
                big.max(1), (np.abs(B) * 2.0 ** -s[:, None]).max(0))
        out.append((got, ref, bound))
    return out, scratch.value, nb


# one row and one column past the tiles of 128 x 64 and the K blocks of 64, and
# one before them
SIZES = [(1, 1, 1), (128, 64, 64), (129, 65, 65), (127, 63, 63), (257, 130, 200), (64, 600, 64), (33, 31, 7)]


@pytest.mark.parametrize("grade", [0, 20, 40])
@pytest.mark.parametrize("ta,tb,add", [(0, 0, 0), (0, 0, 1), (1, 0, 0), (1, 1, 0), (1, 1, 1)])
def test_products_of_graded_operands(lib, ta, tb, add, grade):
    for pad in (0, 1):
        res, _, _ = _run(lib, SIZES, ta, tb, add, grade, pad=pad, seed=grade)
        for size, (got, ref, bound) in zip(SIZES, res):
            assert (np.abs(got - ref) <= bound).all(), (size, float((np.abs(got - ref) / bound).max()))


def test_rows_of_zeros(lib):
    """Zero rows and columns give zeros, and do not touch their neighbours."""
    def fill(A, B):
        A[::3] = 0.0
        B[:, 1::4] = 0.0
        A[:, 5:9] = 0.0
        B[2:4] = 0.0
    for got, ref, bound in _run(lib, [(129, 65, 65), (40, 70, 20)], fill=fill, grade=20)[0]:
        assert (np.abs(got - ref) <= bound).all()
        assert (got[::3] == 0.0).all() and (got[:, 1::4] == 0.0).all()


def test_values_that_are_not_finite(lib):
    """An infinity or a NaN makes its row (or column) of the product NaN, and
    the other entries stay what they are."""
    def fill(A, B):
        A[3, 5], A[4, 0], B[2, 4] = np.inf, np.nan, -np.inf
    got, ref, bound = _run(lib, [(70, 66, 65)], fill=fill)[0][0]
    bad = np.zeros(got.shape, bool)
    bad[3:5] = True
    bad[:, 4] = True
    assert np.isnan(got[bad]).all()
    assert (np.abs(got - ref)[~bad] <= bound[~bad]).all()


def _graded_slab(q, n, nz, parts, primal):
    """A frustum of nz layers, each 1/q of the size of the last: the tangent's
    entries shrink by q per layer."""
    prob = slab_problem(n, n, nz, order=1, lengths=(1.0, 1.0, float(nz)), parts=parts, primal=primal)
    c = prob["coords"]
    s = float(q) ** -c[:, 2]
    prob["coords"] = np.stack([(c[:, 0] - 0.5) * s, (c[:, 1] - 0.5) * s, -s], axis=1)
    prob["fibers"] = dict(prob["fibers"], z0=-1.0, z1=0.0)
    fe = FEProblem(prob)
    sf = s[fe.free_nodes]
    X = fe.coords[fe.free_nodes]
    d = (0.02 * X[:, 2:3] * np.sin(X / sf[:, None] + 1.0)).reshape(-1)
    return prob, fe, d


def _apply(prob, d, r, **kw):
    P = pkg.Problem(prob)
    P.assemble_tangent(torch.as_tensor(d, device="cuda"), 0.0)
    pc = pkg.BDDC(P, precision=pkg.FP64, **kw).setup()
    z = torch.empty(len(r), dtype=torch.float64, device="cuda")
    pc.apply(torch.as_tensor(r, device="cuda"), z)
    return z.cpu().numpy()


# layers from 1 to 8^-13 and 2^-20 of the first one's size
@pytest.mark.parametrize("q,n,nz", [(8, 1, 14), (2, 2, 21)])
def test_inverse_of_a_graded_tangent(q, n, nz):
    prob, fe, d = _graded_slab(q, n, nz, (1, 1, 1), "V")
    K = fe.tangent(d, 0.0)[0].toarray()
    w = np.sqrt(np.diag(K))
    Ks = K / w[:, None] / w[None, :]
    assert np.linalg.cond(Ks) < 1e4
    r = np.random.default_rng(5).standard_normal(fe.n_free)
    z = _apply(prob, d, w * r, primal="V")
    ref = np.linalg.solve(Ks, r)
    assert np.linalg.norm(w * z - ref) <= 1e-12 * np.linalg.norm(ref)


@pytest.mark.parametrize("kw", [dict(), dict(scaling="deluxe"), dict(coarse="petrov")])
@pytest.mark.parametrize("parts", [(2, 2, 1), (2, 2, 2)])
def test_graded_subdomains_against_the_oracle(parts, kw):
    prob, fe, d = _graded_slab(3, 4, 12, parts, "VE")
    K, (Ke, Kf) = fe.tangent(d, 0.0)
    w = np.sqrt(K.diagonal())
    r = w * np.random.default_rng(6).standard_normal(fe.n_free)
    z = _apply(prob, d, r, primal="VE", **kw)
    ref = OracleBDDC(fe, Ke, Kf, "VE", **kw).apply(r)
    assert np.linalg.norm(w * (z - ref)) <= 1e-9 * np.linalg.norm(w * ref)
