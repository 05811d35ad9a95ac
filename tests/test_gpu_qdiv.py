"""Division by a rounded reciprocal and one correction (csrc/opf_tri.h) against
the division, and what it decides in the gradient's line prox."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gridgen import make_case, scale_case

pytestmark = pytest.mark.gpu

SRC = r"""
#include "opf_tri.h"
__global__ void k(const float *x, const float *q, float *a, float *d, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float rq = __frcp_rn(q[i]);
  a[i] = opfk::qdiv(x[i], q[i], rq);
  d[i] = __fdiv_rn(x[i], q[i]);
}
extern "C" int run(const float *x, const float *q, float *a, float *d, int n) {
  k<<<(n + 255) / 256, 256>>>(x, q, a, d, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def divide(tmp_path_factory):
    import torch
    from paper_2410_17203_gb300.build import ARCH, CSRC, INCLUDE, cuda_lib_dir, nvcc
    d = tmp_path_factory.mktemp("qdiv")
    src, lib = os.path.join(d, "q.cu"), os.path.join(d, "libq.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run([nvcc(), "-std=c++17", "-O3", ARCH, "-shared", "-cudart", "shared", "-Xcompiler", "-fPIC",
                    "-I", CSRC, "-I", INCLUDE, "-o", lib, src, "-Xlinker", "-rpath," + cuda_lib_dir()], check=True)
    fn = ctypes.CDLL(lib).run
    fn.argtypes = [ctypes.c_void_p] * 4 + [ctypes.c_int]

    def run(x, q):
        t = [torch.from_numpy(np.ascontiguousarray(v, np.float32)).cuda() for v in (x, q)]
        out = [torch.empty_like(t[0]) for _ in range(2)]
        torch.cuda.synchronize()
        assert fn(*[v.data_ptr() for v in t + out], t[0].numel()) == 0
        return [v.cpu().numpy() for v in out]
    return run


def _near_boundaries(rng, n):
    """Significands X, Q in [2^23, 2^24), Q odd, whose quotient lies within a
    few 1 / (Q 2^24) of a rounding boundary or a float: X 2^k = M Q + d, |d| <= 4."""
    X, Q = [], []
    while len(X) < n:
        q = int(rng.integers(1 << 22, 1 << 23)) * 2 + 1
        for k in (24, 25):
            x = int(rng.integers(-4, 5)) * pow(1 << k, -1, q) % q
            x += 0 if x >= 1 << 23 else q
            if 1 << 23 <= x < 1 << 24:
                X.append(x)
                Q.append(q)
    return np.array(X[:n], np.float64), np.array(Q[:n], np.float64)


def test_equals_the_division(divide):
    """Every result is the division's, at any scale that leaves room for the residual."""
    rng = np.random.default_rng(0)
    X, Q = _near_boundaries(rng, 200_000)
    pairs = [(X, Q), (-X * 2.0 ** -110, Q), (X * 2.0 ** 60, Q * 2.0 ** -60)]
    n = 1 << 21
    m = lambda: rng.integers(1 << 23, 1 << 24, n).astype(np.float64) * rng.choice([-1.0, 1.0], n)
    pairs.append((m() * 2.0 ** rng.integers(-63, -3, n), np.abs(m()) * 2.0 ** rng.integers(-33, -11, n)))
    pairs.append((m(), (1 << 24) - rng.integers(1, 300, n).astype(np.float64)))   # significands of ones
    pairs.append((np.zeros(4), np.array([1.0, 3.0, 1e-30, 1e30])))
    for x, q in pairs:
        a, d = divide(x.astype(np.float32), q.astype(np.float32))
        np.testing.assert_array_equal(a, d)


@pytest.mark.parametrize("record", [True, False])
@pytest.mark.parametrize("b", [np.inf, 1e-25])
def test_extreme_susceptances_in_the_gradient(b, record):
    """A line of infinite susceptance is that of a very large one; one whose
    square underflows carries nothing, whatever its limit."""
    from paper_2410_17203_gb300 import UnrolledCost
    case = make_case(scale_case(20, 4, 2, seed=8))
    line = next(l for l in range(len(case["line_b"])) if l not in set(int(o) for o in case["outaged"]))

    def at(susceptance, limit=1.0):
        c = dict(case, line_b=np.array(case["line_b"], np.float64), line_u=np.array(case["line_u"], np.float64))
        c["line_b"][line] = susceptance
        c["line_u"][line] *= limit
        d = UnrolledCost(c, rho_p=1.0, rho_theta=1.0, checkpoint_every=4)
        if not record:   # the reverse pass forms the clipping decisions again
            d.set_record_limit(0)
        f, g = d.cost_grad(8)
        d.close()
        return f, g

    f, g = at(b)
    assert np.isfinite(f) and all(np.isfinite(v).all() for v in g.values())
    f1, g1 = at(1e30) if np.isinf(b) else at(b, limit=0.25)
    assert f == pytest.approx(f1, rel=1e-6)
    for k in g:
        np.testing.assert_allclose(g[k], g1[k], rtol=1e-5, atol=1e-6 * max(1.0, np.abs(g1[k]).max()))
    if not np.isinf(b):
        assert g["line_u"][line] == 0.0
