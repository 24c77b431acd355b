"""The FP64 rounds' integer division and the two forms of their reverse messages.

* ``div64`` (devutil.cuh: the quotient of two doubles on the integer units) against CUDA's IEEE
  division: one unit in the last place over the exponent range of its fast path (its own error is
  below 0.51), equal bits where it falls back and where the quotient is exact.
* Round kernels that recompute the reverse messages (graphs whose message store is large and has no
  locality) against those that gather them: the edge-centric variant gathers and sums every row in
  the same order, so x, the residuals and every message are bitwise equal at any round, from a
  cold and from a warm start.
"""
import ctypes
import os
import subprocess
import tempfile

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r'''
#include "devutil.cuh"
__global__ void k_div(int n, const double *a, const double *d, double *q, double *ref) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { q[i] = gabp::div64(a[i], d[i]); ref[i] = a[i] / d[i]; }
}
extern "C" int div_check(int n, const double *a, const double *d, double *q, double *ref) {
  k_div<<<(n + 255) / 256, 256>>>(n, a, d, q, ref);
  return (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def gb():
    import __graft_entry__

    __graft_entry__.build()
    import paper_0811_2518_gb300 as m

    return m


@pytest.fixture(scope="module")
def div_lib():
    tmp = tempfile.mkdtemp()
    cu, so = os.path.join(tmp, "div.cu"), os.path.join(tmp, "div.so")
    open(cu, "w").write(SRC)
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "paper_0811_2518_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    "-o", so, cu], check=True)
    lib = ctypes.CDLL(so)
    lib.div_check.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 4
    lib.div_check.restype = ctypes.c_int
    return lib


def _divide(lib, a, d):
    at, dt = torch.from_numpy(a).cuda(), torch.from_numpy(d).cuda()
    q, ref = torch.empty_like(at), torch.empty_like(at)
    assert lib.div_check(a.size, at.data_ptr(), dt.data_ptr(), q.data_ptr(), ref.data_ptr()) == 0
    return q.cpu().numpy(), ref.cpu().numpy()


def test_div64_within_one_ulp(div_lib):
    rng = np.random.default_rng(7)
    n = 1_000_000
    ends = np.array([1.0, np.nextafter(1.0, 2.0), np.nextafter(2.0, 1.0), 1.5, 1.0 + 2.0 ** -23, 1.0 + 2.0 ** -22,
                     2.0 - 2.0 ** -23, 2.0 - 2.0 ** -22, 4.0 / 3.0])
    m, k = rng.uniform(1.0, 2.0, (2, n))
    m[:n // 10] = rng.choice(ends, n // 10)
    k[n // 20:n // 5] = rng.choice(ends, n // 5 - n // 20)
    e, f = rng.integers(-250, 251, (2, n))
    a = np.ldexp(m, e) * rng.choice([-1.0, 1.0], n)
    d = np.ldexp(k, f) * rng.choice([-1.0, 1.0], n)
    q, ref = _divide(div_lib, a, d)
    assert np.all(np.abs(q - ref) <= np.spacing(np.abs(ref)))
    assert np.mean(q != ref) <= 0.01  # below 0.51 ulp: nearly always IEEE's rounding


def test_div64_exact_and_fallback(div_lib):
    rng = np.random.default_rng(8)
    i, j = rng.integers(1, 1 << 26, (2, 200_000)).astype(np.float64)
    q, _ = _divide(div_lib, i * j, j)  # both products and quotients are exact
    assert np.array_equal(q, i)
    s = np.array([0.0, -0.0, 5e-324, 2.0 ** -1022, 2.0 ** -600, 1.0, -3.0, 2.0 ** 600, 1.7e308, np.inf, -np.inf, np.nan])
    a, d = np.repeat(s, s.size), np.tile(s, s.size)
    q, ref = _divide(div_lib, a, d)
    assert np.array_equal(q, ref, equal_nan=True)
    fin = np.isfinite(ref)
    assert np.array_equal(np.signbit(q[fin]), np.signbit(ref[fin]))


def _run(gb, m, b, rounds, start=None, **opts):
    s = gb.Solver.from_csr(m, history=16, warm_start=int(start is not None), **opts)
    if start is not None:
        s.set_messages(*start)
    x, st, it, rel = s.solve(b, tol=0.0, max_iter=rounds)
    out = (x, *s.messages(), torch.from_numpy(s.residual_history()), rel)
    s.close()
    return out


# the third: 300007 rows of degree ~16 recompute the reverse messages (a third lie over 32 MB away);
# the first two gather (a launch per round, one cooperative launch)
@pytest.mark.parametrize("make", [lambda: synth.grid3d(52, 1.05, 3), lambda: synth.random_sym(5003, 4, 1.1, 3),
                                  lambda: synth.random_sym(300007, 8, 1.1, 3)], ids=["grid", "coop", "recompute"])
def test_node_rounds_equal_edge_rounds(gb, make):
    m = make()
    b = torch.from_numpy(synth.rhs(m.n, 3)).cuda()
    for rounds in (1, 2, 3, 6):
        got, ref = (_run(gb, m, b, rounds, variant=v) for v in (gb.GABP_VARIANT_NODE, gb.GABP_VARIANT_EDGE))
        for g, r in zip(got[:3], ref[:3]):
            assert torch.equal(g, r), rounds
        assert torch.allclose(got[3], ref[3], rtol=1e-13, atol=0.0)  # sums over blocks of another grid
    start = ref[1:3]
    for rounds in (1, 2, 5):
        got, ref = (_run(gb, m, b, rounds, start, variant=v) for v in (gb.GABP_VARIANT_NODE, gb.GABP_VARIANT_EDGE))
        for g, r in zip(got[:3], ref[:3]):
            assert torch.equal(g, r), rounds


@pytest.mark.parametrize("n", [40, 300007])
def test_messages_of_a_run_of_no_rounds_are_zero(gb, n):
    m = synth.random_sym(n, 8, 1.1, 3)
    s = gb.Solver.from_csr(m)
    b = torch.from_numpy(synth.rhs(n, 3)).cuda()
    s.solve(b, tol=1e-10, max_iter=100)
    _, st, it, _ = s.solve(torch.zeros_like(b), tol=1e-10, max_iter=100)
    assert st == gb.GABP_OK and it == 0
    P, h = s.messages()
    assert not bool(P.any()) and not bool(h.any())
    s.close()
