"""The half-warp additive-CCD iteration when its lanes would read different
bounds: other warps lower the bound of the smallest t_p while a half reads it,
so only the leader's reading may count.  The job here answers every such
question differently on the leader and on the other 15 lanes; results are the
oracle's iteration under the leader's answers."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_2510_10256_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "accd16.cuh"
struct Job {
  const double *x, *p, *off;
  const unsigned char *ee, *want;
  int n;
  double bound;
  double* t;
  int* how;
  long long q;
  __device__ int wanted(long long w) const { return cba::half_leader() ? want[w] : !want[w]; }
  __device__ bool load(long long w, cba::Pair16& S) {
    q = w;
    S.off = off[w];
    return cba::load16(x, p, n, (int)(4 * w) + cba::quad_vertex(), ee[w] != 0, S);
  }
  __device__ bool begin(cba::Pair16& S, double d) {
    const double g0 = xsub(d, S.off);
    S.hi = 1.0;
    S.g = xmul(0.1, g0);
    S.tl = xdiv(xmul(xsub(1.0, 0.1), g0), S.lp);
    if (isinf(bound)) S.off = -NAN;  // every later gap is NaN, its sign set (as in inf - inf on the device)
    return true;
  }
  __device__ double cap() const { return cba::half_leader() ? bound : (threadIdx.x & 1 ? 0.0 : 1e-3); }
  __device__ void done(const cba::Pair16&, double v, cba::Done h) const {
    if (!cba::half_leader()) return;
    t[q] = v;
    how[q] = (int)h;
  }
};
__global__ void __launch_bounds__(128) k(Job J, long long m) {
  cba::iterate16(J, m, 4 * (int)gridDim.x, (int)(threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x, 0.9, 10000);
}
extern "C" int run(const double* x, const double* p, const double* off, const unsigned char* ee,
                   const unsigned char* want, int n, double bound, double* t, int* how, long long m, int blocks) {
  k<<<blocks, 128>>>(Job{x, p, off, ee, want, n, bound, t, how, 0}, m);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def so(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("halves")
    src, out = str(d / "halves.cu"), str(d / "halves.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", src, "-o", out], check=True)
    assert os.path.exists(out)
    L = C.CDLL(out)
    L.run.argtypes = [C.c_void_p] * 5 + [C.c_int, C.c_double, C.c_void_p, C.c_void_p, C.c_longlong, C.c_int]
    return L


def _pairs(m, seed):
    """Stencils whose two parts close in on each other at various speeds."""
    rng = np.random.default_rng(seed)
    x = rng.uniform(-1.0, 1.0, (m, 4, 3))
    ee = rng.random(m) < 0.5
    first = np.where(ee[:, None], np.array([1, 1, 0, 0], bool), np.array([1, 0, 0, 0], bool))
    x[..., 2] += np.where(first, 3.0, 0.0)
    p = rng.normal(0.0, 0.2, (m, 4, 3))
    p[..., 2] -= np.where(first, rng.uniform(1.0, 12.0, (m, 1)), 0.0)
    return x, p, ee


@pytest.mark.parametrize("m,blocks", [(1, 1), (7, 1), (64, 2), (203, 3)])
@pytest.mark.parametrize("bound", [1.0, 0.4])
def test_only_the_leaders_reading_counts(so, m, blocks, bound):
    import torch
    dev = torch.device("cuda:0")
    x, p, ee = _pairs(m, m)
    off = np.full(m, 0.0625)
    want = np.arange(m) % 3 != 1
    ref = np.array([O.accd(bool(ee[k]), x[k].reshape(-1), p[k].reshape(-1), off[k])[0] for k in range(m)])

    def on(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    bufs = [on(x.reshape(-1, 3).T), on(p.reshape(-1, 3).T), on(off), on(ee.astype(np.uint8)), on(want.astype(np.uint8))]
    t = torch.full((m,), -1.0, dtype=torch.float64, device=dev)
    how = torch.full((m,), -1, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    assert so.run(*[b.data_ptr() for b in bufs], 4 * m, bound, t.data_ptr(), how.data_ptr(), m, blocks) == 0
    t, how = t.cpu().numpy(), how.cpu().numpy()
    assert np.all(how[~want] == -1) and np.all(how[want] >= 0)
    if bound == 1.0:  # no bound: every wanted pair to its end
        assert np.all(how[want] == 0) and np.array_equal(t[want], ref[want])
    else:             # stopped at the first iterate that reaches the bound
        stop, below = want & (how == 1), want & (ref < 1.0)
        assert np.array_equal(stop[below], ref[below] >= bound)
        assert np.all((t[stop] >= bound) & (t[stop] <= ref[stop]))
        assert np.array_equal(t[want & ~stop], ref[want & ~stop])  # (1 may be reached in one step across the bound)


@pytest.mark.parametrize("m", [1, 5])
def test_a_gap_that_is_no_number_ends_nothing(so, m):
    """As in the one-lane iteration, whose comparisons with NaN are false: only
    the limit of steps ends such a pair."""
    import torch
    dev = torch.device("cuda:0")
    x, p, ee = _pairs(m, 50 + m)
    p *= 8.0  # the first step stays below 1

    def on(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    bufs = [on(x.reshape(-1, 3).T), on(p.reshape(-1, 3).T), on(np.full(m, 0.0625)), on(ee.astype(np.uint8)),
            on(np.ones(m, np.uint8))]
    t = torch.full((m,), -1.0, dtype=torch.float64, device=dev)
    how = torch.full((m,), -1, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    assert so.run(*[b.data_ptr() for b in bufs], 4 * m, float("inf"), t.data_ptr(), how.data_ptr(), m, 1) == 0
    assert np.all(how.cpu().numpy() == 2) and np.all(np.isnan(t.cpu().numpy()))
