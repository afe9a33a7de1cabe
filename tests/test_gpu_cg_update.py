"""One launch of the CG update (k_cg_update) on arrays made here, through the library's own launcher.

x += alpha p, r -= alpha A p with alpha = rz / <p, A p>, the new <r, K r> and <r, r>, and the stopping
test, for rows of an odd number of elements (the last 16-byte vector of a row is half padding) in one
and in several blocks per row.
"""

import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

wdf = pytest.importorskip("paper_2607_14025_gb300.wdf")

SRC = r"""
#include "kernels.cuh"
using namespace wdf;
extern "C" int cg_update(int nint, int len0, int ld, int n, float2 *x, float2 *r, const float2 *p, const float2 *Ap, const float *K, double *rz,
                         double *beta, double *rr, double *thr, double *part1, double *part2, int *active, int *iters, int *arrived,
                         int *nactive, int *vidx, const double *dots, int ndot) {
  Geo g{};
  g.nint = nint;
  g.len0 = len0;
  g.ld = ld;
  CgState s{};
  s.rz = rz;
  s.rz_new = beta;
  s.rr = rr;
  s.thr = thr;
  s.part1 = part1;
  s.part2 = part2;
  s.active = active;
  s.iters = iters;
  s.arrived = arrived;
  s.nactive = nactive;
  s.vidx = vidx;
  try {
    launch_cg_update<float>(g, x, r, p, Ap, K, s, n, dots, ndot, 1000, 1, 0);
  } catch (...) {
    return 1;
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2607_14025_gb300 import build

    so = build.build()
    wdf.load()
    d = tmp_path_factory.mktemp("cg_update")
    src, out = d / "t.cu", d / "t.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I", build.INC, "-I",
                    build.SRC, str(src), "-o", str(out), so, "-Xlinker", "-rpath=" + os.path.dirname(so)], check=True)
    return ctypes.CDLL(str(out))


class Batch:
    """n rows of nint elements (row stride ld), every row with row 0's numbers."""

    def __init__(self, nint, n, seed=3, ndot=5):
        import torch

        ld = (nint + 31) // 32 * 32
        rng = np.random.default_rng(seed)

        def rows():
            a = np.zeros((1, ld, 2), np.float32)
            a[:, :nint] = rng.standard_normal((1, nint, 2))
            return torch.from_numpy(np.repeat(a, n, axis=0)).cuda()

        def dev(a):
            return torch.from_numpy(np.ascontiguousarray(a)).cuda()

        self.nint, self.n, self.ld, self.ndot = nint, n, ld, ndot
        self.x, self.r, self.p, self.Ap = rows(), rows(), rows(), rows()
        self.K = dev(rng.uniform(0.1, 1.0, (1, ld)).astype(np.float32))
        self.rz, self.beta, self.rr, self.thr = dev(np.full(n, 2.0)), dev(np.zeros(n)), dev(np.zeros(n)), dev(np.zeros(n))
        nch = (nint + 2047) // 2048
        self.part1, self.part2 = dev(np.zeros(n * nch)), dev(np.zeros(n * nch))
        self.active, self.iters, self.arrived = (dev(np.full(n, v, np.int32)) for v in (1, 0, 0))
        self.nactive, self.vidx = dev(np.array([7, 0], np.int32)), dev(np.zeros(n, np.int32))
        self.dots = dev(np.full((n, ndot), 1.0))

    def step(self, lib):
        import torch

        torch.cuda.synchronize()
        names = "x r p Ap K rz beta rr thr part1 part2 active iters arrived nactive vidx dots".split()
        ptr = [ctypes.c_void_p(getattr(self, k).data_ptr()) for k in names]
        assert lib.cg_update(self.nint, min(40, self.nint), self.ld, self.n, *ptr, self.ndot) == 0
        torch.cuda.synchronize()
        return {k: getattr(self, k).cpu().numpy() for k in names}


@pytest.mark.parametrize("nint,n", [(447, 5), (8455, 5), (8455, 700), (23171, 3)])
def test_breakdown_stops_the_solve_and_keeps_its_iterate(lib, nint, n):
    b = Batch(nint, n)
    b.dots[1] = -1.0  # <p, A p> < 0
    b.dots[2] = 0.0
    before = {k: getattr(b, k).cpu().numpy() for k in ("x", "r", "rz")}
    a = b.step(lib)
    for i in (1, 2):
        assert np.array_equal(a["x"][i], before["x"][i]) and np.array_equal(a["r"][i], before["r"][i])
        assert a["active"][i] == 0 and a["iters"][i] == 0 and a["rz"][i] == before["rz"][i]
    go = [i for i in range(n) if i not in (1, 2)]
    assert np.all(a["active"][go] == 1) and np.all(a["iters"][go] == 1) and not np.array_equal(a["x"][0], before["x"][0])
    assert np.all(a["arrived"] == 0) and list(a["nactive"]) == [0, n - 2]


@pytest.mark.parametrize("nint,n", [(447, 5), (2049, 3), (8455, 5), (8455, 700)])
def test_row_padding_stays_zero(lib, nint, n):
    """The padding of p and A p is never written by the library, so that of x and r must not depend on it."""
    b = Batch(nint, n)
    b.p[:, nint:] = float("nan")
    b.Ap[:, nint:] = float("nan")
    a = b.step(lib)
    for k in ("x", "r"):
        assert np.all(a[k][:, nint:] == 0.0) and np.isfinite(a[k]).all()
    assert np.isfinite(a["rr"]).all() and np.isfinite(a["rz"]).all()


@pytest.mark.parametrize("nint", [2048, 8455, 23171])
def test_sums_do_not_depend_on_the_size_of_the_batch(lib, nint):
    """<r, K r> and <r, r> of a row alone and in a batch whose blocks take four times as many elements.

    Both add the same FP32 sums of at most 8 elements, all positive, in FP64 and in another order: at most
    256 ceil(nint / 2048) additions of relative error 2^-53 each.
    """
    n = 8 * 152 // ((nint + 8191) // 8192) + 1
    one, many = Batch(nint, 1).step(lib), Batch(nint, n).step(lib)
    bar = 256 * ((nint + 2047) // 2048) * 2.0 ** -53
    for k in ("rz", "rr"):
        assert np.all(many[k] == many[k][0])
        assert abs(many[k][0] - one[k][0]) <= bar * one[k][0]
    assert np.array_equal(many["x"][0], one["x"][0]) and np.array_equal(many["r"][0], one["r"][0])
