"""The Givens update of a GMRES cycle (csrc/givens.cuh) column by column over more columns than
its shared-memory form holds: that form, the one after it, and the boundary between them,
against the same recurrence in numpy.  The header is compiled here into a small driver."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DRIVER = r"""
#include <cuda_runtime.h>
#include "givens.cuh"
__global__ void k_column(int j, int m, double nrm, double *hcol, double *H, double *cs, double *sn, double *g, double *res) {
  afmpb::givens_update_block(j, m, nrm, hcol, H, cs, sn, g, res);
}
// columns: [m][m + 1], column j = its j + 1 dots and the new norm; out: H, cs, sn, g, res by column
extern "C" int cycle(int m, const double *columns, double beta, double *H, double *cs, double *sn, double *g, double *res) {
  double *d = nullptr;
  const size_t c = m + 1, total = c * c + 5 * c;
  if (cudaMalloc(&d, sizeof(double) * total) != cudaSuccess) return 1;
  cudaMemset(d, 0xff, sizeof(double) * total);                     // NaN: nothing unwritten is read
  double *dH = d, *dcs = d + c * c, *dsn = dcs + c, *dg = dsn + c, *dres = dg + c, *dh = dres + c;
  cudaMemcpy(dg, &beta, sizeof(double), cudaMemcpyHostToDevice);
  for (int j = 0; j < m; ++j) {
    cudaMemcpy(dh, columns + j * c, sizeof(double) * (j + 1), cudaMemcpyHostToDevice);
    k_column<<<1, 256>>>(j, m, columns[j * c + j + 1], dh, dH, dcs, dsn, dg, dres + j);
  }
  cudaMemcpy(H, dH, sizeof(double) * m * c, cudaMemcpyDeviceToHost);
  cudaMemcpy(cs, dcs, sizeof(double) * m, cudaMemcpyDeviceToHost);
  cudaMemcpy(sn, dsn, sizeof(double) * m, cudaMemcpyDeviceToHost);
  cudaMemcpy(g, dg, sizeof(double) * c, cudaMemcpyDeviceToHost);
  cudaMemcpy(res, dres, sizeof(double) * m, cudaMemcpyDeviceToHost);
  const int rc = cudaDeviceSynchronize() != cudaSuccess || cudaGetLastError() != cudaSuccess;
  cudaFree(d);
  return rc;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1710_06316_gb300 import _build
    d = tmp_path_factory.mktemp("givens")
    (d / "driver.cu").write_text(DRIVER)
    so = d / "libgivens.so"
    subprocess.check_call([_build.nvcc(), *_build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                           "-I", _build.CSRC, str(d / "driver.cu"), "-o", str(so)])
    return ctypes.CDLL(str(so))


def recurrence(columns, beta):
    m = len(columns)
    R, cs, sn = np.zeros((m, m + 1)), np.zeros(m), np.zeros(m)
    g, res = np.zeros(m + 1), np.zeros(m)
    g[0] = beta
    for j in range(m):
        h = columns[j, :j + 2].copy()
        for i in range(j):
            h[i], h[i + 1] = cs[i] * h[i] + sn[i] * h[i + 1], -sn[i] * h[i] + cs[i] * h[i + 1]
        den = np.hypot(h[j], h[j + 1])
        cs[j], sn[j] = (h[j] / den, h[j + 1] / den) if den > 0 else (1.0, 0.0)
        h[j], h[j + 1] = den, 0.0
        g[j], g[j + 1] = cs[j] * g[j], -sn[j] * g[j]
        res[j] = abs(g[j + 1])
        R[j, :j + 2] = h
    return R, cs, sn, g, res


@pytest.mark.parametrize("m", [1, 2, 255, 256, 257, 300])
def test_columns_equal_the_recurrence(lib, m):
    """Rotations keep a column's norm and round each entry four times; a column meets up to m of
    them, and its rotation those of the columns before: 8 m eps of the column, m times that for
    what the cosines and sines of all columns carry on."""
    rng = np.random.default_rng(m)
    columns = np.zeros((m, m + 1))
    for j in range(m):
        columns[j, :j + 1] = 0.1 * rng.standard_normal(j + 1)
        columns[j, j] += 1.0
        columns[j, j + 1] = rng.uniform(0.2, 1.0)
    if m > 256:
        columns[256, :258] = 0.0                        # den == 0 in the form on global memory
    out = [np.full(s, np.nan) for s in ((m, m + 1), m, m, m + 1, m)]
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert lib.cycle(ctypes.c_int(m), p(columns), ctypes.c_double(3.0), *[p(a) for a in out]) == 0
    ref = recurrence(columns, 3.0)
    bar = 8 * m * m * np.finfo(float).eps
    for j in range(m):
        assert np.abs(out[0][j, :j + 2] - ref[0][j, :j + 2]).max() <= bar * max(1.0, np.linalg.norm(columns[j]))
    for a, b in zip(out[1:], ref[1:]):
        assert np.abs(a - b).max() <= bar * 3.0
