"""The reciprocal and the inverse root behind every pivot of the factorisation, and the reflector of a column of the reduction, against
80-bit arithmetic on the host and against CUDA's own 1 / x, rsqrt, sqrt and division on the device.

The bounds, in units of 2^-53 of the value: the iteration leaves e^3 (e <= 2^-19 from the hardware's 20 bits: 2^-57, 0.07 units) besides
what rounds.  Reciprocal: the last multiply-add, 1 unit.  Inverse root: besides that the product d y, half a unit of the result,
1.5.  Reflector: the norm squared (2 units, half of which stays in the norm), the root (1.6) and two to four roundings: 8.  A start of
ten bits would leave 2^-30, 2^23 units."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_16029_b200", "csrc")
UNIT = np.longdouble(2) ** -53

SOURCE = r"""
#include <algorithm>
#include <cstring>
#include <vector>
#include "../../include/ngalore.h"
#include "common.cuh"
#include "ritz_eigen.cuh"
__global__ void scalars(const double* a, const double* s, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double beta, tau, scale;
  ngalore::eig_reflector(a[i], s[i], beta, tau, scale);
  const double nrm = sqrt(a[i] * a[i] + s[i]), b = a[i] >= 0.0 ? -nrm : nrm;
  const double v[10] = {ngalore::tf_reciprocal(s[i]), ngalore::tf_inverse_root(s[i]), beta, tau, scale,
                        1.0 / s[i], rsqrt(s[i]), b, (b - a[i]) / b, 1.0 / (a[i] - b)};
  for (int k = 0; k < 10; ++k) out[k * n + i] = v[k];
}
extern "C" int evaluate(const double* a, const double* s, double* out, int n) {
  scalars<<<(n + 127) / 128, 128>>>(a, s, out, n);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    from paper_2410_16029_b200.build import NVCC_FLAGS

    d = tmp_path_factory.mktemp("scalars")
    src, lib = d / "scalars.cu", d / "libscalars.so"
    src.write_text(SOURCE.replace('"../../include', '"' + os.path.join(CSRC, "../../include")))
    subprocess.run([os.environ.get("NVCC", "nvcc"), *NVCC_FLAGS, "-I", CSRC, "-o", str(lib), str(src)], check=True, capture_output=True)
    fn = ctypes.CDLL(str(lib)).evaluate
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]

    def run(a, s):
        x = [torch.from_numpy(np.ascontiguousarray(v, dtype=np.float64)).cuda() for v in (a, s)]
        out = torch.empty(10, len(a), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(x[0].data_ptr(), x[1].data_ptr(), out.data_ptr(), len(a)) == 0
        return out.cpu().numpy()

    return run


def _spread(lo, hi, n, seed):
    """Log-spaced, with powers of two and their neighbours, where an approximation by table changes its entry."""
    rng = np.random.default_rng(seed)
    p = 2.0 ** np.arange(np.ceil(np.log2(lo)), np.floor(np.log2(hi)))
    return np.concatenate([np.exp(rng.uniform(np.log(lo), np.log(hi), n)), p, np.nextafter(p, 0.0), np.nextafter(p, np.inf)])


def _units(got, want):
    return float(np.max(np.abs((got.astype(np.longdouble) - want) / want) / UNIT))


@pytest.mark.parametrize("lo,hi", [(1e-28, 1e4), (0.5, 2.0), (1e-280, 1e280)])
def test_reciprocal_and_inverse_root(evaluate, lo, hi):
    x = _spread(lo, hi, 1 << 18, 1)
    out = evaluate(np.zeros_like(x), x)
    e = x.astype(np.longdouble)
    print(lo, hi, _units(out[0], 1 / e), _units(out[1], 1 / np.sqrt(e)))
    assert _units(out[0], 1 / e) <= 1.1 and _units(out[1], 1 / np.sqrt(e)) <= 1.6
    # CUDA's own: 1 / x to half a unit in the last place (1 of these units), rsqrt to one (2 of them)
    assert _units(out[0], out[5].astype(np.longdouble)) <= 2.1 and _units(out[1], out[6].astype(np.longdouble)) <= 3.6


@pytest.mark.parametrize("lo,hi", [(1e-12, 1.0), (1e-152, 1e-130), (3e-141, 3e-140), (1e130, 1e152), (3e139, 3e140)])
def test_reflector(evaluate, lo, hi):
    """alpha and the square root of sigma on either side of the line where the roots and quotients come from CUDA's functions instead
    (squares of 1e-280 and 1e280)."""
    alpha, root = _spread(lo, hi, 1 << 16, 2), _spread(lo, hi, 1 << 16, 3)
    rng = np.random.default_rng(4)
    rng.shuffle(alpha), rng.shuffle(root)
    alpha *= rng.choice([-1.0, 1.0], alpha.size)
    sigma = root * root
    out = evaluate(alpha, sigma)
    a, s = alpha.astype(np.longdouble), sigma.astype(np.longdouble)
    nrm = np.sqrt(a * a + s)
    beta = np.where(a >= 0, -nrm, nrm)
    want = [beta, (beta - a) / beta, 1 / (a - beta)]
    print(lo, hi, [_units(out[2 + k], want[k]) for k in range(3)])
    for k in range(3):
        assert _units(out[2 + k], want[k]) <= 8
        assert _units(out[2 + k], out[7 + k].astype(np.longdouble)) <= 16


def test_reflector_of_a_column_that_is_done(evaluate):
    out = evaluate(np.array([0.0, 3.0, -2.0, 1.0]), np.array([0.0, 0.0, 0.0, np.nan]))
    assert np.array_equal(out[2], [0.0, 3.0, -2.0, 1.0]) and not out[3].any() and not out[4].any()
