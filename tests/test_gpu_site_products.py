"""The integer inner products of two sites' 24 doubles (fx_products of wd_fixed.cuh)
on the device, against exact rational arithmetic."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KERNEL = """
#include "wd_fixed.cuh"
__global__ void products(int n, const double* w, const double* a, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double wv[24], av[24], norm2 = 0;
  double2 dot = make_double2(0, 0);
  for (int k = 0; k < 24; ++k) {
    wv[k] = w[24 * i + k];
    av[k] = a[24 * i + k];
  }
  const bool taken = wd::fx_products(wv, av, norm2, dot);
  out[4 * i] = taken;
  out[4 * i + 1] = norm2;
  out[4 * i + 2] = dot.x;
  out[4 * i + 3] = dot.y;
}
extern "C" int run(int n, const double* w, const double* a, double* out) {
  products<<<(n + 63) / 64, 64>>>(n, w, a, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def products(tmp_path_factory):
    import torch

    from paper_0911_3191_gb300 import build
    d = tmp_path_factory.mktemp("products")
    src, lib = d / "products.cu", d / "products.so"
    src.write_text(KERNEL)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", os.path.abspath(build.CSRC), "-shared", "-o",
                    str(lib), str(src)], check=True, capture_output=True)
    fn = ctypes.CDLL(str(lib)).run

    def call(w, a):
        dw, da = torch.from_numpy(w).cuda(), torch.from_numpy(a).cuda()
        out = torch.zeros((len(w), 4), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert fn(len(w), *(ctypes.c_void_p(t.data_ptr()) for t in (dw, da, out))) == 0
        return out.cpu().numpy()
    return call


def _exact(w, a):
    w, a = [Fraction(float(x)) for x in w], [Fraction(float(x)) for x in a]
    re = sum(p * q for p, q in zip(w, a))
    im = sum(w[k] * a[k + 1] - w[k + 1] * a[k] for k in range(0, 24, 2))
    return sum(x * x for x in a), re, im


def _modulus(x):
    return np.hypot(x[::2], x[1::2])


@pytest.mark.parametrize("spread", [0, 10, 40, "disjoint", "zeros"])
def test_products_no_worse_than_fp64(products, spread):
    """Every product that the integers take is off by no more than 24 FP64 multiply-adds may be, 24 x 2^-53 of the
    sum of |w| |a|.  Gaussian sites are taken, and so are zeros; sites whose large numbers do not meet are not."""
    rng = np.random.default_rng(41)
    n = 400
    w, a = rng.normal(size=(n, 24)), rng.normal(size=(n, 24))
    if spread == "disjoint":  # 1 beside 2^-20 ... 2^-40, elsewhere in the other vector
        small = np.exp2(-20 - 20 * rng.random((n, 12)))
        w[:, 12:] *= small
        a[:, :12] *= small
    elif spread == "zeros":
        w[:100], a[100:200] = 0.0, 0.0
        w[200:, 4:], a[200:, 6:] = 0.0, -0.0
    else:
        w *= np.exp2(-spread * rng.random((n, 24)))
        a *= np.exp2(-spread * rng.random((n, 24)))
    out = products(w, a)
    taken = out[:, 0] == 1
    if spread == 0 or spread == "zeros":
        assert taken[:200].all()
    if spread == "disjoint":
        assert not taken.any()
    for i in np.flatnonzero(taken):
        norm2, re, im = _exact(w[i], a[i])
        terms = float((_modulus(w[i]) * _modulus(a[i])).sum())
        err = [abs(Fraction(float(got)) - want) for got, want in zip(out[i, 1:], (norm2, re, im))]
        assert err[0] <= 24 * 2.0 ** -53 * float(norm2), i
        assert max(err[1:]) <= 24 * 2.0 ** -53 * terms, i
