"""GPU: the reciprocal square root, square root and reciprocal of the FP64 panels
(csrc/common.cuh) over every exponent, at the branches' limits and at mantissas next to
powers of two, against extended precision; and factors of matrices scaled by powers of
two over most of the range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2311_00921_gb300 import build, hss
from paper_2311_00921_gb300 import inputs as I

pytestmark = pytest.mark.gpu
LD = np.longdouble

SOURCE = r"""
#include "common.cuh"
__global__ void steps(const double* d, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double inv = inv_sqrt(d[i]);
  out[i] = inv;
  out[n + i] = sqrt_from(d[i], inv);
  out[2 * n + i] = inv_pos(d[i]);
}
extern "C" int run_steps(const double* d, int n, double* out) {
  steps<<<(n + 255) / 256, 256>>>(d, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    import torch
    folder = tmp_path_factory.mktemp("steps")
    src, lib = folder / "steps.cu", folder / "libsteps.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o",
                    str(lib), str(src)], check=True)
    run = ctypes.CDLL(os.fspath(lib)).run_steps

    def call(d):
        x = torch.as_tensor(d).cuda()
        out = torch.zeros(3, len(d), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert run(ctypes.c_void_p(x.data_ptr()), len(d), ctypes.c_void_p(out.data_ptr())) == 0
        return out.cpu().numpy()

    return call


def _bits(exponent, mantissa):
    e, m = np.broadcast_arrays(np.asarray(exponent, np.uint64), np.asarray(mantissa, np.uint64))
    return ((e << np.uint64(52)) | m).reshape(-1).view(np.float64)


def test_roots_and_reciprocals(steps):
    rng = np.random.default_rng(0)
    top = (1 << 52) - 1
    edge = np.array([0, 1, 2, top, top - 1, 1 << 51, (1 << 51) - 1, 1 << 28, top - (1 << 28)], np.uint64)
    exps = np.arange(1, 2047, dtype=np.uint64)[:, None]
    d = np.concatenate([
        _bits(exps, edge[None]), _bits(exps, rng.integers(0, 1 << 52, (2046, 40), dtype=np.uint64)),
        _bits(0, np.concatenate([edge[1:], 1 << rng.integers(0, 52, 200, dtype=np.uint64)])),
        _bits(np.array([[31], [32], [33], [2014], [2015], [2016]], np.uint64),
              rng.integers(0, 1 << 52, (6, 500), dtype=np.uint64))])
    inv, root, rec = steps(d)
    with np.errstate(over="ignore"):
        x = d.astype(LD)
        exact = (1 / np.sqrt(x), np.sqrt(x), 1 / x)
        # one rounding after 2^-63 (or CUDA's square root and division: two roundings)
        for got, ref in zip((inv, root), exact):
            assert np.all(np.abs(got - ref) <= 2.0 ** -52 * ref)
        ref = exact[2].astype(np.float64)   # overflows for the smallest, denormal for the largest
        ok = np.isfinite(ref)
        assert np.all(np.abs(rec[ok] - exact[2][ok]) <= np.maximum(2.0 ** -52 * exact[2][ok], 2.0 ** -1074))
        assert np.all(np.isinf(rec[~ok]))


def test_special_values(steps):
    inv, root, rec = steps(np.array([np.inf, np.nan]))
    assert inv[0] == 0.0 and root[0] == np.inf and rec[0] == 0.0
    assert np.isnan(inv[1]) and np.isnan(root[1]) and np.isnan(rec[1])


@pytest.mark.parametrize("exponent", [-400, -399, -63, 63, 401, 440])
def test_matrix_scaled_by_a_power_of_two(exponent):
    """2^e A has the solution 2^-e x and the log-determinant + n e log 2."""
    h = I.random_hss(2, 150, 40, seed=3)
    b = I.rhs(h.n, 3, 4)
    scale = 2.0 ** exponent

    def solve():
        dev = hss.HSS(h)
        dev.factorize("fp64")
        return dev.solve(hss.colmajor(b)).cpu().numpy(), dev.logdet()

    x, ld = solve()
    h.D = [scale * d for d in h.D]
    h.S = {l: [scale * s for s in h.S[l]] for l in h.S}
    xs, lds = solve()
    assert np.linalg.norm(xs * scale - x) <= 1e-13 * np.linalg.norm(x)
    assert abs(lds - ld - h.n * exponent * np.log(2.0)) <= 1e-12 * abs(lds)
