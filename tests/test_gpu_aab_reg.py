"""AAb_Solver with SA in registers, at the edges of its splits, against the oracle."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest
import torch

from oracle import mihs_oracle as o
from paper_1912_03514_gb300 import _build, mihs
from paper_1912_03514_gb300 import workloads as W
from tests._tol import U32
from tests.test_gpu_parity import _fp32_amplification, _sa_case

pytestmark = pytest.mark.gpu
DEV = "cuda"


# m, d: one block and one row or column more than it holds, per width of the kernel (256, 512, 1024, 2048 columns),
# each count of rows per warp, column slices narrower than a warp, a last block without rows or columns, the largest
# sketch of 16 blocks and the first that leaves this form
SPLITS = [(1, 1), (8, 4), (9, 5), (32, 256), (33, 255), (160, 256), (161, 256), (80, 512), (81, 509), (40, 1024),
          (41, 1021), (16, 2048), (17, 2045), (96, 640), (320, 1024), (321, 1024), (640, 1024), (641, 1024),
          (256, 2048), (257, 2048), (1281, 257), (2560, 64), (1279, 300), (130, 36)]


@pytest.mark.parametrize("m,d", SPLITS)
def test_register_form_matches_oracle(m, d):
    lam, k = 0.3, 12
    SA, g = _sa_case(m, d, 7 * m + d)
    amp, ref = _fp32_amplification(SA.numpy().astype(np.float64), g.numpy().astype(np.float64), lam, k)
    pad = torch.full((m, d + 3), float("nan"))  # rows that are not 16-byte aligned, with NaN beyond them
    pad[:, :d] = SA
    passes = torch.zeros(1, dtype=torch.int32, device=DEV)
    delta = mihs.aab_solve(SA.to(DEV), g.to(DEV), lam, eps_sub=0.0, max_inner=k, passes=passes)
    assert int(passes.item()) == min(k, m, d)
    tol = 20 * max(amp, 4 * U32 * math.sqrt(d))
    assert o.rel_error(delta.double().cpu().numpy(), ref) <= tol
    if m * d <= 600_000:  # larger sketches need aligned rows in their other form
        delta2 = mihs.aab_solve(pad.to(DEV)[:, :d], g.to(DEV), lam, eps_sub=0.0, max_inner=k)
        assert torch.equal(delta, delta2)
    assert mihs.device_status() == 0


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
@pytest.mark.parametrize("m,d", [(40, 1024), (130, 36), (257, 300), (200, 2048)])
def test_register_form_decodes_quantised(m, d, prec):
    """The quantised sketch gives what its decoded values give in fp32 storage, bit by bit."""
    SA, g = _sa_case(m, d, 11 * m + d)
    q, sc = mihs.quantize_sa(SA.to(DEV), prec)
    if prec == "bf16":
        dec = q[:, :d].float()
    else:
        f = q.view(torch.float8_e4m3fn)[:, :d].float()
        dec = f * sc.repeat_interleave(128, 0)[:m].repeat_interleave(128, 1)[:, :d]
    a = mihs.aab_solve_q(q, prec, sc, d, g.to(DEV), 0.3, eps_sub=0.0, max_inner=9)
    b = mihs.aab_solve(dec.contiguous(), g.to(DEV), 0.3, eps_sub=0.0, max_inner=9)
    assert torch.equal(a, b)


NORM_KERNEL = """
#include "aab_kernel.cuh"
__global__ void norms(const float* x, float* nrm, float* inv, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) mihs::aabk::norm_of(x[i], nrm[i], inv[i]);
}
extern "C" int run(const float* x, float* nrm, float* inv, int n) {
  norms<<<(n + 255) / 256, 256>>>(x, nrm, inv, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_norm_and_reciprocal_are_rounded_like_ieee(tmp_path):
    """Every exponent of fp32, both lines between the two ways of computing them, zero, infinity and NaN: within half
    a unit in the last place and a thousandth of the root, and of the rounded root's reciprocal."""
    src, so = tmp_path / "norms.cu", tmp_path / "norms.so"
    src.write_text(NORM_KERNEL)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-I", _build.CSRC, "-shared", str(src), "-o", str(so)],
                   check=True)
    rng = np.random.default_rng(5)
    bits = rng.integers(1, 0x7F800000, 1 << 21, dtype=np.int64).astype(np.uint32)  # all exponents alike
    line = np.array([1e-30, 3e38], np.float32).view(np.uint32)
    near = (line[:, None].astype(np.int64) + np.arange(-300, 301)).reshape(-1).astype(np.uint32)
    four = (np.float32(1).view(np.uint32) + np.arange(1 << 20, dtype=np.int64) * 16).astype(np.uint32)  # [1, 4)
    x = np.concatenate([bits, near, four, np.array([0, 1, 0x7F7FFFFF], np.uint32)]).view(np.float32)
    xd = torch.from_numpy(np.concatenate([x, np.array([np.inf, np.nan], np.float32)])).to(DEV)
    nd, vd = torch.empty_like(xd), torch.empty_like(xd)
    lib = ctypes.CDLL(os.fspath(so))
    p = ctypes.c_void_p
    assert lib.run(p(xd.data_ptr()), p(nd.data_ptr()), p(vd.data_ptr()), ctypes.c_int(xd.numel())) == 0
    nrm, inv = nd.cpu().numpy(), vd.cpu().numpy()
    assert np.isposinf(nrm[-2]) and inv[-2] == 0 and np.isnan(nrm[-1]) and np.isnan(inv[-1])
    assert nrm[-5] == 0 and np.isposinf(inv[-5])
    nrm, inv = nrm[:-2], inv[:-2]
    on = x > 0
    half = 0.5 + 2.0 ** -10
    assert np.all(np.abs(nrm - np.sqrt(x.astype(np.float64))) <= half * np.spacing(nrm))
    want = 1.0 / nrm[on].astype(np.float64)
    assert np.all(np.abs(inv[on] - want) <= half * np.spacing(want.astype(np.float32)))
