"""The integer forms of FP64 additions, subtractions, divisions and square roots
(csrc/integer_fp64.cuh) give IEEE 754's results for every operand: numpy's, bit for
bit (any NaN for a NaN), over special values, ties, cancellation, neighbours and the
ends of the range. Needs a GPU."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2106_02159_gb300 import binding as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "integer_fp64.cuh"
__global__ void apply(const double *a, const double *b, double *out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = eh::add_alu(a[i], b[i]);
  out[n + i] = eh::sub_alu(a[i], b[i]);
  out[2 * n + i] = eh::add_abs_alu(a[i], b[i]);
  out[3 * n + i] = eh::sub_near(a[i], b[i]);
  out[4 * n + i] = eh::div_alu(a[i], b[i]);
  out[5 * n + i] = eh::sqrt_alu(a[i]);
}
extern "C" int apply_all(const double *a, const double *b, double *out, int n) {
  apply<<<(n + 127) / 128, 128>>>(a, b, out, n);
  return (int)cudaDeviceSynchronize();
}
"""


def _operands():
    rng = np.random.default_rng(11)
    bits = [0, 1, 2, (1 << 52) - 1, 1 << 52, (1 << 52) + 1, 0x7FF << 52, (0x7FF << 52) - 1, 0x7FF8 << 48]
    for e in (1, 2, 53, 69, 70, 71, 969, 1022, 1023, 1024, 1976, 2044, 2045, 2046):
        bits += [e << 52, (e << 52) + 1, (e << 52) + (1 << 51), (e << 52) + (1 << 52) - 1]
    special = np.array(bits, dtype=np.uint64)
    special = np.concatenate([special, special | np.uint64(1 << 63)])
    pairs = [np.stack(np.meshgrid(special, special), -1).reshape(-1, 2)]
    k = 200_000
    any_bits = rng.integers(0, 1 << 64, (k, 2), dtype=np.uint64)
    pairs.append(any_bits)
    near = any_bits.copy()  # exponents within 60 of one another
    near &= np.uint64(0x800FFFFFFFFFFFFF)
    near |= rng.integers(990, 1050, (k, 2)).astype(np.uint64) << np.uint64(52)
    pairs.append(near)
    close = near.copy()  # a few units in the last place apart
    close[:, 1] = close[:, 0] + rng.integers(0, 9, k).astype(np.uint64) - np.uint64(4)
    pairs.append(close)
    few = near.copy()  # short significands: exact results and ties
    few &= ~np.uint64((1 << 40) - 1)
    few[:, 1] |= rng.integers(0, 4, k).astype(np.uint64)
    pairs.append(few)
    squares = near.copy()  # neighbours of squares
    r = rng.random(k).astype(np.float32).astype(np.float64)
    squares[:, 0] = (r * r).view(np.uint64) + rng.integers(0, 3, k).astype(np.uint64)
    pairs.append(squares)
    ab = np.ascontiguousarray(np.concatenate(pairs).T)
    return ab[0].view(np.float64), ab[1].view(np.float64)


def test_integer_forms_equal_ieee(tmp_path):
    src, lib = tmp_path / "apply.cu", tmp_path / "apply.so"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", *B.NVCC_FLAGS, "-I", B.CSRC, "-o", str(lib), str(src)], check=True)
    a, b = _operands()
    n = a.size
    da, db = torch.from_numpy(a.copy()).cuda(), torch.from_numpy(b.copy()).cuda()
    out = torch.empty((6, n), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(t.data_ptr()) for t in (da, db, out)]
    assert ctypes.CDLL(os.fspath(lib)).apply_all(*p, n) == 0
    with np.errstate(all="ignore"):
        want = np.stack([a + b, a - b, np.abs(a) + np.abs(b), a - b, a / b, np.sqrt(a)])
    got = out.cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(nan, np.isnan(got))
    wrong = ~nan & (want.view(np.uint64) != got.view(np.uint64))
    for q, name in enumerate(("add", "sub", "add_abs", "sub_near", "div", "sqrt")):
        assert not wrong[q].any(), (name, a[wrong[q]][:3], b[wrong[q]][:3])
