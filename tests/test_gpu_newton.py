"""GPU: quick_div, quick_rcp and quick_sqrt (newton.cuh) against CUDA's correctly rounded FP64
division, reciprocal and square root.

Tolerance, from the seeds' documented 20-bit mantissas: a seed is good to 2^-19, one Newton step to
2^-38, the corrected value to 2^-75 before its one rounding.  So a result is never more than one unit
in the last place from the library's, and it differs at all only where the exact value lies within
2^-75 (relative) of the middle between two numbers, 2^-53 to 2^-52 apart: at most 2^-21 of random operands,
2 expected of 2^22; 16 or more have a probability below 1e-9.  Powers of two times 2^-399 .. 2^399 are exact."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "newton.cuh"
using namespace dmrg;
__global__ void k(int op, const double* a, const double* b, long n, double* mine, double* lib) {
  for (long i = blockIdx.x * 256l + threadIdx.x; i < n; i += gridDim.x * 256l) {
    mine[i] = op == 0 ? quick_div(a[i], b[i]) : op == 1 ? quick_rcp(b[i]) : quick_sqrt(b[i]);
    lib[i] = op == 0 ? a[i] / b[i] : op == 1 ? 1.0 / b[i] : sqrt(b[i]);
  }
}
extern "C" int run(int op, const double* a, const double* b, long n, double* mine, double* lib) {
  k<<<256, 256>>>(op, a, b, n, mine, lib);
  return int(cudaDeviceSynchronize());
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1507_00161_gb300.build import CSRC, FLAGS, _nvcc
    where = tmp_path_factory.mktemp("newton")
    src, out = where / "newton.cu", where / "newton.so"
    src.write_text(SOURCE)
    subprocess.run([_nvcc(), *FLAGS, "-shared", "-I", os.fspath(CSRC), os.fspath(src), "-o", os.fspath(out)],
                   check=True)
    return ctypes.CDLL(os.fspath(out))


def _operands(kind, n, rng):
    """Positive numbers, exponents up to `span` (the square root's and quotient's ranges lie inside)."""
    if kind == "wide":      # any mantissa, 2^-399 .. 2^399
        return np.ldexp(1.0 + rng.random(n), rng.integers(-399, 399, n))
    if kind == "near one":
        return np.ldexp(1.0 + rng.random(n), rng.integers(-1, 2, n))
    if kind == "edges":     # mantissas close to a power of two from both sides, ends of the range
        x = np.ldexp(1.0, rng.integers(-398, 399, n))
        return np.maximum(x + rng.integers(-4, 5, n) * np.spacing(x), 2.0 ** -399)
    if kind == "low bits":  # all of the lower 32 bits set, which the seeds ignore
        x = np.ldexp(1.0 + rng.random(n), rng.integers(-399, 399, n))
        return (x.view(np.uint64) | np.uint64(0xffffffff)).view(np.float64)
    # squares and products of 26-bit mantissas, and their neighbours: roots and quotients near ties
    m = rng.integers(2 ** 26, 2 ** 27, n).astype(np.float64)
    x = m * rng.integers(2 ** 25, 2 ** 26, n) if kind == "products" else m * m
    return x + rng.integers(-1, 2, n) * np.spacing(x)


@pytest.mark.parametrize("op", [0, 1, 2])
@pytest.mark.parametrize("kind", ["wide", "near one", "edges", "low bits", "products", "squares"])
def test_against_the_library(lib, op, kind):
    n = 2 ** 22
    rng = np.random.default_rng(17)
    a, b = _operands(kind, n, rng), _operands(kind, n, rng)
    if op == 0:   # quotients stay normal
        b = np.ldexp(np.frexp(b)[0], np.frexp(b)[1] % 180)
    dev = [torch.from_numpy(v).cuda() for v in (a, b)] + [torch.empty(n, dtype=torch.float64, device="cuda")
                                                         for _ in range(2)]
    assert lib.run(op, *(ctypes.c_void_p(v.data_ptr()) for v in dev[:2]), ctypes.c_long(n),
                   *(ctypes.c_void_p(v.data_ptr()) for v in dev[2:])) == 0
    mine, ref = (v.cpu().numpy() for v in dev[2:])
    ulp = np.abs(mine.view(np.int64) - ref.view(np.int64))
    print(f"\n[newton] op {op}, {kind}: {np.count_nonzero(ulp)} of {n} differ, at most {ulp.max()} ulp")
    assert ulp.max() <= 1
    if kind in ("wide", "near one", "low bits"):
        assert np.count_nonzero(ulp) < 16
