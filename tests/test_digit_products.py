"""Products of digit planes (options f64_tc), one by one against double-double sums, in the
forms the library uses them: through the epilogue, as a dense product, with K split; rows of
every spread, every row and column of its own magnitude, K beyond 65536 (guard bits of the
integer sums), more tiles than SMs with ragged rows.

Seven planes: with 2^e, 2^f the powers of two above the largest magnitudes of a row and a
column, the cut leaves 2^-56 2^e in every element, the products that are not formed
2^-61.6 2^(e+f) per k, the FP32 sum of the low digit levels (6 x 2^-40 2^(e+f) per k at most)
2^-24 of itself per chunk of 256, and the result is rounded once:
  2^-56 (2^e sum|b| + 2^f sum|a|) + K (1 + K / 256) 2^-60 2^(e+f) + 2^-53 |c|.
Six planes: 2^-36 K 2^(e+f)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2607_00981_gb300.build import CSRC, nvcc

from ._helpers import gpu_lib

SRC = r"""
#include <vector>
#include "elem.cuh"
#include "kernels.h"
using namespace rcc;
// form 0: the epilogue, 1: dense [N][M], 2: K split.  C [M][N] of the host; nonzero on an error.
extern "C" int product(int ns, int form, const double* A, const double* B, int M, int N, int K, int Kpad, double* C) {
  std::vector<void*> mem;
  auto dev = [&](const void* h, size_t n) {
    void* p = nullptr;
    if (cudaMalloc(&p, n) != cudaSuccess) return (void*)nullptr;
    mem.push_back(p);
    if (h) cudaMemcpy(p, h, n, cudaMemcpyHostToDevice);
    else cudaMemset(p, 0, n);
    return p;
  };
  std::vector<i64> rb(M), co(N);
  std::vector<int> rs(M, 0);
  std::vector<double> al(M, 1.0);
  for (int m = 0; m < M; ++m) rb[m] = (i64)m * N;
  for (int n = 0; n < N; ++n) co[n] = n;
  double *a = (double*)dev(A, (size_t)M * Kpad * 8), *b = (double*)dev(B, (size_t)N * Kpad * 8);
  double* c = (double*)dev(nullptr, (size_t)M * N * 8);
  EpiArgs e{};
  e.C = c;
  e.M = M;
  e.N = N;
  e.row_base = (const i64*)dev(rb.data(), M * sizeof(i64));
  e.row_sel = (const int*)dev(rs.data(), M * sizeof(int));
  e.row_alpha = (const double*)dev(al.data(), M * sizeof(double));
  e.col_off = (const i64*)dev(co.data(), N * sizeof(i64));
  const i64 words = 4 << 20;
  double* scratch = (double*)dev(nullptr, words * 8);
  int* status = (int*)dev(nullptr, 8);
  void *pa = dev(nullptr, (size_t)ns * M * Kpad * 2), *pb = dev(nullptr, (size_t)ns * N * Kpad * 2);
  int *ea = (int*)dev(nullptr, M * 4), *eb = (int*)dev(nullptr, N * 4);
  for (int q = 0; q < 2; ++q) {
    const double* x = q ? b : a;
    if (ns == kSlicesX) launch_slice_f64x(x, q ? N : M, Kpad, q ? pb : pa, q ? eb : ea, 0);
    else launch_slice_f64(x, q ? N : M, Kpad, q ? pb : pa, q ? eb : ea, 0);
  }
  int st = launch_gemm_f64e(pa, ea, pb, eb, Kpad, ns, e, status, 0, form == 2 ? scratch : nullptr, words, 0,
                            form == 1 ? c : nullptr);
  std::vector<double> h((size_t)M * N);
  if (cudaMemcpy(h.data(), c, h.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess) st = 1;
  int flag = 0;
  cudaMemcpy(&flag, status, 4, cudaMemcpyDeviceToHost);
  for (int m = 0; m < M; ++m)
    for (int n = 0; n < N; ++n) C[(size_t)m * N + n] = form == 1 ? h[(size_t)n * M + m] : h[(size_t)m * N + n];
  for (void* p : mem) cudaFree(p);
  return st || flag;
}
"""


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    gpu_lib()
    d = tmp_path_factory.mktemp("products")
    (d / "p.cu").write_text(SRC)
    so, lib = str(d / "p.so"), os.path.dirname(CSRC)
    subprocess.run([nvcc(), "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "-shared", "-I", CSRC, str(d / "p.cu"), "-o", so, "-L", lib, "-l:librccsdt.so", "-Xlinker",
                    "-rpath=" + lib, "-lcuda"], check=True, capture_output=True)
    fn = C.CDLL(so).product
    fn.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_void_p] + [C.c_int] * 4 + [C.c_void_p]

    def run(ns, form, A, B):
        (M, K), N = A.shape, B.shape[0]
        kpad = (K + 63) // 64 * 64
        a, b = np.zeros((M, kpad)), np.zeros((N, kpad))
        a[:, :K], b[:, :K] = A, B
        out = np.zeros((M, N))
        assert fn(ns, form, a.ctypes.data, b.ctypes.data, M, N, K, kpad, out.ctypes.data) == 0
        return out

    return run


def _exact(A, B):
    """sum_k a_k b_k in double-double (TwoProduct by splitting, TwoSum)."""
    def split(x):
        t = 134217729.0 * x
        h = t - (t - x)
        return h, x - h

    hi, lo = np.zeros((A.shape[0], B.shape[0])), np.zeros((A.shape[0], B.shape[0]))
    for k in range(A.shape[1]):
        a, b = A[:, k, None], B[None, :, k]
        p = a * b
        (ah, al), (bh, bl) = split(a), split(b)
        e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
        s = hi + p
        t = s - hi
        lo += ((hi - (s - t)) + (p - t)) + e
        hi = s
    return hi, lo


def _rows(kind, M, N, K, rng):
    A, B = rng.standard_normal((M, K)), rng.standard_normal((N, K))
    if kind.startswith("spike"):  # one large element per row, which meets a zero
        k = rng.integers(0, K, M)
        A[np.arange(M), k] = float(kind[5:])
        B[:, k] = 0.0
    elif kind.startswith("graded"):  # rows and columns graded against each other
        g = np.exp(np.linspace(0, np.log(float(kind[6:])), K))
        A, B = A * g, B * g[::-1]
    elif kind.startswith("lognormal"):
        w = float(kind[9:])
        A, B = A * np.exp(w * rng.standard_normal(A.shape)), B * np.exp(w * rng.standard_normal(B.shape))
    elif kind == "scales":  # every row and column of its own magnitude
        A *= 2.0 ** rng.integers(-200, 200, (M, 1))
        B *= 2.0 ** rng.integers(-200, 200, (N, 1))
    elif kind == "zeros":  # rows of zeros, and rows without a common nonzero
        A[::3], B[1::4] = 0.0, 0.0
        A[1::3, : K // 2], B[2::4, K // 2:] = 0.0, 0.0
    elif kind == "equal":  # one rounding error many times over
        A[:, 1:], B[:] = 0.1, 0.3
        A[:, 0] = 1.0
    return A, B


def _within(out, A, B, ns):
    K = A.shape[1]
    hi, lo = _exact(A, B)
    top = [2.0 ** np.where(x.any(1), np.frexp(np.abs(x).max(1))[1], -1000.0) for x in (A, B)]
    guard = 0
    while ns == 7 and 65536 << (2 * guard) < K:
        guard += 1
    top = [t * 2.0 ** guard for t in top]
    both = top[0][:, None] * top[1]
    bar = 2.0 ** -36 * K * both
    if ns == 7:
        bar = (2.0 ** -56 * (top[0][:, None] * np.abs(B).sum(1) + top[1] * np.abs(A).sum(1)[:, None])
               + K * (1 + K / 256) * 2.0 ** -60 * both + 2.0 ** -53 * np.abs(hi))
    err = np.abs((out - hi) - lo)
    assert np.all(err <= bar), (err / np.maximum(bar, 1e-300)).max()


KINDS = ["normal", "scales", "equal", "spike1e2", "spike1e6", "graded1e-4", "graded1e-8", "lognormal3", "zeros"]


@pytest.mark.gpu
@pytest.mark.parametrize("form", [0, 1, 2], ids=["epilogue", "dense", "k-split"])
@pytest.mark.parametrize("ns", [6, 7])
@pytest.mark.parametrize("kind", KINDS)
def test_rows_of_every_spread(product, kind, ns, form):
    A, B = _rows(kind, 150, 70, 2000, np.random.default_rng(5))
    _within(product(ns, form, A, B), A, B, ns)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (31, 33, 16), (129, 65, 47), (128, 64, 64), (33, 20, 65600), (1300, 1000, 60)])
@pytest.mark.parametrize("ns", [6, 7])
@pytest.mark.parametrize("form", [0, 1, 2], ids=["epilogue", "dense", "k-split"])
def test_edges_of_tiles_and_of_the_integer_sums(product, M, N, K, ns, form):
    rng = np.random.default_rng(K)
    A, B = rng.uniform(0.5, 1.0, (M, K)), rng.uniform(0.5, 1.0, (N, K))  # all of one sign: the longest sums
    _within(product(ns, form, A, B), A, B, ns)


@pytest.mark.gpu
def test_seven_planes_on_even_rows_are_below_an_fp64_chain(product):
    """Where the terms are of one magnitude the error is an FP64 sum's or less."""
    A, B = _rows("normal", 150, 70, 2000, np.random.default_rng(9))
    hi, lo = _exact(A, B)
    chain = np.zeros(hi.shape)
    for k in range(A.shape[1]):
        chain += A[:, k, None] * B[None, :, k]
    rms = [np.sqrt(np.mean(((x - hi) - lo) ** 2)) for x in (product(7, 0, A, B), product(7, 2, A, B), chain)]
    assert max(rms[:2]) < rms[2]


@pytest.mark.gpu
@pytest.mark.parametrize("ns", [6, 7])
def test_nonfinite_rows_and_columns_give_nan(product, ns):
    rng = np.random.default_rng(2)
    A, B = rng.standard_normal((70, 100)), rng.standard_normal((70, 100))
    A[3, 7], A[40, 2], B[66, 1] = np.inf, np.nan, -np.inf
    out = product(ns, 0, A, B)
    bad = np.zeros((70, 70), dtype=bool)
    bad[[3, 40]] = True
    bad[:, 66] = True
    assert np.array_equal(np.isnan(out), bad) and np.all(np.isfinite(out[~bad]))
