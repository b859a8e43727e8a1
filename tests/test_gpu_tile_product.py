"""The 32 x 32 x 32 tile products of the blocked dense routines (csrc/common.cuh,
tile_product), one tile at a time, against exact integer arithmetic.

Bound: an FMA chain over n products errs by at most n 2^-53 sum_t |A_rt B_tc|.
The fixed-point product has to stay within the same bound wherever that sum is
at least 2^-20 of max_t |A_rt| max_t |B_tc| (its own absolute error is 2^-74 of
the product of the maxima, after the inner index is balanced where the routine
asks for it); below that it has to stay within 2^-74 of the product itself.
"""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_01728_gb300", "csrc")
NB = 32

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "common.cuh"
using namespace dpgmg;
namespace dpgmg { void count_launch() {} }

// A: [r][t], B: [t][c], row-major 32 x 32, columns t >= kb zero
template <class T, bool BT, bool AT, bool BAL>
__global__ void __launch_bounds__(CTA_THREADS) k_tile(const T* A, const T* B, T* C, int kb) {
  extern __shared__ __align__(16) unsigned char raw[];
  T* At = reinterpret_cast<T*>(raw);
  T *Bt = At + TL * NB, *Z = Bt + NB * TL;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T a[4], b[4], acc[4];
  for (int i = 0; i < 4; ++i) {
    a[i] = AT ? A[lane * NB + 4 * w + i] : A[(4 * w + i) * NB + lane];
    b[i] = BT ? B[lane * TL + 4 * w + i] : B[(4 * w + i) * TL + lane];
    acc[i] = Ops<T>::zero();
  }
  tile_product<T, BT, AT, BAL>(a, b, At, Bt, Z, kb, acc);
  for (int q = 0; q < 4; ++q) C[(w + 8 * q) * TL + lane] = acc[q];
}

template <class T>
static void run(int variant, int kb, const T* A, const T* B, T* C) {
  const size_t sm = 3 * NB * NB * sizeof(T);
#define GO(BT, AT, BAL)                                                                                        \
  cudaFuncSetAttribute(k_tile<T, BT, AT, BAL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);            \
  k_tile<T, BT, AT, BAL><<<1, CTA_THREADS, sm>>>(A, B, C, kb)
  switch (variant) {
    case 0: GO(true, false, false); break;
    case 1: GO(false, false, false); break;
    case 2: GO(false, true, false); break;
    case 3: GO(false, true, true); break;
    default: GO(false, false, true); break;
  }
}

int main(int argc, char** argv) {
  FILE* in = fopen(argv[1], "rb");
  FILE* out = fopen(argv[2], "wb");
  int h[3];   // variant, kb, doubles per entry
  double *A, *B, *C;
  const size_t most = 2 * NB * NB;
  cudaMalloc(&A, most * 8);
  cudaMalloc(&B, most * 8);
  cudaMalloc(&C, most * 8);
  std::vector<double> v(most);
  while (fread(h, 4, 3, in) == 3) {
    const size_t n = (size_t)h[2] * NB * NB;
    for (double* d : {A, B}) {
      if (fread(v.data(), 8, n, in) != n) return 2;
      cudaMemcpy(d, v.data(), n * 8, cudaMemcpyHostToDevice);
    }
    if (h[2] == 1) run<double>(h[0], h[1], A, B, C);
    else run<double2>(h[0], h[1], (double2*)A, (double2*)B, (double2*)C);
    cudaMemcpy(v.data(), C, n * 8, cudaMemcpyDeviceToHost);
    fwrite(v.data(), 8, n, out);
  }
  if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return 3;
  fclose(out);
  return 0;
}
"""

VARIANTS = {"rows of B^T": 0, "plain": 1, "rows of A^T": 2, "rows of A^T, balanced": 3, "plain, balanced": 4}


def matrix(rng, kb, cplx):
    shape = (NB, NB)
    A, B = rng.standard_normal(shape), rng.standard_normal(shape)
    if cplx:
        A, B = A + 1j * rng.standard_normal(shape), B + 1j * rng.standard_normal(shape)
    return A, B


def make(kind, rng, kb, cplx):
    A, B = matrix(rng, kb, cplx)
    if kind == "scaled":          # rows of A and columns of B over 200 decades
        A = A * 10.0 ** rng.uniform(-100, 100, NB)[:, None]
        B = B * 10.0 ** rng.uniform(-100, 100, NB)[None, :]
    elif kind == "inverse":       # A diag(d), diag(1 / d) B with d over 12 decades
        d = 10.0 ** rng.uniform(-6, 6, NB)
        A, B = A * d[None, :], B / d[:, None]
    elif kind == "shadowed":      # the largest entries of A meet the smallest of B: their products are 2^-18
        big = np.arange(NB) % 2 == 0   # of the product of the maxima
        A = A * np.where(big, 1.0, 2.0 ** -18)[None, :]
        B = B * np.where(big, 2.0 ** -18, 1.0)[:, None]
        A, B = A[rng.permutation(NB)], B
    elif kind == "spread":        # every entry with its own magnitude
        A = A * 10.0 ** rng.uniform(-6, 0, A.shape)
        B = B * 10.0 ** rng.uniform(-6, 0, B.shape)
    elif kind == "zeros":
        A[rng.random(A.shape) < 0.7] = 0
        A[3], B[:, 5], B[min(2, kb - 1)] = 0, 0, 0
    elif kind == "top":           # exponents at the top of the range
        A, B = A * 2.0 ** 1021, B * 2.0 ** -40
    elif kind == "small":
        A, B = A * 1e-150, B * 1e-150
    A[:, kb:], B[kb:] = 0, 0
    return A, B


def exact(A, B):
    """(integers, power of two): A B exactly, and sum |A| |B| in floating point."""
    def ints(M):
        m, e = np.frexp(M)
        e0 = int(e[M != 0].min()) if np.any(M != 0) else 0
        return np.array([[int(x * 2.0 ** 53) << max(int(k) - e0, 0) if x else 0 for x, k in zip(r, q)]
                         for r, q in zip(m, e)], dtype=object), e0 - 53
    (a, ea), (b, eb) = ints(A), ints(B)
    return a.dot(b), ea + eb


def to_float(n, e):
    """n 2^e to the nearest double (n an integer)."""
    if n == 0:
        return 0.0
    s = max(n.bit_length() - 60, 0)
    return float(np.ldexp(float(n >> s if s else n), e + s))


def errors(C, A, B):
    P, e = exact(A, B)
    err = np.empty((NB, NB))
    for r in range(NB):
        for c in range(NB):
            m, k = np.frexp(C[r, c])
            x, ke = int(m * 2.0 ** 53), int(k) - 53
            lo = min(ke, e)
            err[r, c] = abs(to_float((x << (ke - lo)) - (int(P[r, c]) << (e - lo)), lo))
    return err


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("tile")
    (d / "driver.cu").write_text(DRIVER)
    subprocess.run([nvcc, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "driver.cu"), "-o", str(d / "driver")],
                   check=True)

    def run(cases):
        with open(d / "in", "wb") as f:
            for variant, kb, A, B in cases:
                cplx = np.iscomplexobj(A)
                f.write(struct.pack("3i", variant, kb, 2 if cplx else 1))
                for M in (A, B):
                    f.write(np.ascontiguousarray(M, dtype=np.complex128 if cplx else np.float64).tobytes())
        subprocess.run([str(d / "driver"), str(d / "in"), str(d / "out")], check=True)
        raw, out, o = (d / "out").read_bytes(), [], 0
        for _, _, A, _ in cases:
            t = np.complex128 if np.iscomplexobj(A) else np.float64
            n = NB * NB * np.dtype(t).itemsize
            out.append(np.frombuffer(raw[o:o + n], dtype=t).reshape(NB, NB))
            o += n
        return out
    return run


KINDS = ["normal", "scaled", "shadowed", "spread", "zeros", "top", "small"]


@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("variant", list(VARIANTS))
def test_tiles_against_exact_products(driver, variant, cplx):
    rng = np.random.default_rng(11)
    kinds = KINDS + (["inverse"] if variant.endswith("balanced") else [])
    cases = [(VARIANTS[variant], kb, *make(k, rng, kb, cplx)) for k in kinds for kb in (1, 5, 31, 32)]
    for (_, kb, A, B), C, k in zip(cases, driver(cases), np.repeat(kinds, 4)):
        # one real product per output component: complex tiles as real ones of twice the inner length
        if cplx:
            parts = [(C.real, np.hstack([A.real, -A.imag]), np.vstack([B.real, B.imag])),
                     (C.imag, np.hstack([A.real, A.imag]), np.vstack([B.imag, B.real]))]
        else:
            parts = [(C, A, B)]
        for c, a, b in parts:
            err = errors(c, a, b)
            with np.errstate(over="ignore"):
                s = np.abs(a) @ np.abs(b)
                top = np.abs(a).max(1)[:, None] * np.abs(b).max(0)[None, :]
            n = a.shape[1]
            bound = n * 2.0 ** -53 * s + np.where(s > 2.0 ** -20 * top, 0, 2.0 ** -74 * top) + 2.0 ** -1073
            assert np.all(err <= bound), (k, kb, float(np.max(err / np.maximum(bound, 1e-320))))


@pytest.mark.parametrize("cplx", [False, True], ids=["real", "complex"])
@pytest.mark.parametrize("variant", list(VARIANTS))
def test_values_that_are_not_finite(driver, variant, cplx):
    """An infinity or a NaN reaches the outputs it multiplies and no others."""
    rng = np.random.default_rng(3)
    for bad in (np.inf, -np.inf, np.nan):
        A, B = make("normal", rng, NB, cplx)
        A[7, 4] = bad
        B[6, 9] = bad
        C, = driver([(VARIANTS[variant], NB, A, B)])
        hit = np.zeros((NB, NB), dtype=bool)
        hit[7], hit[:, 9] = True, True
        assert np.array_equal(~np.isfinite(C), hit)
