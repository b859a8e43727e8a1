"""Rounding error of the class product (csrc/classes.cuh, k_class_apply) on given
blocks, against 64-bit sums, beside that of 16 interleaved FP32 chains (the order
of the streaming smoother, which the class product stands in for).

Both are random walks of FP32 roundings over the same products.  Chains of eight
joined in pairs and added chunk by chunk have 0.95 to 1.05 times the mean square
root error of 16 chains for 54 to 800 terms, one chain over all terms 1.8 to 3.5
times; 1.25 leaves room for the scatter of the sample.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_01728_gb300", "csrc")

DRIVER = r"""
#include <cstdio>
#include <cstring>
#include <vector>
#include "classes.cuh"
using namespace dpgmg;
namespace dpgmg { void count_launch() {} }

template <class T> static std::vector<T> rd(FILE* f, size_t n) {
  std::vector<T> v(n);
  if (fread(v.data(), sizeof(T), n, f) != n) exit(2);
  return v;
}
template <class T> static T* up(const std::vector<T>& v) {
  T* d;
  cudaMalloc(&d, v.size() * sizeof(T) + 256);
  cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return d;
}

// header: members M, block size n, vector length N, offU, real (0, 1), shape;
// then the members' DOFs (M x n), the block (n rows of the stored length), the vector
int main(int argc, char** argv) {
  FILE* in = fopen(argv[1], "rb");
  FILE* out = fopen(argv[2], "wb");
  int h[6];
  const int outs[5] = {64, 64, 64, 32, 32}, mems[5] = {32, 16, 8, 32, 16};
  while (fread(h, 4, 6, in) == 6) {
    const int M = h[0], n = h[1], N = h[2], real = h[4], shape = h[5];
    const auto dofs = rd<int32_t>(in, (size_t)M * n);
    const auto w = rd<float>(in, (size_t)n * (real ? patch_ldr(n) : 2 * patch_ld(n)));
    const auto r = rd<float2>(in, N);
    std::vector<int64_t> ptr, vptr(M, 0);
    std::vector<int32_t> mem;
    std::vector<uint8_t> rf(M, (uint8_t)real);
    for (int m = 0; m <= M; ++m) ptr.push_back((int64_t)m * n);
    for (int m = 0; m < M; ++m) mem.push_back(m);
    std::vector<int4> items;
    for (int a = 0; a < n; a += outs[shape])
      for (int q = 0; q < M; q += mems[shape]) items.push_back(make_int4(q, std::min(mems[shape], M - q), a, shape));
    float2* p;
    cudaMalloc(&p, (size_t)M * n * sizeof(float2));
    cudaMemset(p, 0xff, (size_t)M * n * sizeof(float2));
    k_class_apply<float2><<<dim3((unsigned)items.size(), 1), CLS_THREADS>>>(
        up(ptr), up(dofs), up(vptr), up(items), up(mem), reinterpret_cast<const float2*>(up(w)), up(r), 0, p, 0, up(rf),
        (int64_t)h[3]);
    std::vector<float2> y((size_t)M * n);
    if (cudaMemcpy(y.data(), p, y.size() * sizeof(float2), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    fwrite(y.data(), sizeof(float2), y.size(), out);
  }
  fclose(out);
  return 0;
}
"""

SHAPES = {"64x32": (64, 32), "64x16": (64, 16), "64x8": (64, 8), "32x32": (32, 32), "32x16": (32, 16)}


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("classes")
    (d / "driver.cu").write_text(DRIVER)
    subprocess.run([nvcc, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(d / "driver.cu"), "-o", str(d / "driver")],
                   check=True)

    def run(dofs, block, r, off_u, shape):
        real = not np.iscomplexobj(block)
        M, n = dofs.shape
        ld = (n + 3) // 4 * 4 if real else (n + 1) // 2 * 2
        W = np.zeros((n, ld), dtype=np.float32 if real else np.complex64)
        W[:, :n] = block
        with open(d / "in", "wb") as f:
            f.write(np.array([M, n, len(r), off_u, real, shape], dtype=np.int32).tobytes())
            f.write(dofs.astype(np.int32).tobytes() + W.tobytes() + r.astype(np.complex64).tobytes())
        subprocess.run([str(d / "driver"), str(d / "in"), str(d / "out")], check=True)
        return np.fromfile(d / "out", dtype=np.complex64).reshape(M, n)
    return run


def chains(W, g, count):
    """FP32: `count` interleaved FMA chains over the rows of W, added in order.  [members, outputs]"""
    f = np.float32
    parts = []
    for i in range(count):
        s = np.zeros((g.shape[0], W.shape[1]), f)
        for k in range(i, W.shape[0], count):
            s = (W[k].astype(np.float64)[None, :] * g[:, k].astype(np.float64)[:, None] + s).astype(f)
        parts.append(s)
    t = parts[0]
    for p in parts[1:]:
        t = (t + p).astype(f)
    return t


@pytest.mark.parametrize("shape", list(SHAPES))
@pytest.mark.parametrize("n", [5, 16, 17, 54, 110, 155, 302, 488])
@pytest.mark.parametrize("real", [True, False], ids=["real", "complex"])
def test_error_against_16_chains(driver, shape, n, real):
    rng = np.random.default_rng(n)
    M, N = SHAPES[shape][1] + 3, 2000           # a full item and a ragged one
    off_u = N // 2
    below = rng.random(n) < 0.5                 # members of a class have the same kinds of DOFs place by place
    dofs = np.array([np.where(below, rng.permutation(off_u)[:n], off_u + rng.permutation(off_u)[:n]) for _ in range(M)])
    W = rng.standard_normal((n, n)).astype(np.float32)
    r = (rng.standard_normal(N) + 1j * rng.standard_normal(N)).astype(np.complex64)
    if not real:
        W = (W + 1j * rng.standard_normal((n, n)).astype(np.float32)).astype(np.complex64)
    y = driver(dofs, W, r, off_u, list(SHAPES).index(shape)).astype(np.complex128)
    g = r[dofs].astype(np.complex128)
    if real:   # y_a = i^(s_a) sum_k W_ka i^(-s_k) r_k, s = 1 below offU
        s = (dofs < off_u).astype(int)
        g = g * (-1j) ** s
        want = (g @ W.astype(np.float64)) * 1j ** s
        y, want = y * (-1j) ** s, want * (-1j) ** s
        ref = chains(W, np.ascontiguousarray(g.real).astype(np.float32), 16)
        e16 = np.sqrt(np.mean((ref - want.real) ** 2))
        err = np.sqrt(np.mean((y.real - want.real) ** 2)), np.sqrt(np.mean((y.imag - want.imag) ** 2))
    else:      # y_a = sum_k conj(W_ka) r_k: real part of 2 n products
        want = g @ np.conj(W).astype(np.complex128)
        W2 = np.empty((2 * n, n), np.float32)
        W2[0::2], W2[1::2] = W.real, W.imag
        g2 = np.empty((M, 2 * n), np.float32)
        g2[:, 0::2], g2[:, 1::2] = g.real, g.imag
        e16 = np.sqrt(np.mean((chains(W2, g2, 16) - want.real) ** 2))
        err = np.sqrt(np.mean((y.real - want.real) ** 2)), np.sqrt(np.mean((y.imag - want.imag) ** 2))
    if n >= 54:
        assert max(err) < 1.25 * e16, max(err) / e16
    else:        # too few terms to tell the orders apart: n roundings of at most sum |w| |r|
        assert max(err) < 2 * n * 2.0 ** -24 * np.sqrt(np.mean((np.abs(g) @ np.abs(W)) ** 2))
