"""The reciprocal square roots of the FP64 kernels on the GPU, with the seed of its FP32 unit
(inv_root and root_parts of sph_device.cuh, over_root of sph_fixed.cuh), and the gravity tree built
level by level, which only trees of more than 4,096 leaves take."""
import ctypes as C
import os
import shutil
import subprocess
from decimal import Decimal, getcontext

import numpy as np
import pytest

import oracle
import sph_inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_02656_gb300", "csrc")

WRAP = """
#include "sph_device.cuh"
#include "sph_fixed.cuh"
__global__ void k_roots(const double* x, const long long* v, const int* kv,
                        const unsigned long long* R, const int* kr, double* a, double* b, double* c,
                        int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double y0, q;
  sph::root_parts(x[i], y0, q);
  a[i] = sph::inv_root(x[i]);
  b[i] = fma(y0, q, y0);
  c[i] = sph::fx::over_root(v[i], kv[i], R[i], kr[i]);
}
extern "C" int roots(const double* x, const long long* v, const int* kv, const unsigned long long* R,
                     const int* kr, double* out, int n) {
  char* d = nullptr;
  const size_t N = n;
  if (cudaMalloc((void**)&d, 56 * N) != cudaSuccess) return 1;
  double *dx = (double*)d, *o = dx + N;
  long long* dv = (long long*)(o + 3 * N);
  unsigned long long* dR = (unsigned long long*)(dv + N);
  int *dkv = (int*)(dR + N), *dkr = dkv + N;
  cudaMemcpy(dx, x, 8 * N, cudaMemcpyHostToDevice);
  cudaMemcpy(dv, v, 8 * N, cudaMemcpyHostToDevice);
  cudaMemcpy(dR, R, 8 * N, cudaMemcpyHostToDevice);
  cudaMemcpy(dkv, kv, 4 * N, cudaMemcpyHostToDevice);
  cudaMemcpy(dkr, kr, 4 * N, cudaMemcpyHostToDevice);
  k_roots<<<(n + 127) / 128, 128>>>(dx, dv, dkv, dR, dkr, o, o + N, o + 2 * N, n);
  cudaMemcpy(out, o, 24 * N, cudaMemcpyDeviceToHost);
  const cudaError_t e = cudaDeviceSynchronize();
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
"""


@pytest.fixture(scope="module")
def roots(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    src, lib = d / "roots.cu", d / "roots.so"
    src.write_text(WRAP)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), "-o", str(lib), str(src)], check=True)
    f = C.CDLL(str(lib))

    def run(x, v, kv, R, kr):
        arr = [np.ascontiguousarray(a, dtype=t) for a, t in
               zip((x, v, kv, R, kr), (np.float64, np.int64, np.int32, np.uint64, np.int32))]
        out = np.empty((3, len(x)))
        assert f.roots(*[a.ctypes.data_as(C.c_void_p) for a in arr],
                       out.ctypes.data_as(C.c_void_p), C.c_int(len(x))) == 0
        return out
    return run


def test_reciprocal_square_roots(roots):
    """Bound 2^-52, relative.  inv_root: the seed is within 2^-21 (2 ulp of rsqrtf and the truncated
    mantissa), so the series' first omitted term is below 2^-61; x y0 and the last operation round to
    2^-53 each, the first halved.  over_root: seed as above, products short by 3 of 2^-61 each, the
    last rounding 2^-53.  Outside 2^+-1000 inv_root is rsqrt (2 ulp)."""
    getcontext().prec = 50
    rng = np.random.default_rng(11)
    n = 4000
    x = np.concatenate([2.0 ** rng.uniform(-1000, 1000, n - 1200), rng.uniform(1.0, 4.0, 400),
                        1.0 + 2.0 ** -rng.uniform(1, 52, 400), 4.0 - 2.0 ** -rng.uniform(0, 50, 400)])
    v = rng.integers(-(1 << 61), 1 << 61, n)
    v[::7] = rng.integers(1, 1000, v[::7].size)
    v[v == 0] = 1
    R = rng.integers(1 << 52, 1 << 60, n).astype(np.uint64)
    R[::5] = rng.integers(1 << 52, 1 << 53, R[::5].size).astype(np.uint64)
    kv, kr = rng.integers(-300, 300, n), rng.integers(-300, 300, n)
    a, b, c = roots(x, v, kv, R, kr)
    two = Decimal(2)
    for i in range(n):
        ref = 1 / Decimal(float(x[i])).sqrt()
        assert abs(Decimal(float(a[i])) - ref) <= ref * two ** -52, x[i]
        assert a[i] == b[i]
        ref = Decimal(int(v[i])) * two ** int(kv[i]) / (Decimal(int(R[i])) * two ** int(kr[i])).sqrt()
        assert abs(Decimal(float(c[i])) - ref) <= abs(ref) * two ** -52, (v[i], R[i], kv[i], kr[i])
    ends = np.array([1e-307, 5e-308, 1e305, 1.7e308, np.inf])
    a, _, _ = roots(ends, np.ones(5), np.zeros(5), np.full(5, 1 << 55), np.zeros(5))
    np.testing.assert_allclose(a, 1.0 / np.sqrt(ends), rtol=2.0 ** -51)


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32_mixed", 1e-4)])
def test_gravity_tree_built_level_by_level(precision, tol):
    """More than 4,096 leaves: the lowest levels by a launch each, handed over to the one block that
    builds the rest; field and interaction counts against the oracle's tree."""
    from paper_2005_02656_gb300 import Params, SphSim
    s = sph_inputs.uniform_sphere(60, seed_index=92)
    cs = 2.0 * s["h"].max()
    side = [int((s[k].max() - s[k].min()) / cs) for k in "xyz"]
    cells = [np.minimum(((s[k] - s[k].min()) / (s[k].max() - s[k].min()) * m).astype(int), m - 1)
             for k, m in zip("xyz", side)]
    assert np.unique(np.ravel_multi_index(cells, side)).size > 4500
    sim = SphSim(s, Params(periodic=(0, 0, 0), precision=precision))
    g, counts = sim.gravity(1.0, 1e-3, 0.5)
    g, ids = g.cpu().numpy(), sim.t["id"].cpu().numpy()
    assert sim.error_word() == 0
    sim.close()
    rc, ref, st = oracle.gravity_tree(s, eps=1e-3, theta=0.5)
    assert rc == 0
    ref = ref[np.argsort(s["id"])]
    assert np.abs(g[np.argsort(ids)] - ref).max() <= tol * np.abs(ref).max()
    np.testing.assert_array_equal(counts, st)
