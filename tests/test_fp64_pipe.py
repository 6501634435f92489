"""The FP64 kernels' work outside the FP64 pipe: the fixed-point kernel series
(sph_fixed.cuh, compiled for the CPU), and the FP64 pair sums and gravity walk at
the particle counts where their lane split changes."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
import sph_inputs
from helpers import field_errors, oracle_outputs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2005_02656_gb300", "csrc")

WRAP = """
#include "sph_fixed.cuh"
extern "C" void eval(const double* t, double* s, double* s6, double* d, long n) {
  for (long i = 0; i < n; ++i) {
    s[i] = sph::fx::S(t[i]);
    double w;
    sph::fx::S6_d(t[i], w, d[i]);
    s6[i] = sph::fx::S6(t[i]);
    if (w != s6[i]) s6[i] = -1.0;
  }
}
extern "C" void dots(const double* a, const double* b, double* out, long n) {
  using namespace sph::fx;
  for (long i = 0; i < n; ++i, a += 3, b += 3) {
    int ea = 1, eb = 1;
    for (int k = 0; k < 3; ++k) {
      if (exp_above(a[k]) > ea) ea = exp_above(a[k]);
      if (exp_above(b[k]) > eb) eb = exp_above(b[k]);
    }
    Vec3 A, B;
    for (int k = 0; k < 3; ++k) {
      put(A, k, fixed<60>(a[k], ea));
      put(B, k, fixed<61>(b[k], eb));
    }
    out[i] = scaled(dot(A, B), ea + eb - 2 * 1023 - 59);
  }
}
"""


@pytest.fixture(scope="module")
def fixed(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    src, lib = d / "fx.cpp", d / "fx.so"
    src.write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(lib),
                    str(src)], check=True)
    f = C.CDLL(str(lib))

    def run(t, b=None):
        if b is not None:
            out = np.empty(len(t))
            f.dots(*[v.ctypes.data_as(C.c_void_p) for v in (t, b, out)], C.c_long(len(t)))
            return out
        t = np.ascontiguousarray(t, dtype=np.float64)
        out = [np.empty_like(t) for _ in range(3)]
        f.eval(*[a.ctypes.data_as(C.c_void_p) for a in (t, *out)], C.c_long(t.size))
        return out
    return run


def _series(t, k0):
    """sum_{k >= k0} of the Maclaurin series of sin(x)/x (k0 = 0) or of its t-derivative
    (k0 = 1) at x^2 = (pi/2)^2 t, by mpmath."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    S = [mp.sin(mp.pi / 2 * mp.sqrt(v)) / (mp.pi / 2 * mp.sqrt(v)) if v else mp.mpf(1)
         for v in map(mp.mpf, t)]
    if k0 == 0:
        return S
    return [(mp.cos(mp.pi / 2 * mp.sqrt(v)) - s) / (2 * v) if v > 1e-8 else -mp.pi ** 2 / 24
            for v, s in zip(map(mp.mpf, t), S)]


def test_fixed_point_series(fixed):
    """|S error| <= 2^-60 (14 truncated products of at most 3 units of 2^-64 each, a factor of
    at most 2 between the formats, y < 1) plus the rounding of the double; S^6 and its
    derivative likewise, relative to S^5."""
    rng = np.random.default_rng(1)
    t = np.concatenate([rng.uniform(0, 4, 400), 4 - 2.0 ** -rng.uniform(0, 51, 200),
                        2.0 ** -rng.uniform(0, 80, 200)])
    s, s6, d = fixed(t)
    S, dS = _series(t, 0), _series(t, 1)
    for i in range(t.size):
        e = 2.0 ** -60
        assert abs(s[i] - S[i]) <= e + 2.0 ** -53 * S[i], t[i]
        assert abs(s6[i] - S[i] ** 6) <= 6 * (S[i] + e) ** 5 * e + 2.0 ** -52 * S[i] ** 6, t[i]
        ref = 6 * S[i] ** 5 * dS[i]
        if t[i] > 1e-8:
            assert abs(d[i] - ref) <= 40 * (S[i] + e) ** 4 * e + 2.0 ** -51 * abs(ref), t[i]


def test_fixed_point_edges(fixed):
    """The origin, tiny arguments, the support's edge and beyond, infinity and NaN."""
    t = np.array([0.0, 5e-324, 1e-300, 4.0, 4.0 + 1e-15, 1e300, np.inf, np.nan])
    s, s6, d = fixed(t)
    np.testing.assert_array_equal(s, [1, 1, 1, 0, 0, 0, 0, 0])
    np.testing.assert_array_equal(s6, [1, 1, 1, 0, 0, 0, 0, 0])
    np.testing.assert_allclose(d[:3], -np.pi ** 2 / 4, rtol=1e-15)
    np.testing.assert_array_equal(d[3:], 0)
    s, s6, _ = fixed([np.nextafter(4.0, 0.0)])
    assert 0 <= s6[0] <= 1e-90 and 0 <= s[0] < 1e-15


def test_block_fixed_point_dot(fixed):
    """Scalar products of vectors over many scales, with zero, tiny, subnormal and opposite
    components.  Bound, in units of 2^-59 of the powers of two above the largest components:
    3 (low limbs) + 1/2 (rounding) + 6 (two factors truncated by < 1 of 2^60 and 2^61 each, three
    terms), and the rounding of the double."""
    from fractions import Fraction
    rng = np.random.default_rng(2)
    n = 4000
    a, b = (rng.normal(size=(n, 3)) * 2.0 ** rng.uniform(-200, 200, (n, 1)) for _ in range(2))
    a[::7, 1] = 0.0
    a[::11, 2] *= 1e-14
    b[::13, 0] = 5e-324
    b[::17] = np.cross(a[::17], b[::17])
    b[::19] = 0.0
    got = fixed(np.ascontiguousarray(a), np.ascontiguousarray(b))
    for x, y, v in zip(a, b, got):
        exact = sum(Fraction(p) * Fraction(q) for p, q in zip(x, y))
        top = [2.0 ** (np.frexp(np.abs(w).max())[1]) for w in (x, y)]
        bound = 9.5 * Fraction(top[0]) * Fraction(top[1]) / 2 ** 59
        assert abs(Fraction(v) - exact) <= bound + abs(exact) / 2 ** 53, (x, y, v)


# particles per target-lane split: 16 lanes (below 16,384), 8, 4 (from 131,072)
@pytest.mark.gpu
@pytest.mark.parametrize("side,gradh", [(7, 0), (25, 1), (26, 0), (50, 0), (51, 1)])
def test_fp64_lane_splits(side, gradh):
    """FP64 fields against the oracle at both sides of each split (the parity bound 1e-12)."""
    from paper_2005_02656_gb300 import SphSim
    s = sph_inputs.jittered_box(side, seed_index=40 + side)
    rc, _, ref = oracle_outputs(s, ng_target=0, gradh=gradh)
    assert rc == 0
    sim = SphSim(s, gradh=gradh, ng_target=0)
    sim.find_neighbors()
    sim.density()
    sim.iad()
    sim.momentum_energy()
    got = sim.to_numpy()
    assert sim.error_word() == 0
    sim.close()
    e = field_errors(got, ref)
    for k in ("rho", "p", "c", "iad", "a", "du"):
        assert e[k] <= 1e-12, (k, e)


@pytest.mark.gpu
@pytest.mark.parametrize("side,scale", [(5, 1.0), (9, 1e-25), (13, 1e25), (31, 1.0), (48, 1.0)])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-12), ("fp32_mixed", 1e-4)])
def test_gravity_scales(side, scale, precision, tol):
    """The walks against the oracle's tree: ragged last tiles, trees built by one block and level
    by level, and coordinates far outside the FP32 range (opening decisions and FP32 terms work
    on scaled coordinates).  Tolerances of max|g|: the FP64 parity bound and the FP32 one."""
    from paper_2005_02656_gb300 import Params, SphSim
    s = sph_inputs.uniform_sphere(side, seed_index=90 + side)
    for k in ("x", "y", "z", "h"):
        s[k] = s[k] * scale
    eps = 1e-3 * scale
    sim = SphSim(s, Params(periodic=(0, 0, 0), precision=precision))
    g, counts = sim.gravity(1.0, eps, 0.5)
    g, ids = g.cpu().numpy(), sim.t["id"].cpu().numpy()
    assert sim.error_word() == 0
    sim.close()
    rc, ref, st = oracle.gravity_tree(s, eps=eps, theta=0.5)
    assert rc == 0
    ref = ref[np.argsort(s["id"])]
    assert np.abs(g[np.argsort(ids)] - ref).max() <= tol * np.abs(ref).max()
    np.testing.assert_array_equal(counts, st)
