"""Pairs without relative velocity.  A zero vector in block fixed point is zero, so x.v of such a
pair is exactly 0: the viscosity switch is off, in the step and in its reverse, and the work term
of the energy equation vanishes exactly."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
import sph_inputs
from oracle import adjoint as adj

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2005_02656_gb300", "csrc")

WRAP = """
#include "sph_fixed.cuh"
using namespace sph::fx;
extern "C" long fix60(double v, int eb) { return fixed<60>(v, eb); }
extern "C" long fix61(double v, int eb) { return fixed<61>(v, eb); }
extern "C" long dots(const double* a, const double* b) {
  int e[2] = {1, 1};
  const double* v[2] = {a, b};
  Vec3 V[2];
  for (int i = 0; i < 2; ++i) {
    for (int k = 0; k < 3; ++k) if (exp_above(v[i][k]) > e[i]) e[i] = exp_above(v[i][k]);
    for (int k = 0; k < 3; ++k) put(V[i], k, fixed<61>(v[i][k], e[i]));
  }
  return dot(V[0], V[1]);
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "fx.so"), str(d / "fx.cpp")], check=True)
    f = C.CDLL(str(d / "fx.so"))
    for n in ("fix60", "fix61"):
        getattr(f, n).restype = C.c_long
        getattr(f, n).argtypes = [C.c_double, C.c_int]
    f.dots.restype = C.c_long
    f.dots.argtypes = [C.c_void_p, C.c_void_p]
    return f


def test_zero_and_subnormals_have_no_fixed_point_value(fx):
    for eb in range(1, 2049):
        for v in (0.0, -0.0, 5e-324, -5e-324, 2.2250738585072009e-308):
            assert fx.fix60(v, eb) == 0 and fx.fix61(v, eb) == 0, (v, eb)


def test_small_values_are_truncated_exactly(fx):
    """v 2^(61 - (eb - 1023)), truncated toward zero, down to the smallest normal numbers."""
    from fractions import Fraction
    rng = np.random.default_rng(4)
    for f in (1, 2, 5, 40, 61, 62, 63, 64, 90, 1000, 2000):
        for up in (1, 2, 30, 61, 62, 63, 70):
            v = np.ldexp(rng.uniform(1.0, 2.0), f - 1023) * rng.choice([-1.0, 1.0])
            eb = f + up
            x = Fraction(float(v)) * Fraction(2) ** (61 - (eb - 1023))
            assert fx.fix61(float(v), eb) == int(x), (f, up)


def test_product_with_a_zero_vector_is_zero(fx):
    rng = np.random.default_rng(5)
    zeros = [np.zeros(3), -np.zeros(3), np.array([5e-324, 0.0, -1e-310])]
    for z in zeros:
        for _ in range(50):
            d = rng.normal(size=3) * 2.0 ** rng.uniform(-300, 300)
            for a, b in ((z, d), (d, z)):
                assert fx.dots(a.ctypes.data, b.ctypes.data) == 0


def _state(kind):
    s = sph_inputs.jittered_box(10, seed_index=78, vel_sigma=0.0)
    if kind == "uniform":
        for k, v in (("vx", 0.3), ("vy", -0.7), ("vz", 0.1)):
            s[k][:] = v
            s[k + "h"][:] = v
    return s


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["rest", "uniform"])
@pytest.mark.parametrize("steps", [1, 4])
def test_gradient_without_relative_velocity(kind, steps):
    """Against the reference adjoint, per field at the existing bound (1e-6 of its largest)."""
    from paper_2005_02656_gb300 import Params, Rollout
    import torch
    s = _state(kind)
    box, prm = oracle.Box(s["lo"], s["hi"], s["periodic"]), oracle.Params()
    ref = adj.reference_gradients(box, s, prm, adj.record(box, s, prm, steps))
    ro = Rollout(s["x"].shape[0], steps, steps, Params(box_lo=s["lo"], box_hi=s["hi"],
                                                       periodic=s["periodic"]))
    st = {k: torch.as_tensor(s[k], dtype=torch.float64, device=ro.device)
          for k in ("x", "y", "z", "vx", "vy", "vz", "vxh", "vyh", "vzh", "h", "m", "u", "du_prev")}
    fin = ro.forward(st, 1.0)
    g = torch.zeros_like(fin)
    g[3:6] = st["m"][None, :] * fin[3:6]
    g[7] = 2.0 * (fin[7] - 1.0)
    gi, ga = ro.backward(g)
    gi, ga = gi.cpu().numpy(), float(ga.cpu())
    ro.close()
    got = {"x": gi[0:3].T, "v": (gi[3:6] + gi[6:9]).T, "u": gi[9]}
    for k, v in got.items():
        assert np.abs(v - ref[k]).max() <= 1e-6 * np.abs(ref[k]).max(), k
    assert abs(ga - ref["alpha"]) <= 1e-6 * max(abs(ref["alpha"]), np.abs(got["u"]).max())


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["rest", "uniform"])
@pytest.mark.parametrize("precision", ["fp64", "fp32_mixed"])
def test_no_work_without_relative_velocity(kind, precision):
    from paper_2005_02656_gb300 import SphSim
    sim = SphSim(_state(kind), precision=precision, ng_target=0)
    sim.find_neighbors()
    sim.density()
    sim.iad()
    sim.momentum_energy()
    got = sim.to_numpy()
    assert sim.error_word() == 0
    sim.close()
    assert np.all(got["du"] == 0.0)
    assert np.abs(got["ax"]).max() > 0.0
