"""Values that are not finite in the FP64 kernels' block fixed point: they have no fixed-point
form, so the products they enter have to come out not finite by other means."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import sph_inputs

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2005_02656_gb300", "csrc")

WRAP = """
#include "sph_fixed.cuh"
using namespace sph::fx;
extern "C" int not_finite() { return kNotFinite; }
extern "C" long fix(double v, int eb) { return fixed<61>(v, eb); }
extern "C" double any(long x, int k) { return scaled<true>(x, k); }
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "fx.so"), str(d / "fx.cpp")], check=True)
    f = C.CDLL(str(d / "fx.so"))
    f.fix.restype, f.fix.argtypes = C.c_long, [C.c_double, C.c_int]
    f.any.restype, f.any.argtypes = C.c_double, [C.c_long, C.c_int]
    return f


def test_products_with_a_vector_that_is_not_finite(fx):
    """k of a product is the sum of up to three powers of two less 1023 each and at most 59; one of
    them kNotFinite makes every value NaN, the others at 1 or 2047; finite ones never give NaN."""
    nf = fx.not_finite()
    for v in (0.0, 1.0, -3e300, np.inf, -np.inf, np.nan):
        assert fx.fix(v, nf) == 0, v
    for others in ((1, 1), (1, 2047), (2047, 2047), (1023, 1023), (nf, 1), (nf, nf)):
        for low in (60, 59, 0):
            k = nf + sum(others) - 3 * 1023 - low
            for x in (0, 1, -1, (1 << 62) - 1, -(1 << 61)):
                assert np.isnan(fx.any(x, k)), (others, x)
    for e in ((1, 1, 1), (2047, 2047, 2047), (2047, 1, 1023)):
        for x in (0, 1, -1, (1 << 62) - 1):
            assert not np.isnan(fx.any(x, sum(e) - 3 * 1023 + 1)), (e, x)


def _rollout_gradient(s, g_of):
    import torch

    from paper_2005_02656_gb300 import Params, Rollout
    ro = Rollout(s["x"].shape[0], 1, 1, Params(box_lo=s["lo"], box_hi=s["hi"],
                                               periodic=s["periodic"], ng_target=0))
    st = {k: torch.as_tensor(s[k], dtype=torch.float64, device=ro.device)
          for k in ("x", "y", "z", "vx", "vy", "vz", "vxh", "vyh", "vzh", "h", "m", "u", "du_prev")}
    fin = ro.forward(st, 1.0)
    g = torch.zeros_like(fin)
    g[3:6] = st["m"][None, :] * fin[3:6]
    g[7] = 2.0 * (fin[7] - 1.0)
    g_of(g)
    gi, _ = ro.backward(g)
    gi = gi.cpu().numpy()
    ro.close()
    return gi


@pytest.mark.gpu
@pytest.mark.parametrize("row", [0, 1, 2, 3, 4, 5, 6])       # seeds of x y z vx vy vz u
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_seed_that_is_not_finite_reaches_every_adjoint_it_enters(row, value):
    """g = dL/d(acc) (rows 0 to 5) or e = dL/d(du) (row 6) of particle j enters every pair of j:
    the position adjoints of j and of its neighbours are not finite in any component, their energy
    adjoints neither (e meets P_b of approaching neighbours only: j alone), nor the velocity adjoint
    of j (it has approaching neighbours).  Particles out of the step's reach (three
    sums of 2 h: density, IAD, momentum) keep the bits of the finite seed."""
    s = sph_inputs.jittered_box(20, seed_index=79, vel_sigma=0.05, shuffle=False)
    j = 4210
    want = _rollout_gradient(s, lambda g: None)
    got = _rollout_gradient(s, lambda g: g[row].__setitem__(j, value))
    d = np.stack([s[k] - s[k][j] for k in "xyz"], 1)
    d -= np.round(d)
    r = np.sqrt((d * d).sum(1))
    near = r < 2.0 * s["h"]
    far = r > 7.0 * s["h"].max()
    assert near.sum() > 50 and far.sum() > 100
    for k in (0, 1, 2) if row == 6 else (0, 1, 2, 9):
        assert not np.isfinite(got[k][near]).any(), k
    for k in (3, 4, 5, 9):
        assert not np.isfinite(got[k][j]), k
    np.testing.assert_array_equal(got[:, far], want[:, far])


def _sphere(speed):
    """A sphere in homologous flow v = speed * x: every pair recedes (speed > 0) or approaches."""
    s = sph_inputs.uniform_sphere(14, seed_index=80)
    for k in "xyz":
        s["v" + k] = speed * s[k]
        s["v" + k + "h"] = s["v" + k].copy()
    return s


def _both(s, **opts):
    from helpers import oracle_outputs
    from paper_2005_02656_gb300 import SphSim
    with np.errstate(all="ignore"):
        _, _, ref = oracle_outputs(s, ng_target=0, max_nb=400)
    sim = SphSim(s, ng_target=0, max_nb=400, **opts)
    sim.find_neighbors()
    sim.density()
    sim.iad()
    sim.momentum_energy()
    got, flags = sim.to_numpy(), sim.error_word()
    sim.close()
    return got, ref, flags


@pytest.mark.gpu
@pytest.mark.parametrize("speed", [1e200, 1e240, 1e280, 1e295])
def test_receding_pairs_near_the_end_of_the_range(speed):
    """Receding pairs have no viscosity: du = sum m W X v.C d stays in range and within the FP64
    parity bound (1e-12 of the sum of magnitudes, which is linear in the speed without
    viscosity), up to where v.C d itself ends."""
    from helpers import oracle_outputs
    got, ref, _ = _both(_sphere(speed))
    _, _, unit = oracle_outputs(_sphere(1.0), ng_target=0, max_nb=400, alpha=0.0)
    assert np.isfinite(ref["du"]).all() and np.isfinite(got["du"]).all()
    assert (np.abs(got["du"] - ref["du"]) <= 1e-12 * speed * unit["sdu"]).all()
    a = np.stack([got[k] - ref[k] for k in ("ax", "ay", "az")], 1)
    assert (np.abs(a).max(1) <= 1e-12 * ref["sa"]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("speed", [-1e200, -1e240, -1e280, -1e295])
def test_approaching_pairs_past_the_range_overflow(speed):
    """w^2 of Eq. 5 overflows: not finite and flagged, as in FP64."""
    from paper_2005_02656_gb300 import _lib
    got, ref, flags = _both(_sphere(speed))
    assert flags & _lib.FLAG_NONFINITE
    for k in ("ax", "ay", "az", "du"):
        np.testing.assert_array_equal(np.isfinite(got[k]), np.isfinite(ref[k]))
        assert not np.isfinite(got[k]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf, 1e300])
@pytest.mark.parametrize("opts", [{}, {"kernel_mode": "table"}])
def test_one_velocity_that_is_not_finite(value, opts):
    """Not finite where the plain sums are not, and the parity bound everywhere else."""
    from paper_2005_02656_gb300 import _lib
    s = sph_inputs.jittered_box(12, seed_index=81, vel_sigma=0.05)
    s["vy"][17] = value
    got, ref, flags = _both(s, **opts)
    assert flags & _lib.FLAG_NONFINITE
    for k in ("ax", "ay", "az", "du"):
        fin = np.isfinite(ref[k])
        np.testing.assert_array_equal(np.isfinite(got[k]), fin, err_msg=k)
        assert fin.sum() > 0.5 * fin.size, k
        scale = ref["sdu"] if k == "du" else ref["sa"]
        if not opts:                     # (the oracle has the exact kernel here)
            ok = fin & np.isfinite(scale)
            assert (np.abs(got[k][ok] - ref[k][ok]) <= 1e-12 * scale[ok]).all(), k
