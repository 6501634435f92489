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
extern "C" double edge(long x, int k) { return sph::fx::scaled<true>(x, k); }
// for d (3 per entry), 2 h_a, 1 / h_b^2, v, a: S^6 at t = r^2 / h_b^2, its product with a, v.d / r
// (0 where r is below 1/16 of the power of two above 2 h_a), and (a S^6) d_x
extern "C" void pair(const double* d, const double* h2, const double* hinv2, const double* v,
                     const double* a, double* out, long n) {
  using namespace sph::fx;
  for (long i = 0; i < n; ++i, d += 3, v += 3, out += 4) {
    const int ed = exp_above(h2[i]), kr = 2 * (ed - 1023) - 60;
    int ev = 1;
    for (int k = 0; k < 3; ++k) if (exp_above(v[k]) > ev) ev = exp_above(v[k]);
    Vec3 D, V;
    for (int k = 0; k < 3; ++k) {
      put(D, k, fixed<61>(d[k], ed));
      put(V, k, fixed<61>(v[k], ev));
    }
    const int64_t R = dot(D, D), vd = dot(V, D);
    uint64_t y;
    const bool in = (uint64_t)R >> 60 == 0 && fraction_of((uint64_t)R, kr, hinv2[i], y);
    out[0] = in ? S6_at(y) : 0.0;
    out[1] = in ? S6_at_times(y, a[i]) : 0.0;
    out[2] = R >> 52 && vd ? over_root(vd, ev + ed - 2 * 1023 - 60, (uint64_t)R, kr) : 0.0;
    out[3] = middle(a[i]) && middle(out[0])
                 ? times(mant(a[i]) * mant(out[0]), fixed<61>(d[0], ed), ed - 1023 - 61) : 0.0;
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
        if isinstance(t, tuple):
            out = np.empty((len(t[1]), 4))
            f.pair(*[np.ascontiguousarray(v).ctypes.data_as(C.c_void_p) for v in t],
                   out.ctypes.data_as(C.c_void_p), C.c_long(len(t[1])))
            return out
        t = np.ascontiguousarray(t, dtype=np.float64)
        out = [np.empty_like(t) for _ in range(3)]
        f.eval(*[a.ctypes.data_as(C.c_void_p) for a in (t, *out)], C.c_long(t.size))
        return out
    run.edge = f.edge
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


def test_pair_in_fixed_point(fixed):
    """The pair quantities the FP64 kernels take from block fixed point, against mpmath.  R carries
    an error of at most 3.5 units of 2^-60 of 2^(2 e) (2^e the power of two above 2 h_a) plus the
    truncation of d (6 units of 2^-61 times |d| / 2^e <= 1): 7 units together; y = R K 2^-60 with
    K = 2^(2e) / (4 h_b^2), plus 2^-57.  |dS^6/dy| <= 10."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    rng = np.random.default_rng(3)
    n = 600
    h = 2.0 ** rng.uniform(-30, 30, n)
    hb = h * 2.0 ** rng.uniform(-0.7, 0.7, n)
    hb[::29] = h[::29] * 4.0
    u = rng.normal(size=(n, 3))
    r = 2 * h * rng.uniform(0, 1, n) ** (1 / 3)
    r[::13] *= 1e-3
    d = u / np.linalg.norm(u, axis=1)[:, None] * r[:, None] * (1 - 1e-12)
    v = rng.normal(size=(n, 3)) * 2.0 ** rng.uniform(-40, 40, (n, 1))
    a = 2.0 ** rng.uniform(-90, 90, n)
    hinv2 = 1.0 / (hb * hb)
    out = fixed((d, 2 * h, hinv2, v, a))
    for i in range(n):
        D, V = [mp.mpf(x) for x in d[i]], [mp.mpf(x) for x in v[i]]
        r2 = sum(x * x for x in D)
        t = r2 * mp.mpf(hinv2[i])
        x = mp.pi / 2 * mp.sqrt(t)
        S6 = (mp.sin(x) / x) ** 6 if t < 4 else mp.mpf(0)
        top = 2.0 ** np.frexp(2 * h[i])[1]
        err = 10 * (7 * 2.0 ** -60 * top * top * hinv2[i] / 4 + 2.0 ** -57) + 2.0 ** -52 * S6
        assert abs(out[i, 0] - S6) <= err, i
        assert abs(out[i, 1] - a[i] * S6) <= a[i] * (err + 2.0 ** -52 * S6), i
        if out[i, 2]:
            vd = sum(p * q for p, q in zip(V, D))
            vtop = 2.0 ** np.frexp(np.abs(v[i]).max())[1]
            # v.d to 9.5 units of 2^-60, 1/r to 7 units of 2^-60 of top^2 / r^2 (halved), rounding
            tol = (9.5 * 2.0 ** -60 * vtop * top / mp.sqrt(r2)
                   + abs(vd) / mp.sqrt(r2) * (3.5 * 2.0 ** -60 * top * top / r2 + 2.0 ** -52))
            assert abs(out[i, 2] - vd / mp.sqrt(r2)) <= tol, i
        if out[i, 3]:
            e = mp.mpf(a[i]) * mp.mpf(out[i, 0]) * D[0]
            assert abs(out[i, 3] - e) <= a[i] * out[i, 0] * top * 2.0 ** -60 + 2.0 ** -52 * abs(e), i


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


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [{}, {"sinc_n": 5.0}, {"gradh": 1}, {"kernel_mode": "table"}])
def test_fp64_close_pairs_and_uneven_h(opts):
    """Pairs at 1e-2 to 1e-9 of h (below the range where r is taken from fixed point), smoothing
    lengths over a factor of 4, one axis at rest, and every kernel form, against the oracle."""
    from paper_2005_02656_gb300 import SphSim
    s = sph_inputs.jittered_box(14, seed_index=77)
    rng = np.random.default_rng(8)
    n = s["x"].shape[0]
    s["h"] = s["h"] * np.exp(rng.uniform(-0.7, 0.6, n))
    for k, f in enumerate((1e-2, 1e-4, 1e-6, 1e-9)):
        i, j = 50 + 2 * k, 51 + 2 * k
        for ax, c in zip("xyz", (1.0, -0.5, 0.25)):
            s[ax][j] = s[ax][i] + c * f * s["h"][i]
    s["vz"][:] = 0.0
    kw = {k: (1 if v == "table" else v) for k, v in opts.items()}
    rc, _, ref = oracle_outputs(s, ng_target=0, max_nb=800, **kw)
    assert rc == 0
    sim = SphSim(s, ng_target=0, max_nb=800, **opts)
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


def test_scaled_past_the_range(fixed):
    fixed.edge.restype = C.c_double
    fixed.edge.argtypes = [C.c_long, C.c_int]
    for x in (1, -1, 3, (1 << 62) - 1, -(1 << 61)):
        for k in (-1200, -1023, -80, 0, 900, 962, 1023, 1100, 3000):
            want = np.ldexp(float(x), k) if abs(np.ldexp(float(x), k)) >= 2.0 ** -1022 else 0.0
            assert fixed.edge(x, k) == want, (x, k)
    assert fixed.edge(0, 3000) == 0.0


@pytest.mark.gpu
@pytest.mark.parametrize("side,ng", [(8, 20), (12, 150), (16, 620)])
def test_reverse_lists_of_every_length(side, ng):
    """Reverse lists below, at and past the 128 entries a warp ranks at a time and the 512 it
    keeps in shared memory, by the closed forms of a rollout's gradient: sum_a dL/dx_a = 0 and
    sum_a dL/dv_a = sum_a m_a v_a(K) within the FP64 bound on sums of n terms (1e-10 of the
    terms' sum of magnitudes); and the same bits from a second reverse pass."""
    import torch

    from paper_2005_02656_gb300 import Params, Rollout
    s = sph_inputs.jittered_box(side, seed_index=91, vel_sigma=0.05)
    s["h"][:] = 0.5 / side * (3.0 * ng / (4.0 * np.pi)) ** (1.0 / 3.0)
    ro = Rollout(side ** 3, 2, 1, Params(box_lo=s["lo"], box_hi=s["hi"], periodic=s["periodic"],
                                         max_nb=1024, ng_target=0))
    st = {k: torch.as_tensor(s[k], dtype=torch.float64, device=ro.device)
          for k in ("x", "y", "z", "vx", "vy", "vz", "vxh", "vyh", "vzh", "h", "m", "u", "du_prev")}
    fin = ro.forward(st, 1.0)
    g = torch.zeros_like(fin)
    g[3:6] = st["m"][None, :] * fin[3:6]
    g[7] = 2.0 * (fin[7] - 1.0)
    gi, ga = ro.backward(g)
    again, _ = ro.backward(g)
    assert torch.equal(gi, again)
    ro.close()
    gi = gi.cpu().numpy()
    p = (s["m"][None, :] * fin[3:6].cpu().numpy())
    for k in range(3):
        assert abs(gi[k].sum()) <= 1e-10 * np.abs(gi[k]).sum()
        dv = gi[3 + k] + gi[6 + k]
        assert abs(dv.sum() - p[k].sum()) <= 1e-10 * (np.abs(dv).sum() + np.abs(p[k]).sum())
