"""The node stack of the FP32-mixed gravity walk: how many nodes a turn takes, and that no order of
opening, accepting and deciding nodes one by one overruns it."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2005_02656_gb300", "csrc")

WRAP = """
#include <random>
#include <vector>
#include "sph_walk.cuh"
using namespace sph::grav;
extern "C" int stack() { return kStack32; }
extern "C" int take(int sp) { return walk_take(sp); }
extern "C" int on(int sp) { return walk_on(sp); }
// A walk over a tree of kLevels levels below the root: per popped node, opened by all its targets
// with probability open (children pushed in pop order), decided one by one with probability mix
// (children pushed after those), accepted otherwise.  Returns the deepest stack.
extern "C" int walk(double open, double mix, int children, unsigned seed, long turns) {
  std::mt19937 rng(seed);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  std::vector<int> st(1, 0);
  int deepest = 1;
  for (long t = 0; t < turns && walk_on((int)st.size()); ++t) {
    const int n = walk_take((int)st.size());
    std::vector<int> first, later;
    for (int i = 0; i < n; ++i) {
      const int l = st.back();
      st.pop_back();
      const double r = u(rng);
      if (l == kLevels || r >= open + mix) continue;
      auto& v = r < open ? first : later;
      for (int c = 0; c < children; ++c) v.push_back(l + 1);
    }
    st.insert(st.end(), first.begin(), first.end());
    st.insert(st.end(), later.begin(), later.end());
    if ((int)st.size() > deepest) deepest = (int)st.size();
  }
  return walk_on((int)st.size()) || st.empty() ? deepest : kStack32 + 1;
}
"""


@pytest.fixture(scope="module")
def w(tmp_path_factory):
    d = tmp_path_factory.mktemp("walk")
    (d / "w.cpp").write_text(WRAP)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "w.so"), str(d / "w.cpp")], check=True)
    f = C.CDLL(str(d / "w.so"))
    f.walk.argtypes = [C.c_double, C.c_double, C.c_int, C.c_uint, C.c_long]
    return f


def test_take_leaves_room(w):
    """A turn takes at least one node, never more than the stack holds or a warp has lanes, and more
    than one only where all their children leave a depth-first walk its room."""
    for sp in range(1, w.stack() + 1):
        t = w.take(sp)
        assert 1 <= t <= min(sp, 32)
        if t > 1:
            assert sp + 7 * t <= w.stack() - 64
        if w.on(sp):
            assert sp - t + 8 * t <= w.stack()
    assert not w.on(0) and w.on(1) and w.on(w.stack() - 7)
    assert not any(w.on(sp) for sp in range(w.stack() - 6, w.stack() + 1))


@pytest.mark.parametrize("open_,mix", [(1.0, 0.0), (0.0, 1.0), (0.5, 0.5), (0.6, 0.2), (0.2, 0.1)])
def test_no_walk_overruns_the_stack(w, open_, mix):
    turns = 4_000_000 if open_ == 1.0 else 300_000     # the full tree: every node opened
    for seed in range(1 if open_ == 1.0 else 4):
        assert w.walk(open_, mix, 8, seed, turns) <= w.stack()
    assert w.walk(1.0, 0.0, 8, 0, turns) > 300         # (the room is used)


def test_the_walk_is_guarded():
    """The kernel's loop asks walk_on, and a walk that ends with nodes left raises a flag."""
    with open(os.path.join(CSRC, "sph_gravity.cu")) as f:
        s = f.read()
    k = s[s.index("k_walk32("):s.index("inline int blocks_for")]
    assert "while (walk_on(sp))" in k and "walk_take(sp)" in k
    assert "if (sp > 0 && lane == 0) raise_flag(err, SPH_FLAG_CELL_OVERFLOW)" in k
