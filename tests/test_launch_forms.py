"""The launch forms that the particle count picks: the staged search by one CTA or one warp per
cell, and the pair passes' pipelined and general forms in one launch, on both sides of the
search's line (64 particles per SM) with cells of every class: pipelined (few candidates), 449 to
832, more than 832, several windows, and list form."""
import numpy as np
import pytest

import sph_inputs
from helpers import field_errors, oracle_outputs

pytestmark = pytest.mark.gpu

TOL = {"rho": 1e-5, "iad": 1e-5, "a": 1e-4, "du": 1e-4}   # the FP32-mixed parity bounds


def _state(side, big):
    s = sph_inputs.jittered_box(side, seed_index=60 + side)
    if big:                       # two particles' h make every cell large
        s["h"][[5, 1234]] *= big
    return s


@pytest.mark.parametrize("side", [21, 22])            # 9,261 and 10,648 particles
@pytest.mark.parametrize("big", [0, 1.25, 1.8, 2.6])
def test_search_and_pass_forms(side, big):
    from paper_2005_02656_gb300 import SphSim
    s = _state(side, big)
    mb = 2048 if big else 160
    rc, _, ref = oracle_outputs(s, ng_target=0, max_nb=mb)
    assert rc == 0
    sim = SphSim(s, precision="fp32_mixed", max_nb=mb, ng_target=0)
    sim.find_neighbors()
    sim.density()
    sim.iad()
    sim.momentum_energy()
    counts, ids = sim.get_neighbors()
    got = sim.to_numpy(by_id=False)
    assert sim.error_word() == 0
    sim.close()
    order = np.argsort(got["id"], kind="stable")
    got = {k: v[order] for k, v in got.items()}
    counts, ids = counts.cpu().numpy()[order], ids.cpu().numpy()[order]
    np.testing.assert_array_equal(counts, ref["nn"])
    for a in range(counts.shape[0]):
        np.testing.assert_array_equal(ids[a, :counts[a]], ref["nbr"][a, :counts[a]])
    e = field_errors(got, ref)
    for k, tol in TOL.items():
        assert e[k] <= tol, (k, e)


@pytest.mark.parametrize("side,big", [(7, 0), (13, 0), (13, 1.8), (19, 2.6), (28, 0), (29, 0)])
def test_list_search_by_shared_and_single_warps(side, big):
    """The list search with several warps per cell (up to 160 particles per SM: 24,320) and
    one: periodic axes of two cells, cells of more than 32 and more than 64 targets, several
    windows, and both sides of the line.  Whole neighbour sets, and the FP64 density."""
    from paper_2005_02656_gb300 import SphSim
    s = _state(side, 0)
    if big:
        s["h"][[5, 1234]] *= big
    mb = 2048 if big else 160
    rc, _, ref = oracle_outputs(s, ng_target=0, max_nb=mb)
    assert rc == 0
    sim = SphSim(s, precision="fp64", max_nb=mb, ng_target=0)
    sim.find_neighbors()
    sim.density()
    counts, ids = sim.get_neighbors()
    got = sim.to_numpy(by_id=False)
    assert sim.error_word() == 0
    sim.close()
    order = np.argsort(got["id"], kind="stable")
    counts, ids = counts.cpu().numpy()[order], ids.cpu().numpy()[order]
    np.testing.assert_array_equal(counts, ref["nn"])
    for a in range(counts.shape[0]):
        np.testing.assert_array_equal(ids[a, :counts[a]], ref["nbr"][a, :counts[a]])
    np.testing.assert_allclose(got["rho"][order], ref["rho"], rtol=1e-12)
