"""Stage calls on a state without particles: accepted, and nothing is launched that could read
another search's counters."""
import numpy as np
import pytest

import sph_inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{"precision": "fp64"}, {"precision": "fp32_mixed"},
                                  {"precision": "fp32_mixed", "pair_mode": "lists"}])
@pytest.mark.parametrize("first", [0, 1])
def test_empty_stage_calls(opts, first):
    """On a new context, and on one whose last search had 512 particles."""
    from paper_2005_02656_gb300 import SphSim
    s = sph_inputs.jittered_box(8, seed_index=82)
    sim = SphSim(s, ng_target=0, **opts)
    if first:
        for f in (sim.find_neighbors, sim.density, sim.iad, sim.momentum_energy):
            f()
    rho = sim.t["rho"].clone()
    before = sim.lib.sph_launch_count(sim.ctx)
    sim.n = sim._st.n = 0
    for f in (sim.find_neighbors, sim.density, sim.iad, sim.momentum_energy):
        f()
    assert sim.lib.sph_launch_count(sim.ctx) == before
    assert sim.error_word() == 0
    assert bool((sim.t["rho"] == rho).all())
    # the full state again
    sim.n = sim._st.n = s["x"].shape[0]
    for f in (sim.find_neighbors, sim.density, sim.iad, sim.momentum_energy):
        f()
    assert np.isfinite(sim.to_numpy()["ax"]).all() and sim.error_word() == 0
    sim.close()
