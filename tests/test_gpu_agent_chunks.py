"""The agent-based biofilm's ordered list and its statistics over many chunks of nodes, against the FP64
oracle (exact): sizes at the edges of a chunk (2048 nodes) and of the scan over the chunks (1024 of them)."""
import numpy as np
import pytest

import mfc_inputs as mi
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


@pytest.mark.parametrize("shape", [(64, 32), (64, 33), (683, 3), (2100, 1000)], ids=str)
def test_agent_step_from_a_given_biomass(P, shape):
    cls = mi.bernoulli_block(shape, 0.2, 7)
    rng = np.random.default_rng(5)
    bio = np.where((rng.random(cls.size) < 0.02) & (cls == 0), 400.0 + 150.0 * rng.random(cls.size), 0.0)
    g = P.Lattice(shape)
    g.set_geometry(cls)
    g.step_coupled(2)
    _, _, c, _ = g.read_fields()
    g.write_biomass(bio)
    sg = g.agent_step(P.agent_params(seed=3, growth=0.1, max_walk=200), 1)
    o = oracle.Oracle(shape, cls)
    so = o.agent_step(oracle.agent_table1(seed=3, mu=0.1, max_walk=200), 1, bio, conc=c)
    assert np.array_equal(g.read_biomass(), bio)
    for k in ("attached", "front", "spread", "walks_failed", "walk_steps", "biofilm_nodes"):
        assert sg[k] == so[k], (k, sg[k], so[k])
    assert so["spread"] > 0
    # sums of up to 2.1e6 positive doubles in two orders differ by at most n eps = 5e-10
    assert sg["total_biomass"] == pytest.approx(so["total_biomass"], rel=1e-9)
    g.close()
