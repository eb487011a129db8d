"""Thin lattices: the kernels that take several nodes or steps per thread give the bits of single steps there
too, and are no slower than one node per thread and step."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


def _lattice(P, shape, **kw):
    g = P.Lattice(shape, **dict(dict(tau=0.8, tau_c=0.7, u_in=0.01, k_sink=1e-3), **kw))
    rng = np.random.default_rng(3)
    g.set_geometry(rng.choice([0] * 20 + [3, 4, 5], int(np.prod(shape))).astype(np.uint8))
    return g


def _best(g, steps, call):
    t = []
    for _ in range(6):
        g.synchronize()
        t0 = time.perf_counter()
        call(steps)
        g.synchronize()
        t.append(time.perf_counter() - t0)
    return min(t)


@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_3d_thin_planes_cost_no_more_than_one_node_per_thread(P, prec):
    """A plane of 2x2 nodes fills two lanes of a block: its other warps repeated the last pair's work."""
    with _lattice(P, (2, 2, 20000), precision=getattr(P, prec)) as g:
        assert g.plain_plan(1)["kernel"] == "row"
        pairs = _best(g, 60, g.step_coupled_plain)
        g.set_launch(block=128, offsets32=0)
        assert pairs < _best(g, 60, g.step_coupled_plain)


FLAT = [(200000, 1), (200001, 2), (110000, 5), (200000, 4), (400001, 3), (60000, 6), (130001, 8), (7, 2), (1, 1)]


@pytest.mark.parametrize("shape", FLAT, ids=str)
@pytest.mark.parametrize("prec,ade_q", [("MFC_FP32", 0), ("MFC_FP16_DEV", 0), ("MFC_FP32", 9)])
def test_2d_flat_lattices_compute_what_single_steps_compute(P, shape, prec, ade_q):
    out = []
    for n in (11, 1):
        with _lattice(P, shape, precision=getattr(P, prec), ade_q=ade_q) as g:
            assert g.plain_plan(11)["kernel"] == "tile"
            for _ in range(11 // n):
                g.step_coupled_plain(n)
            out.append([g.read_populations(w) for w in (P.MFC_POP_FLOW, P.MFC_POP_ADE)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("shape", [(200000, 1), (200000, 4), (400000, 2), (110000, 5)], ids=str)
@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_2d_flat_lattices_cost_no_more_than_single_steps(P, shape, prec):
    """Tiles were chosen as if their rows beyond a lattice cost nothing: up to five times a single step's time."""
    with _lattice(P, shape, precision=getattr(P, prec)) as g:
        several = _best(g, 48, g.step_coupled_plain)
        assert several < _best(g, 48, lambda n: [g.step_coupled_plain(1) for _ in range(n)])
