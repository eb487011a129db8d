"""3-D plain steps with periodic axes: a state and a geometry shifted along the periodic axes step, bit for bit,
to the shifted result, so every image of a boundary population has to be in its place; and they cost little
more than steps between walls."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, PE, IO = 0, 1, 2  # boundary kinds
KW = dict(tau=0.7, tau_c=0.6, u_in=0.005, k_sink=5e-4, k_half=0.05)


@pytest.fixture(scope="module")
def P():
    import paper_1802_07525_gb300 as p
    from paper_1802_07525_gb300 import build
    build.build()
    return p


@pytest.mark.parametrize("shape", [(12, 7, 9), (9, 8, 5), (65, 3, 4), (1, 5, 6), (2, 1, 3), (40, 33, 20)], ids=str)
@pytest.mark.parametrize("bc", [(PE, PE, PE), (PE, PE, IO), (W, PE, PE), (PE, W, IO), (PE, W, PE)], ids=str)
@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_shift_along_periodic_axes(P, shape, bc, prec):
    rng = np.random.default_rng(7)
    n = int(np.prod(shape))
    grid = tuple(reversed(shape))
    cls = rng.choice([0, 0, 0, 0, 0, 3, 4, 5], n).astype(np.uint8)
    f = 1 / 19 + 1e-3 * rng.standard_normal((19, n))
    g = 1 / 7 + 1e-2 * rng.standard_normal((7, n))
    shift = [int(rng.integers(1, s + 1)) if b == PE else 0 for s, b in zip(shape, bc)]

    def moved(a):
        return np.ascontiguousarray(np.roll(a.reshape((-1,) + grid), shift[::-1], axis=(1, 2, 3)).reshape(a.shape[0], n))

    out = []
    for m in (lambda a: a, moved):
        with P.Lattice(shape, bc=bc, precision=getattr(P, prec), **KW) as lat:
            lat.set_geometry(m(cls[None])[0])
            lat.write_populations(P.MFC_POP_FLOW, m(f))
            lat.write_populations(P.MFC_POP_ADE, m(g))
            assert lat.plain_plan(6)["kernel"] == "row"
            lat.step_coupled_plain(6)
            lat.step_flow(3)
            lat.step_ade(3)
            out.append([lat.read_populations(w) for w in (P.MFC_POP_FLOW, P.MFC_POP_ADE)])
    for a, b in zip(*out):
        assert np.isfinite(a).all() and np.array_equal(moved(a), b)


@pytest.mark.parametrize("prec", ["MFC_FP32", "MFC_FP16_DEV"])
def test_periodic_axes_cost_less_than_twice_the_walls(P, prec):
    """Images written through general loops over memory made the step four times as long (FP32)."""
    shape, steps = (128, 128, 128), 40

    def best(bc):
        with P.Lattice(shape, bc=bc, precision=getattr(P, prec), **KW) as lat:
            lat.set_geometry(np.zeros(int(np.prod(shape)), np.uint8))
            t = []
            for _ in range(6):
                lat.synchronize()
                t0 = time.perf_counter()
                lat.step_coupled_plain(steps)
                lat.synchronize()
                t.append(time.perf_counter() - t0)
            return min(t)

    assert best((PE, PE, IO)) < 2 * best((W, W, IO))
