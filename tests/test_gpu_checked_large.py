"""The checking build on lattices large enough for strips (2-D, from a million nodes on) and for two steps per
launch (3-D): no element offset out of range, no guard byte changed.  A child process loads the checking
library, as in test_gpu_checked_build.py."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

CASES = [((1203, 853), 0, 0, (2, 0), "strip"), ((1203, 853), 1, 0, (2, 0), "strip"), ((1021, 1013), 0, 9, (2, 0), "strip"),
         ((2049, 509), 1, 9, (2, 0), "strip"), ((1021, 1013), 0, 0, (0, 0), "strip"), ((17, 65535), 0, 0, (2, 0), "strip"),
         ((119, 119, 120), 0, 0, (0, 0, 2), "march"), ((60, 114, 64), 0, 0, (0, 0, 2), "march"),
         ((120, 113, 67), 0, 0, (0, 0, 0), "march"), ((245, 59, 134), 0, 0, (0, 0, 2), "march")]


def _exercise():
    sys.path.insert(0, ROOT)
    import paper_1802_07525_gb300 as P
    assert P.lib().mfc_check_build() == 1
    for shape, prec, aq, bc, kernel in CASES:
        for k_half in (0.0, 0.05):
            with P.Lattice(shape, bc=bc, precision=prec, ade_q=aq, tau=0.7, tau_c=0.9, u_in=0.03, c_in=0.8,
                           k_sink=0.01, k_half=k_half) as g:
                rng = np.random.default_rng(len(shape))
                r = rng.random(int(np.prod(shape)))
                g.set_geometry(np.where(r < 0.15, 3, np.where(r < 0.3, 4, np.where(r < 0.35, 5, 0))).astype(np.uint8))
                assert g.plain_plan(100)["kernel"] == kernel, shape
                for n in (2, 3, 6):
                    g.step_coupled_plain(n)
                g.step_flow(5)
                g.step_ade(5)
                g.synchronize()  # raises where an offset was out of range
                assert g.check_canaries() == 0, shape
    print("checked build: no offset out of range, guards intact")


def test_checked_build_of_strips_and_columns():
    from paper_1802_07525_gb300 import build
    build.build(check_bounds=True)
    env = dict(os.environ, MFC_LIBRARY="check")
    r = subprocess.run([sys.executable, os.path.abspath(__file__)], env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "no offset out of range" in r.stdout


if __name__ == "__main__":
    _exercise()
