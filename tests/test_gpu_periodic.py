"""FP32 update outside the patch in boxes with periodic axes, against the
oracle: every combination of axes, the patch across a periodic end, one tile
and four tiles per block, and an ensemble."""
import itertools

import numpy as np
import pytest

from parity import frames_ou, lib_to_oracle_perm, make_pair

pytestmark = pytest.mark.gpu

AXES = [bc for bc in itertools.product((0, 1), repeat=3) if any(bc)]


def _pair(n, bc, seed):
    fr = frames_ou(seed, 4, 2e-3)
    for a in range(3):
        if bc[a]:  # the linear flow must not vary along a periodic axis
            fr[:, :, a] = 0.0
    c = tuple(1.25 if bc[a] else 0.5 * (n[a] - 1) for a in range(3))
    g, o = make_pair(n, 0.9, fr, 2, bc=bc, precision="fp32")
    g.add_icosphere(2, 3.5, 0.02, center=c)
    r, _, t = g.mesh()
    o.set_mesh(r, t, 0.02)
    return g, o


def _check(g, o, steps):
    o.step(steps)
    # deviations of about 1e-2 in FP32 over a few steps, as for the boxes without a droplet
    assert np.abs(g.populations()[lib_to_oracle_perm()] - o.populations()).max() < 1e-6
    assert np.abs(g.mesh()[0] - o.mesh()[0]).max() < 1e-6
    assert g.status() == 0


# (82, 81, 80): above the size up to which a block takes four tiles
@pytest.mark.parametrize("n", [(21, 18, 19), (82, 81, 80)])
@pytest.mark.parametrize("bc", AXES)
def test_outside_update_on_periodic_axes(n, bc):
    g, o = _pair(n, bc, 5)
    g.step(5)
    g.sync()
    _check(g, o, 5)


def test_ensemble_on_periodic_axes():
    from paper_2403_01161_gb300.sim import Ensemble

    pairs = [_pair((17 + 2 * k, 20 - k, 18), bc, k) for k, bc in enumerate(AXES + [(0, 0, 0)])]
    E = Ensemble([g for g, _ in pairs])
    E.step(5)
    E.sync()
    for g, o in pairs:
        _check(g, o, 5)
