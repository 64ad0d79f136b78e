"""The droplet patch exactly: from the positions its kernel saw (those before
the last step, or the mesh as attached), floors of the bounding box, one node
of stencil below and two above, one node of motion on each side, clamped at
walls and wrapped on periodic axes."""
import numpy as np
import pytest

from parity import frames_ou
from test_gpu_stencil import _mesh, N

pytestmark = pytest.mark.gpu

CASES = [((0, 0, 0), (0.0, 0.0, 0.0)), ((0, 0, 0), (-1e-9, 1e-9, -2e-16)), ((0, 0, 0), (3.0, -2.5, 4.0)),
         ((1, 1, 1), (10.0, -9.0, 11.5)), ((1, 0, 1), (-3 * 22 - 9.5, 0.0, 5 * 24 + 12.0)), ((0, 1, 0), (0.0, 10.0 - 1e-9, 0.0))]


def _expected(r, bc):
    lo, ext = [], []
    for a in range(3):
        l, h = int(np.floor(r[:, a].min())) - 2, int(np.floor(r[:, a].max())) + 3
        if bc[a]:
            if h - l + 1 >= N[a]:
                l, h = 0, N[a] - 1
            l, h = l % N[a], l % N[a] + h - l
        else:
            l, h = max(l, 0), min(h, N[a] - 1)
        lo.append(l)
        ext.append(h - l)
    return lo, ext


def _sim(bc, shift, precision):
    from paper_2403_01161_gb300.sim import Sim

    r, t = _mesh(shift)
    g = Sim(N, 0.9, frames_ou(8, 3, 4e-3), 4, bc=bc, precision=precision)
    g.add_mesh(r, t, 0.02)
    return g


@pytest.mark.parametrize("bc,shift", CASES)
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_patch_of_a_droplet(bc, shift, precision):
    g = _sim(bc, shift, precision)
    seen = g.mesh()[0]
    for _ in range(8):
        lo, ext = g.patch()
        assert (list(lo), list(ext)) == _expected(seen, bc)
        seen = g.mesh()[0]
        g.step(1)
        g.sync()


def test_patches_of_an_ensemble():
    from paper_2403_01161_gb300.sim import Ensemble

    sims = [_sim(bc, shift, "fp32") for bc, shift in CASES]
    E = Ensemble(sims)
    seen = [g.mesh()[0] for g in sims]
    for _ in range(5):
        for g, r, (bc, _) in zip(sims, seen, CASES):
            lo, ext = g.patch()
            assert (list(lo), list(ext)) == _expected(r, bc)
        seen = [g.mesh()[0] for g in sims]
        E.step(1)
        E.sync()
