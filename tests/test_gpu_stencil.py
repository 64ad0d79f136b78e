"""Stencils and patches where the weights, the wrap and the bounding box can go
wrong: nodes on lattice points and one rounding below them, droplets across a
periodic end (and several periods away), against the oracle."""
import numpy as np
import pytest

import oracle as O
from parity import frames_ou, make_pair

pytestmark = pytest.mark.gpu

N = (22, 20, 24)


def _mesh(shift):
    from paper_2403_01161_gb300.sim import icosphere

    r, t = icosphere(2, 4.0, tuple(0.5 * (k - 1) for k in N))
    # quarters: many coordinates exactly on lattice points and midway
    return np.round(r * 4) / 4 + np.asarray(shift), t


@pytest.mark.parametrize("bc,shift", [
    ((0, 0, 0), (0.0, 0.0, 0.0)), ((0, 0, 0), (-1e-9, 1e-9, -2e-16)), ((0, 0, 0), (0.25, -0.125, 1e-12)),
    ((1, 1, 1), (10.0, -9.0, 11.5)), ((1, 0, 1), (-3 * 22 - 9.5, 0.0, 5 * 24 + 12.0)), ((0, 1, 0), (0.0, 10.0 - 1e-9, 0.0))])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_nodes_on_lattice_points_and_across_periodic_ends(bc, shift, precision):
    r, t = _mesh(shift)
    g, o = make_pair(N, 0.9, frames_ou(8, 3, 4e-3), 4, bc=bc, precision=precision)
    g.add_mesh(r, t, 0.02)
    o.set_mesh(r, t, 0.02)
    for k in range(3):
        # the patch of the next step: floors of the bounding box, stencil reach and one node of motion
        lo, ext = g.patch()
        ra = g.mesh()[0]
        for a in range(3):
            want_lo, want_hi = int(np.floor(ra[:, a].min())) - 2, int(np.floor(ra[:, a].max())) + 3
            if bc[a]:
                assert lo[a] <= want_lo % N[a] and ext[a] >= min(want_hi - want_lo, N[a] - 1) or ext[a] == N[a] - 1
            else:
                assert lo[a] <= max(want_lo, 0) + 1 and lo[a] + ext[a] >= min(want_hi, N[a] - 1) - 1
        g.step(2)
        g.sync()
        o.step(2)
        rg, ro = g.mesh()[0], o.mesh()[0]
        # FP32: velocities of about 0.05 to a few 2^-24 a step, positions to 2^-24 of the stencil fraction
        assert np.abs(rg - ro).max() < (1e-12 if precision == "fp64" else 2e-7)
        assert not np.array_equal(rg, r)
