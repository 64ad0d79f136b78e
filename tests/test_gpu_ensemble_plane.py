"""A member whose z plane holds 2^22 nodes and more: the batched kernels divide
node numbers by the plane exactly at any size, so it runs as it does alone."""
import numpy as np
import pytest
import torch

from parity import frames_ou

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(2048, 2048), (2051, 2053)])
def test_member_with_a_large_z_plane(nx, ny):
    from paper_2403_01161_gb300.sim import Ensemble, Sim

    def make():
        g = Sim((nx, ny, 12), 1.0, frames_ou(3, 2, 1e-5), 3)
        g.add_icosphere(2, 2.0, 0.02, center=(nx - 9.5, ny - 8.25, 5.5))
        return g

    a, b = make(), make()
    E = Ensemble([a])
    E.step(4)
    E.sync()
    b.step(4)
    b.sync()
    nodes = 12 * nx * ny
    stride = (nodes + 63) // 64 * 64
    tail = [76 * stride, 16 * nodes, 16 * nodes, (nodes + 3) // 4 * 4]  # populations, force, velocity, flags
    start = a.ws.numel() - sum((n + 255) // 256 * 256 for n in tail)
    fa, fb = (g.ws[start:start + 76 * stride].view(torch.float32).view(19, stride)[:, :nodes] for g in (a, b))
    # the same arithmetic node by node, except for the order of the additions into the force near the droplet
    worst = max(float((x - y).abs().max()) for x, y in zip(fa, fb))
    assert worst < 1e-6 and float(fa.abs().max()) > 1e-3
    assert (a.patch()[0] == b.patch()[0]).all() and (a.patch()[1] == b.patch()[1]).all()
    assert np.abs(a.mesh()[0] - b.mesh()[0]).max() < 1e-6
