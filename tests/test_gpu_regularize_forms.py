"""Mesh regularisation in the forms that a context without room for the widest
cluster gets, and the one-block kernel of meshes above 32768 nodes."""
import ctypes

import numpy as np
import pytest
import torch

from test_gpu_regularize_cluster import _mesh, _reference, _rings

pytestmark = pytest.mark.gpu


# tube2x8191: the largest mesh of the call
@pytest.mark.parametrize("kind", ["level0", "level3", "tube1x70", "tube2x8191"])
@pytest.mark.parametrize("widest", [0, 8, 16])
def test_noalloc_forms_against_numpy(kind, widest):
    from paper_2403_01161_gb300 import _lib as L

    r, t = _mesh(kind)
    r = r + 0.02 * np.random.default_rng(6).standard_normal(r.shape)
    ptr, idx = _rings(t, len(r))
    want, it, ok = _reference(r, ptr, idx, 0.1, 0.51, 0.01, 40, 1)
    dev = [torch.as_tensor(x, device="cuda") for x in (r, ptr.astype(np.int32), idx.astype(np.int32))]
    res = torch.zeros(2, dtype=torch.int32, device="cuda")
    L.check(L.load().ibl_test_regularize_noalloc(*[ctypes.c_void_p(x.data_ptr()) for x in dev], len(r), 0.1, 0.51, 0.01, 40,
                                                 1, ctypes.c_void_p(res.data_ptr()),
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), widest))
    torch.cuda.synchronize()
    assert res.tolist() == [it, int(ok)]
    # rounding of a few sums of up to the valence's terms an iteration, not amplified by the averaging
    tol = 40 * np.finfo(float).eps * np.abs(r).max() * max(np.diff(ptr).max(), 6)
    assert np.abs(dev[0].cpu().numpy() - want).max() <= tol


def test_mesh_above_the_cluster_on_one_block():
    from paper_2403_01161_gb300.sim import Sim, icosphere

    r, t = icosphere(6, 8.0, (15.5, 15.5, 15.5))
    r = (r - 15.5) * [1.3, 0.9, 0.9] + 15.5
    assert len(r) > 32768
    g = Sim((32, 32, 32), 1.0, np.zeros((1, 3, 3)), 1)
    g.add_mesh(r, t, 0.01)
    g.set_regularization(tol=1e-3, max_iter=60)
    it = g.regularize_now()
    ptr, idx = _rings(t, len(r))
    want, n, ok = _reference(r, ptr, idx, 0.1, 0.51, 1e-3, 60, 1)
    assert ok and it == n
    assert np.abs(g.mesh()[0] - want).max() <= 240 * np.finfo(float).eps * np.abs(r).max()


def test_other_widths_are_refused():
    from paper_2403_01161_gb300 import _lib as L

    buf = ctypes.c_void_p(torch.zeros(16, dtype=torch.float64, device="cuda").data_ptr())
    assert L.load().ibl_test_regularize_noalloc(buf, buf, buf, 1, 0.1, 0.51, 0.01, 1, 1, buf, None, 4) == L.IBL_EINVAL
