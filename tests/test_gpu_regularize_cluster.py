"""Mesh regularisation on the cluster where its partition can go wrong: fewer
nodes than CTAs, nodes that do not divide evenly, valences above the weight
table, neighbour lists above the address table, the largest mesh of the
allocation-free call, and ensembles whose members differ in size and
parameters, more of them than one launch's large clusters hold."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _rings(t, nv):
    e = np.unique(np.concatenate([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), axis=0)
    return np.concatenate([[0], np.cumsum(np.bincount(e[:, 0], minlength=nv))]), e[:, 1]


def _reference(r, ptr, idx, alpha, gamma, tol, max_iter, sign):
    nv = len(r)
    src = np.repeat(np.arange(nv), np.diff(ptr))
    n = np.diff(ptr)[:, None].astype(float)

    def ring(x):
        s = np.zeros_like(x)
        np.add.at(s, src, x[idx])
        return s

    xq, it, ok = r, 0, False
    while it < max_iter and not ok:
        it += 1
        xp = alpha * r + (1 - alpha) / n * ring(xq)
        xb = xp - (alpha * r + (1 - alpha) * xq)
        x = xp - (gamma * xb + sign * (1 - gamma) / n * ring(xb))
        ok = np.sqrt(((x - xq) ** 2).sum(1)).max() < tol
        xq = x
    return xq, it, ok


def _tube(rings, around):
    """Closed tube: two poles of valence `around` and `rings` rings of `around` nodes."""
    k = np.arange(around)
    r = [np.stack([np.cos(2 * np.pi * k / around), np.sin(2 * np.pi * k / around), np.full(around, 0.3 * j)], 1)
         for j in range(rings)]
    r = np.concatenate([[[0, 0, -0.3]], *r, [[0, 0, 0.3 * rings]]])
    t = []
    for j in range(around):
        a, b = 1 + j, 1 + (j + 1) % around
        t.append((0, b, a))
        for i in range(rings - 1):
            lo, hi = i * around, (i + 1) * around
            t += [(a + lo, b + lo, b + hi), (a + lo, b + hi, a + hi)]
        t.append((a + (rings - 1) * around, b + (rings - 1) * around, len(r) - 1))
    return 5.0 * r, np.array(t)


def _mesh(kind):
    from paper_2403_01161_gb300.sim import icosphere

    if kind.startswith("level"):
        r, t = icosphere(int(kind[5:]), 5.0, (0.0, 0.0, 0.0))
        return r * [1.5, 0.8, 0.9], t
    rings, around = (int(x) for x in kind[4:].split("x"))
    return _tube(rings, around)


# tube1x70: poles above the weight table; tube2x3000: a pole's list above the address table of its CTA;
# tube126x129: 16256 nodes, close to the largest mesh; tube2x8191: exactly the largest, 16384 nodes
@pytest.mark.parametrize("kind", ["level0", "level1", "level3", "tube1x70", "tube2x3000", "tube126x129", "tube2x8191"])
@pytest.mark.parametrize("sign", [1, 0])
def test_noalloc_against_numpy(kind, sign):
    from paper_2403_01161_gb300 import _lib as L

    r, t = _mesh(kind)
    r = r + 0.02 * np.random.default_rng(5).standard_normal(r.shape)
    ptr, idx = _rings(t, len(r))
    want, it, ok = _reference(r, ptr, idx, 0.1, 0.51, 0.01, 40, 1 if sign else -1)
    dev = [torch.as_tensor(x, device="cuda") for x in (r, ptr.astype(np.int32), idx.astype(np.int32))]
    res = torch.zeros(2, dtype=torch.int32, device="cuda")
    L.check(L.load().ibl_regularize_noalloc(*[ctypes.c_void_p(x.data_ptr()) for x in dev], len(r), 0.1, 0.51, 0.01, 40, sign,
                                            ctypes.c_void_p(res.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    torch.cuda.synchronize()
    assert res.tolist() == [it, int(ok)]
    # rounding of a few sums of up to `around` terms an iteration, not amplified by the averaging
    tol = 40 * np.finfo(float).eps * np.abs(r).max() * max(np.diff(ptr).max(), 6)
    assert np.abs(dev[0].cpu().numpy() - want).max() <= tol


def test_noalloc_skips_nan_nodes_like_the_exit_test_does():
    """A non-finite node spoils its neighbourhood but not the exit test (its maximum skips NaN)."""
    from paper_2403_01161_gb300 import _lib as L

    r, t = _mesh("level2")
    ptr, idx = _rings(t, len(r))
    r[7] = np.nan
    dev = [torch.as_tensor(x, device="cuda") for x in (r, ptr.astype(np.int32), idx.astype(np.int32))]
    res = torch.zeros(2, dtype=torch.int32, device="cuda")
    L.check(L.load().ibl_regularize_noalloc(*[ctypes.c_void_p(x.data_ptr()) for x in dev], len(r), 0.1, 0.51, 0.01, 100, 1,
                                            ctypes.c_void_p(res.data_ptr()),
                                            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    torch.cuda.synchronize()
    assert res.tolist()[1] == 1 and res.tolist()[0] < 100


@pytest.mark.parametrize("members", [3, 9, 67])
def test_batched_regularisation_matches_one_at_a_time(members):
    from paper_2403_01161_gb300 import inputs
    from paper_2403_01161_gb300.sim import Ensemble, Sim

    def make(k):
        n = (20 + 2 * (k % 3),) * 3
        g = Sim(n, 1.0, inputs.ou_gradients(k, 2, 1.0, 5.0, 4e-3), 9, precision="fp64")
        g.add_icosphere(k % 3 + 1, 3.0 + 0.25 * (k % 4), 0.02)
        if k % 5 != 4:  # every fifth member is not regularised
            g.set_regularization(alpha=0.05 + 0.05 * (k % 3), tol=0.01 / (1 + k % 2), every=2 + k % 3)
            g.set_regularization_keep_volume(k % 2 == 0)
            if k % 4 == 3:
                g.set_regularization_trigger(1.3)
        return g

    a, b = [make(k) for k in range(members)], [make(k) for k in range(members)]
    E = Ensemble(a)
    E.step(12)
    E.sync()
    for k, (x, y) in enumerate(zip(a, b)):
        y.step(12)
        y.sync()
        assert x.regularization_stats()[0] == y.regularization_stats()[0]
        assert abs(x.regularization_stats()[1] - y.regularization_stats()[1]) < 1e-10
        assert np.abs(x.mesh()[0] - y.mesh()[0]).max() < 1e-12, k
        assert (x.patch()[0] == y.patch()[0]).all() and (x.patch()[1] == y.patch()[1]).all()
