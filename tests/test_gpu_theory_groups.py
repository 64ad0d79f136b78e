"""Linear theory where its lane groups and eigen-solve can go wrong: frame
counts around the group widths, repeated and nearly repeated eigenvalues,
resting frames, and non-finite gradients."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps


def _full(o):
    S = np.empty(o.shape[:-1] + (3, 3))
    for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        S[..., i, j] = S[..., j, i] = o[..., c]
    return S


def _frames(kind, n_traj, n_frames, rng):
    A = rng.standard_normal((n_traj, n_frames, 3, 3)) * 1e-4
    A -= np.trace(A, axis1=2, axis2=3)[..., None, None] / 3 * np.eye(3)
    if kind != "random":
        q, _ = np.linalg.qr(rng.standard_normal((n_traj, 3, 3)))
        d = {"stretch": (2.0, -1.0, -1.0), "squeeze": (1.0, 1.0, -2.0), "near": (1.0, 1.0 - 1e-6, -2.0 + 1e-6),
             "shear": (1.0, 0.0, -1.0), "axes": (2.0, -1.0, -1.0), "rest": (0.0, 0.0, 0.0)}[kind]
        if kind == "axes":
            q = np.broadcast_to(np.eye(3), q.shape)
        E = np.einsum("tia,a,tja->tij", q, np.array(d) * 1e-4, q)
        A = np.repeat(E[:, None], n_frames, axis=1)
    return A


@pytest.mark.parametrize("kind", ["random", "stretch", "squeeze", "near", "shear", "axes", "rest"])
@pytest.mark.parametrize("n_frames", [1, 2, 3, 8, 9, 31, 32, 33, 64, 65, 257])
def test_frames_around_the_group_widths(kind, n_frames):
    from paper_2403_01161_gb300.theory import linear_theory

    n_traj, hold, tau, R, chi = 5, 120.0, 700.0, 9.0, 1.0
    A = _frames(kind, n_traj, n_frames, np.random.default_rng(n_frames))
    out = linear_theory(A, tau, R, hold, chi, substeps=256).cpu().numpy()
    a = O.lt_coefficients(chi)[0] / tau
    scale = 2 * R * R * O.lt_coefficients(chi)[1] * 1e-3 / a
    for t in range(n_traj):
        # RK4 error of one step is |z|^5/120 of the distance to the fixed point; rounding: a few eps per frame
        rk4 = n_frames * 256 * (a * hold / 256) ** 5 / 120
        tol = scale * (2 * rk4 + 20 * n_frames * EPS) + 4 * EPS * R * R
        assert np.abs(_full(out[t]) - O.lt_trajectory(A[t], hold, tau, R, chi)).max() <= tol
    # observables of the S that came back
    S = _full(out)
    lam, vec = np.linalg.eigh(S)
    assert np.abs(out[..., 6] - lam[..., 2] / R ** 2).max() <= 20 * EPS * lam.max() / R ** 2
    p, q = np.sqrt(lam[..., 2]), np.sqrt(lam[..., 0])
    assert np.abs(out[..., 8] - (p - q) / (p + q)).max() <= 20 * EPS * lam.max() / lam.min()
    E = 0.5 * (A + A.transpose(0, 1, 3, 2))
    nE = np.linalg.norm(E, axis=(2, 3))
    if kind == "rest":
        assert np.isnan(out[..., 7]).all()
        return
    v = vec[..., 2]
    beta = np.einsum("tki,tkij,tkj->tk", v, E, v) / nE
    gap = lam[..., 2] - lam[..., 1]
    if kind in ("squeeze", "axes", "stretch", "near"):
        # S and E commute: beta does not depend on the vector chosen in a repeated pair
        assert np.abs(out[..., 7] - beta).max() <= 1e-5
    far = gap > 1e-6 * lam[..., 2]
    assert (np.abs(out[..., 7] - beta)[far] <= (40 * EPS * lam[..., 2] / np.maximum(gap, 1e-300) + 20 * EPS)[far]).all()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n_frames,at", [(40, 0), (40, 17), (100, 63), (100, 99)])
def test_a_bad_gradient_spoils_its_trajectory_from_there_on(bad, n_frames, at):
    from paper_2403_01161_gb300.theory import linear_theory

    A = _frames("random", 4, n_frames, np.random.default_rng(3))
    good = linear_theory(A, 700.0, 9.0, 120.0).cpu().numpy()
    A[2, at, 1, 1] = bad
    out = linear_theory(torch.as_tensor(A), 700.0, 9.0, 120.0).cpu().numpy()
    assert np.array_equal(out[[0, 1, 3]], good[[0, 1, 3]])
    assert np.array_equal(out[2, :at], good[2, :at])
    assert np.isnan(out[2, at:, 1]).all() and np.isnan(out[2, at:, 8]).all()
