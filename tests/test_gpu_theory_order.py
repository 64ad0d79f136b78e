"""Linear theory where two axes of the droplet are closer than FP32 resolves:
gradients along the axes and planar ones (no rotation mixes the close pair),
both orders; then a frame under which the two axes differ, so that beta shows
which one was taken as the longest."""
import itertools

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

EPS = np.finfo(np.float64).eps
TAU, R, HOLD, CHI = 700.0, 9.0, 120.0, 1.0


def _trajectory(T, E2, before):
    """Gradients that end at X = S - R^2 I = T after `before` constant frames and one frame of E2."""
    cr, cs = O.lt_coefficients(CHI)
    d = np.exp(-cr * HOLD / TAU)
    c = 2 * R * R * cs * TAU / cr * (1 - d)  # one frame of E adds c E
    X1 = (T - c * E2) / d
    E1 = X1 * (1 - d) / (c * (1 - d ** before))
    return np.concatenate([np.repeat(E1[None], before, 0), E2[None]])


def _block(theta):
    co, si = np.cos(theta), np.sin(theta)
    return np.array([[co, -si, 0.0], [si, co, 0.0], [0.0, 0.0, 1.0]])


@pytest.mark.parametrize("before", [1, 2, 32, 40])
@pytest.mark.parametrize("delta", [2e-8, -2e-8, 6e-8, -6e-8, 3e-7, -3e-7])
def test_axes_closer_than_fp32_resolves(delta, before):
    from paper_2403_01161_gb300.theory import linear_theory

    A, longest = [], []
    for sign, theta, perm in itertools.product((1, -1), (0.0, 0.3, 0.5 * np.pi - 0.2, 1.1),
                                               itertools.permutations(range(3))):
        V = _block(theta)[:, perm]
        # the first two axes are the close pair: the two longest (sign 1) or the two shortest
        x = sign * 4.0 * np.array([1.0, 1.0 + delta, -2.0 - delta])
        E2 = V @ np.diag([-3e-4, 2e-4, 1e-4]) @ V.T
        A.append(_trajectory(V @ np.diag(x) @ V.T, E2, before))
        longest.append(V[:, np.argmax(x)])
    A, longest = np.array(A), np.array(longest)
    out = linear_theory(A, TAU, R, HOLD, CHI, substeps=256).cpu().numpy()[:, -1]
    S = np.empty((len(A), 3, 3))
    for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        S[:, i, j] = S[:, j, i] = out[:, c]
    lam = np.linalg.eigvalsh(S)
    assert np.abs(out[:, 6] - lam[:, 2] / R ** 2).max() <= 20 * EPS * lam.max() / R ** 2
    p, q = np.sqrt(lam[:, 2]), np.sqrt(lam[:, 0])
    assert np.abs(out[:, 8] - (p - q) / (p + q)).max() <= 20 * EPS * lam.max() / lam.min()
    # the close pair is mixed only by the rounding of X and E2, some eps of their size over a gap of |delta|
    E = A[:, -1]
    beta = np.einsum("ti,tij,tj->t", longest, E, longest) / np.linalg.norm(E, axis=(1, 2))
    assert np.abs(out[:, 7] - beta).max() <= 100 * EPS * R ** 2 / abs(delta)


@pytest.mark.parametrize("n_frames,first", [(20, 20), (64, 40), (100, 50), (100, 100)])
def test_rest_under_a_step_beyond_the_stability_limit(n_frames, first):
    """A droplet at rest stays the sphere however large the multiplier of a step is."""
    from paper_2403_01161_gb300.theory import linear_theory

    A = np.zeros((2, n_frames, 3, 3))
    A[1, first:, 0, 1] = A[1, first:, 1, 0] = 1e-4
    a, hold = O.lt_coefficients(CHI)[0] / TAU, 1e6 * TAU
    z = -a * hold
    m = 1 + z * (1 + z * (0.5 + z * (1 / 6 + z / 24)))
    assert 1e20 < m < 1e30
    out = linear_theory(A, TAU, R, hold, CHI, substeps=1).cpu().numpy()
    rest = np.concatenate([out[0], out[1, :first]])
    assert (rest[:, :3] == R * R).all() and (rest[:, 3:6] == 0).all() and (rest[:, 8] == 0).all()
    if first < n_frames:  # the first strained frame: (1 - m) of the way to the fixed point
        want = 2 * R * R * O.lt_coefficients(CHI)[1] * 1e-4 / a * (1 - m)
        assert abs(out[1, first, 3] / want - 1) <= 20 * EPS


@pytest.mark.parametrize("exponent", [-300, -200, 200, 300])
def test_observables_do_not_depend_on_the_size_of_the_droplet(exponent):
    from paper_2403_01161_gb300.theory import linear_theory

    rng = np.random.default_rng(1)
    A = rng.standard_normal((3, 40, 3, 3)) * 1e-4
    A -= np.trace(A, axis1=2, axis2=3)[..., None, None] / 3 * np.eye(3)
    want = linear_theory(A, TAU, 1.0, HOLD, CHI, substeps=8).cpu().numpy()
    out = linear_theory(A, TAU, 2.0 ** exponent, HOLD, CHI, substeps=8).cpu().numpy()
    S = want[..., :6]
    assert np.abs(out[..., :6] * 2.0 ** -exponent * 2.0 ** -exponent - S).max() <= 8 * EPS * S.max()
    # the eigen-solves of the two sizes may differ: eps over the gap to the next axis
    full = np.empty(S.shape[:-1] + (3, 3))
    for c, (i, j) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
        full[..., i, j] = full[..., j, i] = S[..., c]
    lam = np.linalg.eigvalsh(full)
    assert np.abs(out[..., 6] - want[..., 6]).max() <= 40 * EPS * lam.max()
    assert np.abs(out[..., 8] - want[..., 8]).max() <= 40 * EPS * lam.max() / lam.min()
    gap = (lam[..., 2] - lam[..., 1]) / lam[..., 2]
    assert (np.abs(out[..., 7] - want[..., 7]) <= 80 * EPS / gap).all()
