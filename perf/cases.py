"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a dict of plain values.  `listed()` names the ones that stand for the
workloads of `paper_2403_01161_gb300/config.py`, the benchmark and the tests;
`draw(rng)` gives more of the same ranges (ragged boxes, other radii, levels,
schedules, precisions, ensemble and trajectory counts).  `prepare` builds what
a program holds before the call, `run` is one call through the public entry
points, `work` what one call cannot do without, and `exact` the same result in
64 bits from plain torch, written here from the method's equations.

Kinds:
  droplet     one droplet in a box: `steps` time steps, then its shape record
              (`frames` = 1: one gradient frame through Sim.run_frames, host
              gradient in, host record out)
  lattice     a box without a droplet: `steps` time steps
  ensemble    uneven droplets advanced together by Ensemble.step
  adjoint     D of the final droplet and its gradients w.r.t. sigma and the
              gradient frames, through the autograd function
  theory      the linear theory along many gradient trajectories
  regularize  one mesh regularisation on caller buffers (C ABI)
"""
import ctypes
import math
from types import SimpleNamespace

import numpy as np
import torch

NU_RATIO = 0.472        # R / eta of the paper's largest runs; a droplet's `ratio` below it means a weaker gradient
FRAME_RATIO = 2.25e-3 / 2.3e-2  # gradient frame interval over tau_eta
REG = dict(alpha=0.1, gamma=0.51, tol=0.01, max_iter=100)


def listed():
    return [
        # steady-shear validation box: the smallest simulation, FP64, where launches and latency count
        dict(name="shear_32_fp64", kind="droplet", nx=32, ny=32, nz=32, fp64=True, R=5.0, level=3, Ca=0.1, ratio=0.08,
             tau=1.0, steps=48, reg=0, volume=False, chi=1.0, recentre=False, records=0, frames=0),
        # the forward run of the fitting workload: a small FP32 box that lives in L2
        dict(name="droplet_64", kind="droplet", nx=64, ny=64, nz=64, fp64=False, R=8.0, level=3, Ca=0.2, ratio=0.12,
             tau=1.0, steps=96, reg=0, volume=False, chi=1.0, recentre=False, records=0, frames=0),
        # the headline single droplet, a shape record every 100 steps
        dict(name="droplet_128", kind="droplet", nx=128, ny=128, nz=128, fp64=False, R=12.0, level=4, Ca=0.2, ratio=0.25,
             tau=1.0, steps=300, reg=0, volume=False, chi=1.0, recentre=False, records=100, frames=0),
        # the paper's production box: one gradient frame of the trajectory loop, regularised after every step
        dict(name="production_200", kind="droplet", nx=200, ny=200, nz=200, fp64=False, R=19.0, level=5, Ca=0.2, ratio=NU_RATIO,
             tau=1.5, steps=96, reg=1, volume=False, chi=1.0, recentre=False, records=0, frames=1),
        # the largest box: strong gradients, regularised every 50 steps
        dict(name="stress_256", kind="droplet", nx=256, ny=256, nz=256, fp64=False, R=24.0, level=5, Ca=0.5, ratio=1.0,
             tau=1.0, steps=150, reg=50, volume=False, chi=1.0, recentre=False, records=0, frames=0),
        # a ragged box with every option on: viscosity ratio, boundary field centred on the droplet, volume kept
        dict(name="viscous_72x64x88", kind="droplet", nx=72, ny=64, nz=88, fp64=False, R=8.5, level=4, Ca=0.1, ratio=0.12,
             tau=1.0, steps=60, reg=10, volume=True, chi=3.0, recentre=True, records=0, frames=0),
        # flow without a droplet in an odd-sized channel (periodic along x), smaller than L2
        dict(name="channel_97x75x61", kind="lattice", nx=97, ny=75, nz=61, px=True, py=False, pz=False, fp64=False,
             tau=0.8, rate=4e-4, steps=96),
        # the uneven ensemble: boxes 48^3 to 96^3, each droplet on its own gradient trajectory
        dict(name="ensemble_32", kind="ensemble", members=32, draw=1000, lo=48, hi=96, Rlo=6.0, Rhi=10.0, level=0, Ca=0.2,
             ratio=NU_RATIO, steps=48, reg=0, volume=False, recentre=False, records=0),
        # the statistics ensemble: equal droplets, regularised and centred, one gradient frame (a record at its end)
        dict(name="statistics_16", kind="ensemble", members=16, draw=0, lo=72, hi=72, Rlo=9.0, Rhi=9.0, level=4, Ca=0.05,
             ratio=NU_RATIO, steps=212, reg=10, volume=True, recentre=True, records=212),
        # fitting sigma and the gradients: forward, checkpointed recomputation and reverse sweep
        dict(name="adjoint_64", kind="adjoint", n=64, R=8.0, level=3, Ca=0.2, steps=600, K=100, fp64=False),
        # linear-theory statistics over many trajectories
        dict(name="theory_1000x2000", kind="theory", trajectories=1000, frames=2000, substeps=8, chi=1.0, Ca=0.1),
        # regularising a caller's mesh (level-5 sphere, stretched and jittered) without allocating
        dict(name="regularize_10242", kind="regularize", level=5, R=19.0, noise=0.1),
    ]


def draw(rng):
    kind = rng.choice(["droplet"] * 5 + ["lattice"] * 2 + ["ensemble"] * 2 + ["adjoint", "theory", "regularize"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "droplet":
        fp64 = rng.random() < 0.25
        n = size(28, 72 if fp64 else 180)
        nx, ny, nz = (max(26, int(n * rng.uniform(0.85, 1.15))) for _ in range(3))
        m = min(nx, ny, nz)
        R = round(rng.uniform(4.0, max(4.5, min(24.0, (m - 8) / 4.0))) * 2) / 2
        level = 3 if R < 8 else (4 if R < 16 else 5)
        reg = rng.choice([0, 0, 1, 10, 50])
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, fp64=fp64, R=R, level=level, Ca=round(rng.uniform(0.05, 0.3), 3),
                    ratio=round(0.013 * R, 3), tau=rng.choice([0.8, 1.0, 1.5]), steps=150 if reg == 50 else (60 if reg == 10 else 48),
                    reg=reg, volume=reg > 0 and rng.random() < 0.4, chi=rng.choice([1.0, 1.0, 0.5, 3.0]),
                    recentre=rng.random() < 0.3, records=0, frames=int(rng.random() < 0.3))
    if kind == "lattice":
        fp64 = rng.random() < 0.25
        n = size(20, 96 if fp64 else 220)
        return dict(kind=kind, nx=int(n * rng.uniform(0.7, 1.3)), ny=int(n * rng.uniform(0.7, 1.3)),
                    nz=int(n * rng.uniform(0.7, 1.3)), px=rng.random() < 0.5, py=rng.random() < 0.3, pz=rng.random() < 0.3,
                    fp64=fp64, tau=rng.choice([0.8, 1.0, 1.5]), rate=rng.uniform(1e-4, 2e-4), steps=48)
    if kind == "ensemble":
        reg = rng.choice([0, 0, 10])
        return dict(kind=kind, members=rng.randint(2, 24), draw=rng.randint(1, 9999), lo=40, hi=rng.choice([56, 72, 96]),
                    Rlo=5.0, Rhi=rng.choice([6.0, 7.5, 9.0]), level=0, Ca=round(rng.uniform(0.05, 0.2), 3), ratio=0.15,
                    steps=60 if reg else 48, reg=reg, volume=reg > 0 and rng.random() < 0.5, recentre=rng.random() < 0.4,
                    records=0)
    if kind == "adjoint":
        n = rng.randint(32, 60)
        return dict(kind=kind, n=n, R=round(rng.uniform(4.0, n / 7.0), 1), level=3 if n > 40 else 2, Ca=0.2,
                    steps=rng.randint(90, 300), K=rng.choice([30, 50, 96]), fp64=False)
    if kind == "theory":
        return dict(kind=kind, trajectories=size(16, 2000), frames=size(50, 1000), substeps=rng.choice([1, 4, 8, 50]),
                    chi=rng.choice([0.0, 1.0, 4.0]), Ca=round(rng.uniform(0.02, 0.2), 3))
    level = rng.choice([2, 3, 4, 5])
    return dict(kind=kind, level=level, R=round(rng.uniform(4.0, 8.0) * 2.0 ** (level - 3), 2), noise=round(rng.uniform(0.02, 0.2), 3))


# ---- inputs, from the case and the seed alone -----------------------------

def _traceless(x):
    return x - (np.trace(x, axis1=-2, axis2=-1) / 3.0)[..., None, None] * np.eye(3)


def _ou(rng, n_traj, n_frames, theta, rms):
    """Traceless Ornstein-Uhlenbeck gradients (n_traj, n_frames, 3, 3): frame interval over correlation time theta."""
    a, b, s = math.exp(-theta), math.sqrt(1.0 - math.exp(-2.0 * theta)), rms / math.sqrt(8.0)
    out = np.empty((n_frames, n_traj, 3, 3))
    out[0] = s * _traceless(rng.standard_normal((n_traj, 3, 3)))
    for k in range(1, n_frames):
        out[k] = a * out[k - 1] + b * s * _traceless(rng.standard_normal((n_traj, 3, 3)))
    return np.ascontiguousarray(out.transpose(1, 0, 2, 3))


def _sphere(level):
    """Unit icosphere: positions (nv, 3), outward triangles (nt, 3)."""
    p = (1.0 + 5.0 ** 0.5) / 2.0
    v = np.array([(-1, p, 0), (1, p, 0), (-1, -p, 0), (1, -p, 0), (0, -1, p), (0, 1, p), (0, -1, -p), (0, 1, -p),
                  (p, 0, -1), (p, 0, 1), (-p, 0, -1), (-p, 0, 1)])
    d = np.linalg.norm(v[:, None] - v[None], axis=-1)
    t = np.array([(a, b, c) for a in range(12) for b in range(a + 1, 12) for c in range(b + 1, 12)
                  if max(d[a, b], d[b, c], d[c, a]) < 2.1])
    v = v / np.linalg.norm(v, axis=1, keepdims=True)
    flip = np.einsum("ij,ij->i", np.cross(v[t[:, 1]] - v[t[:, 0]], v[t[:, 2]] - v[t[:, 0]]), v[t].sum(1)) < 0
    t[flip] = t[flip][:, ::-1]
    for _ in range(level):
        e = np.sort(np.concatenate([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        mid = v[u].mean(1)
        m = len(v) + inv.reshape(3, -1)
        v = np.concatenate([v, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        t = np.concatenate([np.stack(q, 1) for q in ((t[:, 0], m[0], m[2]), (t[:, 1], m[1], m[0]), (t[:, 2], m[2], m[1]),
                                                     (m[0], m[1], m[2]))])
    return v, np.ascontiguousarray(t, dtype=np.int32)


def _flow(R, Ca, ratio, tau):
    """Lattice-unit scales of a droplet of radius R: rms gradient, frame length in steps, surface tension."""
    nu = (tau - 0.5) / 3.0
    tau_eta = R * R / (nu * ratio ** 2)
    return SimpleNamespace(rms=1.0 / tau_eta, hold=max(1, int(round(FRAME_RATIO * tau_eta))), sigma=nu * R / (Ca * tau_eta),
                           tau_eta=tau_eta)


def _droplet_inputs(n, R, level, Ca, ratio, tau, n_frames, rng):
    """Frames (n_frames, 3, 3), mesh and scales of one droplet: a sphere strained by some percent, a little off centre."""
    s = _flow(R, Ca, ratio, tau)
    s.frames = _ou(rng, 1, n_frames, FRAME_RATIO / 20.0, s.rms)[0]
    v, t = _sphere(level)
    e = rng.standard_normal((3, 3)) * 0.04
    s.r = R * (v @ (np.eye(3) + _traceless(e + e.T))) + [0.5 * (k - 1) for k in n] + rng.uniform(-0.1, 0.1, 3)
    s.tris = t
    return s


def _single(case, seed):
    n = (case["nx"], case["ny"], case["nz"])
    s = _droplet_inputs(n, case["R"], case["level"], case["Ca"], case["ratio"], case["tau"], 64, np.random.default_rng(seed))
    s.n = n
    if case["frames"]:
        s.hold = case["steps"]
    return s


def _lattice_rate(case, seed):
    rng = np.random.default_rng(seed)
    return _traceless(rng.standard_normal((3, 3)))[None] * (case["rate"] / 2.0)


def _members(case, seed):
    """The droplets of an ensemble: sizes from the case, gradients and shapes from the seed."""
    sizes = np.random.default_rng(case["draw"])
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["members"]):
        R = round(sizes.uniform(case["Rlo"], case["Rhi"]) * 2.0) / 2.0
        choice = [x for x in range(case["lo"], case["hi"] + 1, 8) if x >= 6 * R] or [case["hi"]]
        n = (int(sizes.choice(choice)),) * 3
        s = _droplet_inputs(n, R, case["level"] or (3 if R < 8 else 4), case["Ca"], case["ratio"], 1.0, 16, rng)
        s.n = n
        if case["records"]:
            s.hold = case["records"]
        out.append(s)
    return out


def _adjoint_inputs(case, seed):
    s = _flow(case["R"], case["Ca"], NU_RATIO, 1.0)
    s.frames = _ou(np.random.default_rng(seed), 1, case["steps"] // s.hold + 1, FRAME_RATIO / 20.0, s.rms)[0]
    return s


def _theory_inputs(case, seed):
    s = _flow(19.0, case["Ca"], NU_RATIO, 1.5)
    s.frames = _ou(np.random.default_rng(seed), case["trajectories"], case["frames"], FRAME_RATIO / 20.0, s.rms)
    s.tau_sigma = case["Ca"] * s.tau_eta
    return s


def _mesh_inputs(case, seed):
    rng = np.random.default_rng(seed)
    v, t = _sphere(case["level"])
    r = case["R"] * v * [1.3, 0.85, 0.95]
    edge = case["R"] * 1.1 / 2.0 ** case["level"]
    return r + case["noise"] * edge * rng.standard_normal(r.shape), t


# ---- the calls ------------------------------------------------------------

def _populations(sim, frames):
    """The box's population array as it lies in the workspace, [19][stride] in the storage type: after an even number
    of steps slot i of a node holds population i.  Behind the control block (256 bytes) and the frames, each part
    starting on 256 bytes."""
    size = 8 if sim.params.precision == 1 else 4
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    at = 256 + up(72 * frames) + up(9 * size * frames)
    stride = (sim.nodes + 63) // 64 * 64
    part = sim.ws[at:at + 19 * stride * size].view(torch.float64 if size == 8 else torch.float32)
    nx, ny, nz = sim.n
    return part.view(19, stride)[:, :sim.nodes].view(19, nz, ny, nx)


def _positions(sim):
    return sim.mesh_ws[:24 * sim.nv].view(torch.float64).view(sim.nv, 3)


def _sim(case, s, fp64, tau, bc=(0, 0, 0), frames=None):
    from paper_2403_01161_gb300.sim import Sim

    return Sim(s.n, tau, s.frames if frames is None else frames, s.hold, bc=bc, precision="fp64" if fp64 else "fp32")


def _options(sim, case, s):
    sim.add_mesh(s.r, s.tris, s.sigma)
    if case["reg"]:
        sim.set_regularization(every=case["reg"])
        sim.set_regularization_keep_volume(case["volume"])
    if case["recentre"]:
        sim.set_recentring(True)
    if case["records"]:
        sim.set_readout(case["records"])


def prepare(case, seed):
    kind = case["kind"]
    st = SimpleNamespace(case=case)
    if kind == "droplet":
        s = _single(case, seed)
        # a trajectory loop uploads each frame as it comes: capacity for all of its frames, the first one preset
        frames = np.concatenate([s.frames, np.zeros((4032, 3, 3))]) if case["frames"] else s.frames
        st.sim = _sim(case, s, case["fp64"], case["tau"], frames=frames)
        _options(st.sim, case, s)
        if case["chi"] != 1.0:
            st.sim.set_viscosity_ratio(case["chi"])
        st.sim.prepare(case["steps"])
        st.frames, st.done = s.frames, 0
        st.out = {"r": _positions(st.sim), "f": _populations(st.sim, len(frames))}
    elif kind == "lattice":
        from paper_2403_01161_gb300.sim import Sim

        rate = _lattice_rate(case, seed)
        st.sim = Sim((case["nx"], case["ny"], case["nz"]), case["tau"], rate, 1 << 30,
                     bc=(int(case["px"]), int(case["py"]), int(case["pz"])), precision="fp64" if case["fp64"] else "fp32")
        st.sim.prepare(case["steps"])
        st.out = {"f": _populations(st.sim, 1)}
    elif kind == "ensemble":
        from paper_2403_01161_gb300.sim import Ensemble

        sims = []
        for s in _members(case, seed):
            sims.append(_sim(case, s, False, 1.0))
            _options(sims[-1], case, s)
        st.ensemble = Ensemble(sims)
        st.out = {"r": [_positions(g) for g in sims], "f": [_populations(g, 16) for g in sims]}
    elif kind == "adjoint":
        from paper_2403_01161_gb300.autograd import DropletSpec

        s = _adjoint_inputs(case, seed)
        st.spec = DropletSpec((case["n"],) * 3, 1.0, s.hold, case["level"], case["R"], case["steps"], case["K"],
                              "fp64" if case["fp64"] else "fp32")
        st.sigma = torch.tensor(s.sigma, dtype=torch.float32, device="cuda", requires_grad=True)
        st.frames = torch.tensor(s.frames, dtype=torch.float32, device="cuda", requires_grad=True)
    elif kind == "theory":
        s = _theory_inputs(case, seed)
        st.A, st.s = torch.as_tensor(s.frames, device="cuda"), s
    else:
        r, t = _mesh_inputs(case, seed)
        nv = len(r)
        e = np.unique(np.concatenate([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), axis=0)  # directed edges, sorted
        ptr = np.concatenate([[0], np.cumsum(np.bincount(e[:, 0], minlength=nv))])
        dev = lambda x, dt: torch.as_tensor(np.ascontiguousarray(x), dtype=dt, device="cuda")  # noqa: E731
        st.r0, st.r = dev(r, torch.float64), dev(r, torch.float64)
        st.ptr, st.idx = dev(ptr, torch.int32), dev(e[:, 1], torch.int32)
        st.result = torch.zeros(2, dtype=torch.int32, device="cuda")
    return st


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "droplet":
        if case["frames"]:
            rec = st.sim.run_frames(st.frames[st.done % 64][None], case["steps"])[0]
            st.done += 1
        else:
            st.sim.step(case["steps"])
            rec = st.sim.readout()
        return {"record": rec, **st.out}
    if kind == "lattice":
        st.sim.step(case["steps"])
        return st.out
    if kind == "ensemble":
        st.ensemble.step(case["steps"])
        return st.out
    if kind == "adjoint":
        from paper_2403_01161_gb300.autograd import deformation

        D = deformation(st.sigma, st.frames, st.spec)
        gs, gA = torch.autograd.grad(D, (st.sigma, st.frames))
        return {"D": float(D.detach()), "dsigma": gs, "dA": gA}
    if kind == "theory":
        from paper_2403_01161_gb300.theory import linear_theory

        s = st.s
        return linear_theory(st.A, s.tau_sigma, 19.0, float(s.hold), case["chi"], substeps=case["substeps"])
    from paper_2403_01161_gb300 import _lib

    st.r.copy_(st.r0)  # the caller's mesh of this call
    p = lambda x: ctypes.c_void_p(x.data_ptr())  # noqa: E731
    _lib.check(_lib.load().ibl_regularize_noalloc(
        p(st.r), p(st.ptr), p(st.idx), st.r.shape[0], REG["alpha"], REG["gamma"], REG["tol"], REG["max_iter"], 1,
        p(st.result), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
    return {"r": st.r, "result": st.result}


def work(case):
    """Per step and node 19 populations read and written once (152 bytes in FP32), and some 250 operations; per mesh
    node its position read and written, a 64-point stencil each way and six triangles."""
    kind = case["kind"]

    def steps(nodes, nv, n, size):
        return {"bytes": n * (nodes * 38.0 * size + nv * 48.0), "flops": n * (nodes * 250.0 + nv * 64 * 14.0)}

    if kind in ("droplet", "lattice"):
        nodes = case["nx"] * case["ny"] * case["nz"]
        nv = 10 * 4 ** case["level"] + 2 if kind == "droplet" else 0
        return steps(nodes, nv, case["steps"], 8 if case["fp64"] else 4)
    if kind == "ensemble":
        sizes, nodes, nv = np.random.default_rng(case["draw"]), 0, 0
        for _ in range(case["members"]):
            R = round(sizes.uniform(case["Rlo"], case["Rhi"]) * 2.0) / 2.0
            nodes += int(sizes.choice([x for x in range(case["lo"], case["hi"] + 1, 8) if x >= 6 * R] or [case["hi"]])) ** 3
            nv += 10 * 4 ** (case["level"] or (3 if R < 8 else 4)) + 2
        return steps(nodes, nv, case["steps"], 4)
    if kind == "adjoint":
        # forward sweep and reverse sweep once each; the reverse one reads density, velocity and force of every step
        w = steps(case["n"] ** 3, 10 * 4 ** case["level"] + 2, case["steps"], 8 if case["fp64"] else 4)
        return {"bytes": w["bytes"] * (2 + 14 / 38), "flops": w["flops"] * 3}
    if kind == "theory":
        cells = float(case["trajectories"] * case["frames"])
        return {"bytes": cells * 144, "flops": cells * 300}
    nv = 10 * 4 ** case["level"] + 2
    return {"bytes": nv * (48.0 + 28.0), "flops": nv * 100.0}


# ---- the same results in 64 bits ------------------------------------------

_HALF = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]
_C = [(0, 0, 0)] + _HALF + [tuple(-x for x in c) for c in _HALF]
_OPP = [0] + list(range(10, 19)) + list(range(1, 10))
_W = [1 / 3 if sum(map(abs, c)) == 0 else (1 / 18 if sum(map(abs, c)) == 1 else 1 / 36) for c in _C]


def _dot(c, v):
    """c . v for an integer vector c and three tensors v (0 where c has no component)."""
    out = 0.0
    for a in range(3):
        if c[a]:
            out = out + (v[a] if c[a] > 0 else -v[a])
    return out


def _rebuild(g, A, centre, walls):
    """Populations whose source lies outside the box: moving-wall rules on faces, edges and corners (deviations, rho0 = 1)."""
    if not any(walls):
        return g
    nz, ny, nx = g.shape[1:]
    n = (nx, ny, nz)
    h = g.clone()
    options = [(-1, 0, 1) if walls[a] else (0,) for a in range(3)]
    for s in [(a, b, c) for a in options[0] for b in options[1] for c in options[2]]:
        nb = sum(map(abs, s))
        if nb == 0:
            continue
        where, coords = [], []
        for a in range(3):
            lo, hi = (0, 1) if s[a] < 0 else ((n[a] - 1, n[a]) if s[a] > 0 else ((1, n[a] - 1) if walls[a] else (0, n[a])))
            where.append(slice(lo, hi))
            shape = [1, 1, 1]
            shape[2 - a] = hi - lo
            coords.append((torch.arange(lo, hi, dtype=g.dtype, device=g.device) - centre[a]).view(shape))
        at = (where[2], where[1], where[0])
        G = [g[(i,) + at] for i in range(19)]
        uw = [A[a, 0] * coords[0] + A[a, 1] * coords[1] + A[a, 2] * coords[2] for a in range(3)]
        unknown = [any(s[a] and c[a] * s[a] < 0 for a in range(3)) for c in _C]
        if nb == 1:
            ax = [a for a in range(3) if s[a]][0]
            un = s[ax] * uw[ax]
            tan = [i for i in range(19) if _C[i][ax] == 0]
            rho = 1 + (sum(G[i] for i in tan) + 2 * sum(G[i] for i in range(19) if _C[i][ax] * s[ax] > 0) - un) / (1 + un)
            P = [0.0 if a == ax else sum(_C[i][a] * G[i] for i in tan if _C[i][a]) for a in range(3)]
            for j in range(19):
                if _C[j][ax] * s[ax] < 0:
                    i = _OPP[j]
                    t = tuple(0 if a == ax else _C[i][a] for a in range(3))
                    m = sum(map(abs, t))
                    h[(j,) + at] = G[i] - (2 - m) / 6 * rho * _dot(_C[i], uw) - rho / 3 * _dot(t, uw) + 0.5 * _dot(t, P)
            continue
        e = [a for a in range(3) if not s[a]][0] if nb == 2 else None
        new = {}
        for j in range(1, 19):
            if unknown[j] and not unknown[_OPP[j]]:
                i = _OPP[j]
                v = G[i] - 6 * _W[i] * _dot(_C[i], uw)
                if e is not None and _C[i][e]:
                    v = v + 0.25 * _C[i][e] * (G[e + 1] - G[e + 10]) - _C[i][e] / 12 * uw[e]
                new[j] = v
        buried = [j for j in range(1, 19) if unknown[j] and unknown[_OPP[j]]]
        if nb == 3:  # at a corner a buried pair runs between the walls: no component along the summed normal
            buried = [j for j in range(1, 19) if sum(_C[j][a] * s[a] for a in range(3)) == 0]
            new = {j: v for j, v in new.items() if j not in buried}
        fb = sum(new.get(i, G[i]) for i in range(1, 19) if i not in buried) / (22 if nb == 2 else 18)
        for j in buried:
            new[j] = fb + 3 * _W[j] * _dot(_C[j], uw)
        new[0] = 12 * fb
        for j, v in new.items():
            h[(j,) + at] = v
    return h


def _collide(g, F, omega):
    """BGK + forcing: post-collision populations and the half-force velocity."""
    drho = g.sum(0)
    rho = 1 + drho
    j = [sum((g[i] if _C[i][a] > 0 else -g[i]) for i in range(19) if _C[i][a]) for a in range(3)]
    u = [(j[a] + 0.5 * F[a] if F is not None else j[a]) / rho for a in range(3)]
    base = drho - 1.5 * rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)
    out = []
    for i in range(19):
        cu = _dot(_C[i], u)
        eq = _W[i] * (base + rho * cu * (3 + 4.5 * cu)) if i else _W[i] * base
        v = g[i] + omega * (eq - g[i])
        if F is not None:
            uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
            cF = _dot(_C[i], F)
            v = v + (1 - 0.5 * omega) * _W[i] * (3 * (cF - uF) + 9 * cu * cF)
        out.append(v)
    return torch.stack(out), torch.stack(u)


def _stream(p):
    return torch.stack([torch.roll(p[i], _C[i][::-1], (0, 1, 2)) if i else p[i] for i in range(19)])


def _unknown_slots(f, post, walls):
    """Slots whose source lies outside the box keep what the last even step left there: the node's own opposite."""
    nz, ny, nx = f.shape[1:]
    for i in range(1, 19):
        for a, n in ((0, nx), (1, ny), (2, nz)):
            if walls[a] and _C[i][a]:
                at = [slice(None)] * 3
                at[2 - a] = 0 if _C[i][a] > 0 else n - 1
                f[(i, *at)] = post[(_OPP[i], *at)]
    return f


def _phi(x):
    a = x.abs()
    near = 0.125 * (3 - 2 * a + torch.sqrt((1 + 4 * a - 4 * a * a).clamp_min(1e-300)))
    far = 0.125 * (5 - 2 * a - torch.sqrt((-7 + 12 * a - 4 * a * a).clamp_min(1e-300)))
    return torch.where(a < 1, near, torch.where(a < 2, far, torch.zeros_like(a)))


def _stencil(r, n):
    """Flat lattice indices (nv, 64) and 4-point weights of every mesh node."""
    k = torch.arange(4, device=r.device)
    base = torch.floor(r.detach()).long() - 1
    idx = base[:, :, None] + k
    w = _phi(r[:, :, None] - idx)
    at = idx[:, 0, None, None, :] + n[0] * (idx[:, 1, None, :, None] + n[1] * idx[:, 2, :, None, None])
    ww = w[:, 0, None, None, :] * w[:, 1, None, :, None] * w[:, 2, :, None, None]
    return at.reshape(len(r), 64), ww.reshape(len(r), 64)


def _forces(r, t, sigma):
    x = [r[t[:, k]] for k in range(3)]
    N = torch.linalg.cross(x[1] - x[0], x[2] - x[0])
    m = -0.5 * sigma * N / N.norm(dim=1, keepdim=True)
    F = torch.zeros_like(r)
    for k in range(3):
        F = F.index_add(0, t[:, k], torch.linalg.cross(m, x[(k + 2) % 3] - x[(k + 1) % 3]))
    return F


def _volume(r, t):
    """Enclosed volume and volume centroid."""
    p = [r[t[:, k]] - r[0] for k in range(3)]
    v = (p[0] * torch.linalg.cross(p[1], p[2])).sum(1) / 6
    V = v.sum()
    return V, r[0] + (v[:, None] * (p[0] + p[1] + p[2])).sum(0) / 4 / V


def _inside(r, t, n):
    """Nodes under an odd number of triangles (vertical rays a little off the lattice columns)."""
    lo, hi = torch.floor(r.min(0).values).long() - 1, torch.floor(r.max(0).values).long() + 2
    flag = torch.zeros(n[2], n[1], n[0], dtype=torch.bool, device=r.device)
    X = torch.arange(lo[0], hi[0] + 1, device=r.device)
    Y = torch.arange(lo[1], hi[1] + 1, device=r.device)
    Z = torch.arange(lo[2], hi[2] + 1, device=r.device)
    qx = X.double()[None, :, None] + 2.0 ** 0.5 * 1e-7
    qy = Y.double()[:, None, None] + 3.0 ** 0.5 * 1e-7
    a, b, c = (r[t[:, k]] for k in range(3))
    edge = lambda p, q: (q[:, 0] - p[:, 0]) * (qy - p[:, 1]) - (q[:, 1] - p[:, 1]) * (qx - p[:, 0])  # noqa: E731
    e0, e1, e2 = edge(a, b), edge(b, c), edge(c, a)
    hit = ((e0 > 0) & (e1 > 0) & (e2 > 0)) | ((e0 < 0) & (e1 < 0) & (e2 < 0))
    zc = torch.where(hit, (e1 * a[:, 2] + e2 * b[:, 2] + e0 * c[:, 2]) / (e0 + e1 + e2), torch.full_like(e0, -1e30))
    for k, z in enumerate(Z.tolist()):
        flag[z, Y[0]:Y[-1] + 1, X[0]:X[-1] + 1] = ((zc > z).sum(-1) % 2) == 1
    return flag


def _neighbours(t):
    """Directed edges: centre and neighbour of every one-ring entry."""
    e = torch.unique(torch.cat([t[:, [0, 1]], t[:, [1, 2]], t[:, [2, 0]]]), dim=0)
    return e[:, 0], e[:, 1]


def _regularize(r, t, keep):
    i, j = _neighbours(t)
    ni = torch.bincount(i, minlength=len(r)).double()[:, None]
    ring = lambda x: torch.zeros_like(x).index_add(0, i, x[j]) / ni  # noqa: E731
    V0 = _volume(r, t)[0]
    xo, xq, it = r, r, 0
    while it < REG["max_iter"]:
        it += 1
        xp = REG["alpha"] * xo + (1 - REG["alpha"]) * ring(xq)
        xb = xp - (REG["alpha"] * xo + (1 - REG["alpha"]) * xq)
        v = xp - (REG["gamma"] * xb + (1 - REG["gamma"]) * ring(xb))
        d = (v - xq).norm(dim=1).max().item()
        xq = v
        if d < REG["tol"]:
            break
    if keep:
        V, c = _volume(xq, t)
        xq = c + (V0 / V) ** (1 / 3) * (xq - c)
    return xq


def _shape(r, t):
    """Volume, area, centroid, S (3x3)."""
    ref = r[0]
    p = [r[t[:, k]] - ref for k in range(3)]
    v = (p[0] * torch.linalg.cross(p[1], p[2])).sum(1) / 6
    s = p[0] + p[1] + p[2]
    V = v.sum()
    first = (v[:, None] * s).sum(0) / 4
    M = sum(torch.einsum("t,ta,tb->ab", v, q, q) for q in (*p, s)) / 20
    S = 5 * (M - first[:, None] * first[None] / V) / V
    area = 0.5 * torch.linalg.cross(p[1] - p[0], p[2] - p[0]).norm(dim=1).sum()
    return V, area, ref + first / V, S


def _taylor(S):
    lam = torch.linalg.eigvalsh(S)
    p, q = lam[2].sqrt(), lam[0].sqrt()
    return (p - q) / (p + q)


def _record(r, t, A):
    V, area, xc, S = _shape(r, t)
    lam, vec = torch.linalg.eigh(S)
    E = 0.5 * (A + A.T)
    x = vec[:, 2]
    num = lambda y: [float(q) for q in y]  # noqa: E731
    return {"step": None, "frame": None, "reg_iters": None, "err": None, "V": float(V), "area": float(area), "xc": num(xc),
            "S6": num((S[0, 0], S[1, 1], S[2, 2], S[0, 1], S[0, 2], S[1, 2])), "lam": num(lam), "vmax": [None] * 3,
            "D": float(_taylor(S)), "beta": float(x @ E @ x / E.norm())}


def _step(f, r, t, sigma, A, n, walls, omega, chi, recentre, tau):
    """One step from the streamed populations f: post-collision populations, next f, next positions."""
    centre = [0.5 * (k - 1) for k in n]
    F = idx = w = None
    if r is not None:
        if recentre:
            centre = _volume(r, t)[1]
        idx, w = _stencil(r, n)
        Fn = _forces(r, t, sigma)
        F = [torch.zeros(f[0].numel(), dtype=f.dtype, device=f.device)
             .index_add(0, idx.reshape(-1), (Fn[:, a, None] * w).reshape(-1)).view(f.shape[1:]) for a in range(3)]
        if chi != 1.0:
            omega = torch.where(_inside(r, t, n), 1 / (0.5 + chi * (tau - 0.5)), omega)
    post, u = _collide(_rebuild(f, A, centre, walls), F, omega)
    if r is not None:
        r = r + torch.stack([(u[a].reshape(-1)[idx] * w).sum(1) for a in range(3)], 1)
    return post, _stream(post), r


def _start(n, A):
    """Equilibrium of the linear flow A (x - c) at rest density."""
    x = [torch.arange(k, dtype=torch.float64, device=A.device) - 0.5 * (k - 1) for k in n]
    X = (x[0].view(1, 1, -1), x[1].view(1, -1, 1), x[2].view(-1, 1, 1))
    u = [A[a, 0] * X[0] + A[a, 1] * X[1] + A[a, 2] * X[2] for a in range(3)]
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    return torch.stack([_W[i] * (3 * _dot(_C[i], u) + 4.5 * _dot(_C[i], u) ** 2 - 1.5 * uu) for i in range(19)])


def _advance(n, frames, hold, tau, steps, walls=(1, 1, 1), r=None, t=None, sigma=0.0, reg=0, volume=False, chi=1.0,
             recentre=False):
    frames = torch.as_tensor(frames, dtype=torch.float64, device="cuda")
    f = _start(n, frames[0])
    post = None
    for k in range(steps):
        A = frames[min(k // hold, len(frames) - 1)]
        p, f, r = _step(f, r, t, sigma, A, n, walls, 1.0 / tau, chi, recentre, tau)
        if k % 2 == 0:
            post = p
        if reg and (k + 1) % reg == 0:
            r = _regularize(r, t, volume)
    return _unknown_slots(f, post, walls), r, A


def exact(case, seed):
    kind = case["kind"]
    dev = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    if kind == "droplet":
        s = _single(case, seed)
        t = dev(s.tris).long()
        f, r, A = _advance(s.n, s.frames, s.hold, case["tau"], case["steps"], r=dev(s.r), t=t, sigma=s.sigma,
                           reg=case["reg"], volume=case["volume"], chi=case["chi"], recentre=case["recentre"])
        return {"record": _record(r, t, A), "r": r, "f": f}
    if kind == "lattice":
        f, _, _ = _advance((case["nx"], case["ny"], case["nz"]), _lattice_rate(case, seed), 1 << 30, case["tau"],
                           case["steps"], walls=(not case["px"], not case["py"], not case["pz"]))
        return {"f": f}
    if kind == "ensemble":
        out = {"r": [], "f": []}
        for s in _members(case, seed):
            f, r, _ = _advance(s.n, s.frames, s.hold, 1.0, case["steps"], r=dev(s.r), t=dev(s.tris).long(), sigma=s.sigma,
                               reg=case["reg"], volume=case["volume"], recentre=case["recentre"])
            out["r"].append(r)
            out["f"].append(f)
        return out
    if kind == "adjoint":
        from torch.utils.checkpoint import checkpoint

        s = _adjoint_inputs(case, seed)
        n = (case["n"],) * 3
        v, t = _sphere(case["level"])
        t = dev(t).long()
        # the inputs are 32-bit tensors: their values, carried in 64 bits
        sigma = torch.tensor(s.sigma, dtype=torch.float32, device="cuda").double().requires_grad_()
        frames = torch.tensor(s.frames, dtype=torch.float32, device="cuda").double().requires_grad_()
        f, r = _start(n, frames[0]), dev(case["R"] * v + 0.5 * (case["n"] - 1))

        def one(f, r, sigma, A):
            return _step(f, r, t, sigma, A, n, (1, 1, 1), 1.0, 1.0, False, 1.0)[1:]

        for k in range(case["steps"]):
            f, r = checkpoint(one, f, r, sigma, frames[min(k // s.hold, len(frames) - 1)], use_reentrant=False)
        D = _taylor(_shape(r, t)[3])
        gs, gA = torch.autograd.grad(D, (sigma, frames))
        return {"D": float(D.detach()), "dsigma": gs, "dA": gA}
    if kind == "theory":
        s = _theory_inputs(case, seed)
        R, chi, h = 19.0, case["chi"], float(s.hold) / case["substeps"]
        a = 40 * (chi + 1) / ((2 * chi + 3) * (19 * chi + 16)) / s.tau_sigma
        b = 10 * R * R / (2 * chi + 3)
        A = s.frames
        E = 0.5 * (A + A.transpose(0, 1, 3, 2))
        X = np.zeros((A.shape[0], 3, 3))
        S = np.empty_like(A)
        for k in range(A.shape[1]):
            for _ in range(case["substeps"]):  # classical Runge-Kutta of dX/dt = b E - a X
                k1 = b * E[:, k] - a * X
                k2 = b * E[:, k] - a * (X + h / 2 * k1)
                k3 = b * E[:, k] - a * (X + h / 2 * k2)
                k4 = b * E[:, k] - a * (X + h * k3)
                X = X + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
            S[:, k] = X + R * R * np.eye(3)
        lam, vec = np.linalg.eigh(S)
        x = vec[..., 2]
        beta = np.einsum("tka,tkab,tkb->tk", x, E, x) / np.linalg.norm(E, axis=(2, 3))
        p, q = np.sqrt(np.maximum(lam[..., 2], 0)), np.sqrt(np.maximum(lam[..., 0], 0))
        S6 = np.stack([S[..., i, j] for i, j in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], -1)
        return np.concatenate([S6, (lam[..., 2] / R ** 2)[..., None], beta[..., None], ((p - q) / (p + q))[..., None]], -1)
    r, t = _mesh_inputs(case, seed)
    return {"r": _regularize(dev(r), dev(t).long(), False), "result": None}
