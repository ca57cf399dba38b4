"""Timed workloads of the pose solver, each one call sequence that a user's program makes.

A case is a mesh, a rig, a material, solver options and a number of poses.  What a
program keeps between frames (the solver context with its mesh, the poses of the
next frame, the result buffers) is made by ``prepare``; ``run`` is the call per
frame.  Meshes are voxel bodies cut into tetrahedra: a unit-cube bar, and a capsule
figure with 15 joints (or more, subdivided) posed by forward kinematics.

The SpMV is fixed to one thread per row, and in FP64 to 128 rows per block, as a
program does that wants the same pose to give the same bits on every run: the solver's
own timing of that shape may otherwise split a row's sum (and, in FP64, order the sums
of the tiles) in another way each time.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

from paper_2408_04066_gb300 import mfem

# Material of the figure: Young's modulus 1e5 Pa, Poisson ratio 0.45.
MU = 1.0e5 / (2.0 * 1.45)
LAM = 1.0e5 * 0.45 / (1.45 * 0.10)

# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
_DEFAULTS = dict(call="batch", body="figure", tets=0, joints=15, scale=1.0, model="snh", precision="mixed", poses=1,
                 device=True, penalty=False, forces=False, elements=False, rotation="rig", tets2=0, poses2=0,
                 tets3=0, poses3=0)


def _case(**kw):
    return dict(_DEFAULTS, **kw)


def listed():
    return [
        # a rig editor's smallest scene: one twisted bar, one pose a call, host arrays, FP64
        _case(name="bar-arap-fp64-pose", call="pose", body="bar", tets=1536, joints=2, model="arap", precision="fp64",
              device=False),
        # interactive posing of one character of the flour sack's size, with the stretches and stresses shown
        _case(name="figure11k-snh-pose-elements", call="pose", tets=11193, device=False, elements=True),
        # a few poses of a small co-rotational character held by soft pins and pushed by forces
        _case(name="figure10k-corot-penalty-batch5", tets=10000, model="corot", poses=5, penalty=True, forces=True),
        # a ragged handful of poses of a mid-size character, host arrays
        _case(name="figure50k-snh-batch3", tets=50000, poses=3, device=False),
        # latency of one pose of the large figure, host arrays
        _case(name="figure200k-snh-pose", call="pose", tets=200000, device=False),
        # the same figure, a batch of independent poses on the device: the usual offline bake
        _case(name="figure200k-snh-batch16", tets=200000, poses=16),
        # the quadratic energy on the same bake
        _case(name="figure200k-corot-batch16", tets=200000, model="corot", poses=16),
        # reference results: the FP64 path
        _case(name="figure200k-snh-fp64-batch8", tets=200000, precision="fp64", poses=8),
        # animation: two crowds of characters, the next frame of every stream in one call, warm-started
        _case(name="streams-200k-50k-warm", call="streams", tets=200000, poses=12, tets2=50000, poses2=12),
        # serving: single-pose requests of three resident characters, all in flight at once
        _case(name="served-10k-50k-200k", call="served", tets=10000, poses=6, model="corot", tets2=50000, poses2=6,
              tets3=200000, poses3=4, device=False),
        # a detailed figure, a few poses
        _case(name="figure800k-snh-batch4", tets=800000, poses=4),
        # the film-quality character: 2M tets, 40 joints
        _case(name="character2M-snh-batch16", tets=2000000, joints=40, poses=16),
    ]


def draw(rng):
    """One more case over the same ranges: 1.5k to 1M tets, 1 to 40 poses, every model, precision and call."""
    call = rng.choice(["pose", "batch", "batch", "batch", "streams", "served"])
    precision = "fp64" if call in ("pose", "batch") and rng.random() < 0.25 else "mixed"
    tets = int(round(math.exp(rng.uniform(math.log(1500.0), math.log(1.0e6 if precision == "mixed" else 2.5e5)))))
    # at most ~4M tets (1.6M in FP64) in flight, a quarter of the largest case's poses
    most = max(1, min(40, (4000000 if precision == "mixed" else 1600000) // tets))
    poses = 1 if call == "pose" else int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    c = _case(call=call, tets=tets, joints=rng.choice([15, 15, 22, 40]), precision=precision, poses=poses,
              model=rng.choice(["arap", "corot", "snh", "snh"]), device=call != "pose" and rng.random() < 0.6)
    if call in ("streams", "served"):
        c.update(model="snh" if call == "streams" else c["model"], device=call == "streams",
                 tets=min(tets, 250000), poses=min(poses, 12),
                 tets2=int(round(math.exp(rng.uniform(math.log(1500.0), math.log(6.0e4))))), poses2=rng.randint(1, 12))
    else:
        c.update(penalty=rng.random() < 0.2, forces=rng.random() < 0.2, elements=call == "pose" and rng.random() < 0.5)
    return c


# ---------------------------------------------------------------------------
# Bodies, rigs and poses
# ---------------------------------------------------------------------------
_JOINTS = np.array([[0, 0, .52], [0, 0, .80], [0, 0, .95], [.14, 0, .78], [.38, 0, .78], [.60, 0, .78], [-.14, 0, .78],
                    [-.38, 0, .78], [-.60, 0, .78], [.08, 0, .50], [.09, 0, .27], [.10, 0, .04], [-.08, 0, .50],
                    [-.09, 0, .27], [-.10, 0, .04]])
_PARENT = [-1, 0, 1, 1, 3, 4, 1, 6, 7, 0, 9, 10, 0, 12, 13]
_CAPSULES = [((0, 0, .50), (0, 0, .80), .100), ((0, 0, .86), (0, 0, .95), .065), ((.06, 0, .78), (.62, 0, .78), .038),
             ((-.06, 0, .78), (-.62, 0, .78), .038), ((.08, 0, .50), (.10, 0, .03), .050),
             ((-.08, 0, .50), (-.10, 0, .03), .050)]


def _voxel_tets(occ, h, origin):
    """Six tetrahedra around the main diagonal of every occupied cell."""
    cells = np.argwhere(occ)
    shape = np.array(occ.shape) + 1
    corner = {o: np.ravel_multi_index((cells + o).T, shape) for o in itertools.product((0, 1), repeat=3)}
    used, inv = np.unique(np.concatenate(list(corner.values())), return_inverse=True)
    corner = {o: inv[i * len(cells):(i + 1) * len(cells)] for i, o in enumerate(corner)}
    X = np.stack(np.unravel_index(used, shape), axis=1) * h + origin
    tets = []
    for p in itertools.permutations(range(3)):
        a = [0, 0, 0]
        a[p[0]] = 1
        b = list(a)
        b[p[1]] = 1
        even = sum(p[i] > p[j] for i in range(3) for j in range(i + 1, 3)) % 2 == 0
        path = [(0, 0, 0), tuple(a), tuple(b), (1, 1, 1)]
        if not even:
            path[1], path[2] = path[2], path[1]
        tets.append(np.stack([corner[o] for o in path], axis=1))
    return X, np.stack(tets, axis=1).reshape(-1, 4).astype(np.int32)


def _inside(grid):
    keep = np.zeros(grid.shape[:-1], dtype=bool)
    for a, b, r in _CAPSULES:
        a, ab = np.array(a), np.array(b, dtype=float) - np.array(a)
        t = np.clip(((grid - a) @ ab) / (ab @ ab), 0.0, 1.0)
        keep |= np.sum((grid - a - t[..., None] * ab) ** 2, axis=-1) <= r * r
    return keep


def _figure(tets):
    lo, hi = np.array([-.70, -.15, -.08]), np.array([.70, .15, 1.05])
    h = (6 * 0.0273 / tets) ** (1.0 / 3.0)      # the capsules' volume over six tets a cell, refined below
    for _ in range(3):
        dims = np.ceil((hi - lo) / h).astype(int)
        occ = np.stack([_inside(np.stack(np.meshgrid(lo[0] + (i + .5) * h, lo[1] + (np.arange(dims[1]) + .5) * h,
                                                     lo[2] + (np.arange(dims[2]) + .5) * h, indexing="ij"), -1))[0]
                        for i in range(dims[0])])
        got = 6 * int(occ.sum())
        if abs(got - tets) <= 0.02 * tets:
            break
        h *= (got / tets) ** (1.0 / 3.0)
    return (*_voxel_tets(occ, h, lo), h)


def _rig(n):
    """The figure's skeleton with its bones subdivided to n joints, parents first."""
    bones = [(p, j) for j, p in enumerate(_PARENT) if p >= 0]
    length = np.array([np.linalg.norm(_JOINTS[j] - _JOINTS[p]) for p, j in bones])
    share = (n - len(_JOINTS)) * length / length.sum()
    k = np.floor(share).astype(int)
    k[np.argsort(k - share, kind="stable")[:n - len(_JOINTS) - k.sum()]] += 1
    extra = {j: k[i] for i, (_, j) in enumerate(bones)}
    joints, parent, at = [], [], {}
    for j, p in enumerate(_PARENT):
        up = at.get(p, -1)
        for s in range(1, extra.get(j, 0) + 1):
            joints.append(_JOINTS[p] + s / (extra[j] + 1) * (_JOINTS[j] - _JOINTS[p]))
            parent.append(up)
            up = len(joints) - 1
        joints.append(_JOINTS[j])
        parent.append(up)
        at[j] = len(joints) - 1
    return np.array(joints), np.array(parent, dtype=np.int32)


def _nearest_bone(P, joints, parent):
    """The bone segment nearest each point, as its parent joint."""
    best, who = np.full(len(P), np.inf), np.zeros(len(P), dtype=np.int32)
    for j, p in enumerate(parent):
        if p < 0:
            continue
        ab = joints[j] - joints[p]
        t = np.clip(((P - joints[p]) @ ab) / (ab @ ab), 0.0, 1.0)
        d = np.sum((P - joints[p] - t[:, None] * ab) ** 2, axis=1)
        near = d < best - 1e-10
        best[near], who[near] = d[near], p
    return who


@functools.lru_cache(maxsize=6)     # the asset that a program has loaded
def _asset(body, tets, n_joints):
    if body == "bar":
        X, T = _voxel_tets(np.ones((4, 4, 16), dtype=bool), 1.0, np.zeros(3))
        joints, parent = np.array([[2.0, 2.0, 0.0], [2.0, 2.0, 16.0]]), np.array([-1, -1], dtype=np.int32)
        cluster = (X[T].mean(axis=1)[:, 2] > 8.0).astype(np.int32)
        pins = np.flatnonzero((X[:, 2] == 0.0) | (X[:, 2] == 16.0)).astype(np.int32)
        vhandle = (X[:, 2] > 8.0).astype(np.int32)
    else:
        X, T, h = _figure(tets)
        joints, parent = _rig(n_joints)
        cluster = _nearest_bone(X[T].mean(axis=1), joints, parent)
        vhandle = _nearest_bone(X, joints, parent)
        mids = [0.5 * (joints[j] + joints[p]) for j, p in enumerate(parent) if p >= 0]
        near = np.zeros(len(X), dtype=bool)
        for c in (*joints, *mids):
            near |= np.sum((X - c) ** 2, axis=1) <= (1.5 * h) ** 2
        pins = np.flatnonzero(near).astype(np.int32)
    return dict(X=X, T=T, joints=joints, parent=parent, cluster=cluster, vhandle=vhandle, pins=pins,
                pin_handle=vhandle[pins].astype(np.int32))


def _turn(axis, angle):
    a = axis / np.linalg.norm(axis)
    K = np.array([[0.0, -a[2], a[1]], [a[2], 0.0, -a[0]], [-a[1], a[0], 0.0]])
    return np.eye(3) + math.sin(angle) * K + (1.0 - math.cos(angle)) * (K @ K)


def _chain(joints, parent, turns, shift):
    """Forward kinematics: every joint turns its subtree about itself, the root also shifts."""
    W = np.zeros((len(joints), 4, 4))
    for j, p in enumerate(parent):
        L = np.eye(4)
        L[:3, :3] = turns[j]
        L[:3, 3] = joints[j] - turns[j] @ joints[j] + (shift if p < 0 else 0.0)
        W[j] = L if p < 0 else W[p] @ L
    return W[:, :3, :].reshape(len(joints), 12)


def _poses(body, asset, rng, count):
    """Independent poses: turns up to 45 degrees a joint (20 on a subdivided skeleton, whose chains add up)."""
    joints, parent = asset["joints"], asset["parent"]
    out = []
    for _ in range(count):
        if body == "bar":
            Q = _turn(np.array([0.0, 0.0, 1.0]), rng.uniform(0.25, 1.0) * math.pi / 2)
            t = joints[1] - Q @ joints[1] + np.array([0.0, 0.0, rng.uniform(0.0, 1.0)])
            out.append(np.stack([np.eye(3, 4).reshape(12), np.hstack([Q, t[:, None]]).reshape(12)]))
            continue
        most = math.radians(45.0 if len(joints) == 15 else 20.0)
        turns = [_turn(rng.normal(size=3), rng.uniform(-most, most)) for _ in joints]
        out.append(_chain(joints, parent, turns, rng.uniform(-0.1, 0.1, size=3)))
    return np.ascontiguousarray(out)


_FRAMES = 24


def _clip(asset, rng, count):
    """`count` animation clips of _FRAMES frames at 30 a second, (frames, count, H, 12)."""
    joints, parent = asset["joints"], asset["parent"]
    most = math.radians(45.0 if len(joints) == 15 else 20.0)
    out = np.zeros((_FRAMES, count, len(joints), 12))
    for s in range(count):
        axis, amp = rng.normal(size=(len(joints), 3)), rng.uniform(0.0, most, size=len(joints))
        f, ph = rng.uniform(0.3, 1.0, size=len(joints)), rng.uniform(0.0, 2 * math.pi, size=len(joints))
        rf, rp = rng.uniform(0.3, 1.0, size=3), rng.uniform(0.0, 2 * math.pi, size=3)
        for k in range(_FRAMES):
            t = k / 30.0
            turns = [_turn(axis[j], amp[j] * math.sin(2 * math.pi * f[j] * t + ph[j])) for j in range(len(joints))]
            out[k, s] = _chain(joints, parent, turns, 0.1 * np.sin(2 * math.pi * rf * t + rp))
    return out


def _material(case):
    """Lame constants: the figure's, and 1 (a scale-free energy) for ARAP."""
    return (1.0, 0.0) if case["model"] == "arap" else (MU, LAM)


def _stiffness(case):
    """Penalty stiffness of soft pins."""
    return 10.0 * _material(case)[0]


def _forces(case, asset, rng):
    """A local push on a few dozen vertices around a random one, one field for every pose."""
    X = asset["X"]
    d = np.linalg.norm(X - X[rng.integers(len(X))], axis=1)
    f = np.zeros_like(X)
    f[d <= np.sort(d)[min(len(X) - 1, 40)]] = rng.normal(size=3) * 2e-6 * _material(case)[0] * np.ptp(X, axis=0).max() ** 2
    return f


def _context(case, asset, poses, **over):
    mu, lam = _material(case)
    opts = dict(precision=case["precision"], rotation=case["rotation"], max_batch=max(1, poses), spmv_split=1)
    if case["precision"] == "fp64":
        opts["tile_rows"] = 128
    if case["penalty"]:
        opts.update(constraint="penalty", k_s=_stiffness(case))
    opts.update(over)
    return mfem.Context(asset["X"], asset["T"], asset["joints"], asset["parent"], model=case["model"], mu=mu, lam=lam,
                        pin_verts=asset["pins"], pin_handle=asset["pin_handle"], tet_cluster=asset["cluster"], **opts)


def _parts(case):
    """(tets, poses) of every mesh of the case."""
    return [(case["tets" + s], case["poses" + s]) for s in ("", "2", "3") if case["tets" + s]]


class _Served:
    """A server and its clients' next requests; closed with the program."""

    def __init__(self, meshes):
        self.srv = mfem.Server(max_slots=16)
        self.jobs = []
        for ctx, poses in meshes:
            n = ctx.n
            mid = self.srv.add(ctx)
            self.jobs += [(mid, xf, np.empty((n, 3))) for xf in poses]

    def __del__(self):
        self.srv.close()


# ---------------------------------------------------------------------------
# One frame
# ---------------------------------------------------------------------------
def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["call"] == "streams":
        ctxs, clips = [], []
        for tets, poses in _parts(case):
            a = _asset(case["body"], tets, case["joints"])
            ctxs.append(_context(case, a, poses, init="warm"))
            clips.append(torch.from_numpy(_clip(a, rng, poses)).cuda())
        outs = [torch.empty((p.shape[1], c.n, 3), dtype=torch.float64, device="cuda") for c, p in zip(ctxs, clips)]
        return dict(case=case, ctxs=ctxs, clips=clips, outs=outs, frame=0)
    if case["call"] == "served":
        meshes = []
        for i, (tets, poses) in enumerate(_parts(case)):
            a = _asset(case["body"], tets, case["joints"])
            c = dict(case, model=case["model"] if i == 0 else ("snh" if i == 1 else "corot"))
            meshes.append((_context(c, a, poses), _poses(case["body"], a, rng, poses)))
        return dict(case=case, served=_Served(meshes))
    a = _asset(case["body"], case["tets"], case["joints"])
    xf = _poses(case["body"], a, rng, case["poses"])
    ctx = _context(case, a, case["poses"])
    if case["forces"]:
        ctx.set_forces(_forces(case, a, rng))
    s = dict(case=case, ctx=ctx, xf=xf)
    if case["call"] == "pose":
        s["out"] = np.empty((ctx.n, 3))
    elif case["device"]:
        s["xf"] = torch.from_numpy(xf).cuda()
        s["out"] = torch.empty((case["poses"], ctx.n, 3), dtype=torch.float64, device="cuda")
    else:
        s["out"] = np.empty((case["poses"], ctx.n, 3))
    return s


def run(state):
    case = state["case"]
    if case["call"] == "streams":
        # a clip is played to and fro
        k = state["frame"] % (2 * _FRAMES - 2)
        state["frame"] += 1
        k = k if k < _FRAMES else 2 * _FRAMES - 2 - k
        outs, stats = mfem.solve_multi(state["ctxs"], [c[k] for c in state["clips"]], outs=state["outs"])
        return [{"x": o, "energy": np.array([t["energy"] for t in ts])} for o, ts in zip(outs, stats)]
    if case["call"] == "served":
        sv = state["served"]
        tickets = [sv.srv.submit(mid, xf, out) for mid, xf, out in sv.jobs]
        done = [sv.srv.wait(t) for t in tickets]
        return {"x": [d[0] for d in done], "energy": np.array([d[1]["energy"] for d in done])}
    ctx = state["ctx"]
    if case["call"] == "pose":
        ctx.set_pose(state["xf"][0])
        x, st = ctx.solve(state["out"])
        r = {"x": x, "energy": np.array([st["energy"]])}
        if case["elements"]:
            r["stretch"], r["multiplier"] = ctx.get_elem()
        return r
    x, stats = ctx.solve_batch(state["xf"], out=state["out"])
    return {"x": x, "energy": np.array([t["energy"] for t in stats])}


def work(case):
    """Bytes: the mesh (tets, rest positions, clusters) once, every pose and its positions once.  Flops: the local
    step and its 12 x 12 Hessian of every tet (about 3000) at the start and once more at the solution's
    neighbourhood, which no solver of this energy can leave out."""
    nbytes = flops = 0.0
    for tets, poses in _parts(case):
        n = 0.21 * tets + 60
        nbytes += 20.0 * tets + 24.0 * n + poses * (96.0 * case["joints"] + 24.0 * n)
        flops += 2 * 3000.0 * tets * poses
    if case["elements"]:
        nbytes += 120.0 * case["tets"]
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# The minimiser in 64 bits
# ---------------------------------------------------------------------------
_EXACT_TETS = 210000     # poses x tets a reference solve takes seconds for


def exact(case, seed):
    if case["call"] not in ("pose", "batch") or case["rotation"] != "rig" or case["tets"] * case["poses"] > _EXACT_TETS:
        return None
    rng = np.random.default_rng(seed)
    a = _asset(case["body"], case["tets"], case["joints"])
    xf = _poses(case["body"], a, rng, case["poses"])
    ref = _Reference(case, a, _forces(case, a, rng) if case["forces"] else None)
    got = [ref.solve(p) for p in xf]
    x = torch.stack([g[0] for g in got])
    r = {"x": x[0] if case["call"] == "pose" else x, "energy": np.array([g[1] for g in got])}
    if case["elements"]:
        r["stretch"], r["multiplier"] = got[0][2], got[0][3]
    return r


class _Reference:
    """Newton with block-Jacobi conjugate gradients on the element matrices, plain torch in FP64."""

    def __init__(self, case, asset, force):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda v, d=torch.float64: torch.as_tensor(np.ascontiguousarray(v)).to(dev, d)  # noqa: E731
        self.model, (self.mu, self.lam) = case["model"], _material(case)
        self.X, self.T = t(asset["X"]), t(asset["T"], torch.int64)
        self.cluster, self.vhandle = t(asset["cluster"], torch.int64), t(asset["vhandle"], torch.int64)
        self.pins, self.ph = t(asset["pins"], torch.int64), t(asset["pin_handle"], torch.int64)
        self.ks = _stiffness(case) if case["penalty"] else None
        self.force = None if force is None else t(force)
        D = (self.X[self.T[:, 1:]] - self.X[self.T[:, :1]]).transpose(1, 2)
        self.vol = torch.linalg.det(D) / 6.0
        G = torch.linalg.inv(D)
        self.G = torch.cat([-G.sum(1, keepdim=True), G], dim=1)                 # (m, 4, 3)
        B = torch.zeros(6, 3, 3, dtype=torch.float64, device=dev)               # Mandel basis of symmetric matrices
        for i in range(3):
            B[i, i, i] = 1.0
        for q, (i, j) in enumerate(((1, 2), (0, 2), (0, 1))):
            B[3 + q, i, j] = B[3 + q, j, i] = math.sqrt(0.5)
        self.B = B

    def local(self, x, Q, hess, model):
        mu, lam = self.mu, self.lam
        F = torch.einsum("kai,kaj->kij", x[self.T], self.G)
        A = torch.einsum("kpi,kpj->kij", Q, F)
        S = 0.5 * (A + A.transpose(1, 2))
        eye = torch.eye(3, dtype=S.dtype, device=S.device)
        D = S - eye
        I6 = torch.eye(6, dtype=S.dtype, device=S.device)
        if model != "snh":
            lam = lam if model == "corot" else 0.0
            tr = torch.einsum("kii->k", D)
            psi = mu * (D * D).sum((1, 2)) + 0.5 * lam * tr * tr
            sig = 2 * mu * D + lam * tr[:, None, None] * eye
            tv = torch.einsum("pii->p", self.B)
            H = (2 * mu * I6 + lam * torch.outer(tv, tv)).expand(len(S), 6, 6) if hess else None
            return S, psi, sig, H
        J = torch.linalg.det(S)
        cof = torch.stack([torch.linalg.cross(S[:, 1], S[:, 2]), torch.linalg.cross(S[:, 2], S[:, 0]),
                           torch.linalg.cross(S[:, 0], S[:, 1])], dim=1)
        psi = 0.5 * mu * ((S * S).sum((1, 2)) - 3.0) - mu * (J - 1) + 0.5 * (lam + mu) * (J - 1) ** 2
        k = (lam + mu) * (J - 1) - mu
        sig = mu * S + k[:, None, None] * cof
        if not hess:
            return S, psi, sig, None
        # second derivative of det: d cof(S)[B] is the polarised cofactor
        cb = []
        for q in range(6):
            M = self.B[q].expand_as(S)
            rows = [torch.linalg.cross(S[:, i], M[:, j]) + torch.linalg.cross(M[:, i], S[:, j])
                    for i, j in ((1, 2), (2, 0), (0, 1))]
            cb.append(torch.einsum("pij,kij->kp", self.B, torch.stack(rows, dim=1)))
        j6 = torch.einsum("pij,kij->kp", self.B, cof)
        H = mu * I6 + k[:, None, None] * torch.stack(cb, dim=2) + (lam + mu) * j6[:, :, None] * j6[:, None, :]
        out = []
        for h in (0.5 * (H + H.transpose(1, 2))).split(30000):      # batches that the eigensolver takes
            w, V = torch.linalg.eigh(h)
            out.append((V * w.abs().clamp_min(1e-6 * mu)[:, None, :]) @ V.transpose(1, 2))
        return S, psi, sig, torch.cat(out)

    def energy_grad(self, x, Q, xp, model, hess=False):
        S, psi, sig, H = self.local(x, Q, hess, model)
        E = (self.vol * psi).sum()
        f = torch.einsum("k,kip,kpj,kaj->kai", self.vol, Q, sig, self.G)
        g = torch.zeros_like(x).index_add_(0, self.T.reshape(-1), f.reshape(-1, 3))
        if self.force is not None:
            E, g = E - (self.force * x).sum(), g - self.force
        if self.ks is not None:
            d = x[self.pins] - xp
            E = E + 0.5 * self.ks * (d * d).sum()
            g[self.pins] += self.ks * d
        else:
            g[self.pins] = 0.0
        K = None
        if hess:
            # stretch of a unit move of vertex a along axis i: sym(Q[i, :] outer G_a) in the Mandel basis
            M = torch.einsum("pij,kci,kaj->kpac", self.B, Q, self.G).reshape(len(S), 6, 12)
            K = self.vol[:, None, None] * (M.transpose(1, 2) @ H @ M)
        return E, g, K, S, sig

    def step(self, K, g, tol):
        """dx of K dx = -g to the relative residual tol."""
        n, idx = len(g), self.T.reshape(-1)
        D = torch.zeros(n, 3, 3, dtype=g.dtype, device=g.device)
        Kb = K.reshape(-1, 4, 3, 4, 3)
        D.index_add_(0, idx, torch.stack([Kb[:, a, :, a, :] for a in range(4)], dim=1).reshape(-1, 3, 3))
        if self.ks is not None:
            D[self.pins] += self.ks * torch.eye(3, dtype=g.dtype, device=g.device)
        Di = torch.linalg.inv(D)

        def mul(p):
            y = (K @ p[self.T].reshape(-1, 12, 1)).reshape(-1, 3)
            y = torch.zeros_like(p).index_add_(0, idx, y)
            if self.ks is not None:
                y[self.pins] += self.ks * p[self.pins]
            else:
                y[self.pins] = 0.0
            return y

        def pre(v):
            z = (Di @ v[:, :, None])[:, :, 0]
            if self.ks is None:
                z[self.pins] = 0.0
            return z

        dx, r = torch.zeros_like(g), -g
        z = pre(r)
        p, rz, r0 = z, (r * z).sum(), float(r.norm())
        for it in range(4000):
            if it % 50 == 0 and float(r.norm()) <= tol * r0:
                break
            q = mul(p)
            al = rz / (p * q).sum()
            dx, r = dx + al * p, r - al * q
            z = pre(r)
            rz, old = (r * z).sum(), rz
            p = z + (rz / old) * p
        return dx

    def solve(self, pose):
        W = torch.as_tensor(np.array(pose)).to(self.X).reshape(-1, 3, 4)
        Q = W[:, :, :3][self.cluster]
        place = lambda v, h: torch.einsum("vij,vj->vi", W[h][:, :, :3], v) + W[h][:, :, 3]  # noqa: E731
        x, xp = place(self.X, self.vhandle), place(self.X[self.pins], self.ph)
        x[self.pins] = xp
        if self.model == "snh":      # one co-rotational step first: the rigid guess tears cluster borders
            E, g, K, _, _ = self.energy_grad(x, Q, xp, "corot", True)
            x = x + self.step(K, g, 1e-6)
        g0 = None
        for it in range(30):
            E, g, K, S, sig = self.energy_grad(x, Q, xp, self.model, True)
            gn = float(g.norm())
            g0 = gn if g0 is None else g0
            if gn <= 1e-11 * g0 or (it > 0 and gn > 0.5 * last and gn < 1e-8 * g0):
                break
            last = gn
            dx = self.step(K, g, 1e-7 if self.model != "snh" else 1e-5)
            a, slope = 1.0, float((g * dx).sum())
            while self.model == "snh" and a > 1e-4 and -slope > 1e-10 * abs(float(E)) and \
                    float(self.energy_grad(x + a * dx, Q, xp, self.model)[0]) > float(E) + 1e-4 * a * slope:
                a *= 0.5
            x = x + a * dx
        s6 = torch.stack([S[:, 0, 0], S[:, 1, 1], S[:, 2, 2], S[:, 1, 2], S[:, 0, 2], S[:, 0, 1]], dim=1)
        return x, float(E), s6, (Q @ sig).reshape(-1, 9)
