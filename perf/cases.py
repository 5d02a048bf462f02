"""The work a program has this library do, as cases that can be timed and checked.

Each case is one call pattern of a user's program on a cloth of 1 m (longer
side) with the constants of the 32 x 32 reference cloth scaled to its spacing:

* frame:    advance a running simulation by a few steps, with the normals of a
            rendered frame where asked (the state stays on the GPU);
* host:     a state from host memory, some steps, the state back to host memory;
* batch:    many cloths advanced together, every cloth's state read at the end;
* rollout:  a training step: steps forward from a fixed start, a loss on the
            final positions, gradients for every spring and the start velocities;
* mesh:     a new surface model handed over and its grid read back.

The states are built from the seed in closed form (a cloth draped over a bumpy
sphere, or hanging and blown against one), so a case does not depend on what
the library computed before it.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_2507_11794_gb300 as P
from paper_2507_11794_gb300.rollout import Rollout

DIRS = ((0, 1), (1, 0), (1, 1), (1, -1), (0, 2), (2, 0))  # canonical spring directions (drow, dcol)
TYPE = (0, 0, 1, 1, 2, 2)                                 # structural, shear, bend
DELTA, EPS, RESTITUTION = 1e-4, 1e-7, -0.5


def _case(name, kind, **kw):
    base = {"name": name, "kind": kind, "nx": 32, "ny": 32, "level": 0, "radius": 0.4, "bump": 0.0, "scene": "drape",
            "edges": False, "steps": 1, "substeps": 4, "rate": 1200, "normals": False, "count": 1, "hi": 0,
            "every": 0}
    base.update(kw)
    return base


def listed():
    return [
        # the smallest call: the 32 x 32 cloth on a 320-triangle sphere, one step of 8 substeps, as an
        # interactive program issues it
        _case("frame_32", "frame", level=2, radius=0.3, substeps=8, rate=600),
        # a rendered frame of a hanging cloth in the wind at the paper's largest collision size (65.5K nodes)
        _case("frame_256_normals", "frame", nx=256, ny=256, scene="hang", radius=0.25, normals=True),
        # the paper's largest cloth (640K nodes), hanging in the wind: 5 steps
        _case("hang_800", "frame", nx=800, ny=800, scene="hang", radius=0.25, steps=5),
        # the 256 x 256 cloth lying on the 81,920-triangle model: contact over most of it
        _case("drape_256", "frame", nx=256, ny=256, level=6, bump=0.1, steps=5),
        # the same with the narrow phase of the paper (cloth edges against the surface), from a given state
        _case("edges_256", "host", nx=256, ny=256, level=6, bump=0.1, edges=True),
        # an odd, ragged cloth pulled over a sphere by its leading row, state in and out through host memory
        _case("pull_190x77", "host", nx=190, ny=77, level=4, radius=0.25, scene="pull", steps=10),
        # the benchmark workload (640K nodes blown against the 81,920-triangle model), state in and out
        _case("contact_800", "host", nx=800, ny=800, level=6, radius=0.25, bump=0.1, scene="hang", steps=4),
        # many small cloths, each on its own model, as a sampler or an environment pool steps them
        _case("batch_30_small", "batch", nx=16, hi=64, count=30, level=3, bump=0.1, substeps=10, steps=8),
        # large cloths of mixed sizes: a state larger than the L2 cache
        _case("batch_12_large", "batch", nx=200, hi=512, count=12, level=5, bump=0.1, substeps=10, steps=5),
        # a training step on the 128 x 128 cloth with per-spring constants over the 5,120-triangle sphere
        _case("rollout_128", "rollout", nx=128, ny=128, level=4, radius=0.3, steps=32, every=8),
        # a larger, ragged cloth over a shorter horizon
        _case("rollout_301x222", "rollout", nx=301, ny=222, level=5, steps=12, every=4),
        # a new 81,920-triangle surface model
        _case("mesh_l6", "mesh", level=6, bump=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "host", "batch", "rollout", "mesh"])
    bump = round(rng.uniform(0.0, 0.12), 3)
    if kind == "mesh":
        c = _case("", kind, level=rng.randint(2, 6), bump=round(rng.uniform(0.0, 0.12), 5))
    elif kind == "batch":
        lo = _log(rng, 16, 200)
        c = _case("", kind, nx=lo, hi=rng.randint(lo, min(512, 4 * lo)), count=rng.randint(4, 12 if lo > 64 else 30),
                  level=rng.randint(2, 5), bump=bump, substeps=10, steps=rng.randint(1, 5))
    elif kind == "rollout":
        nx, ny = _log(rng, 16, 301), _log(rng, 16, 222)
        steps = max(2, min(24, (1 << 19) // (nx * ny)))
        c = _case("", kind, nx=nx, ny=ny, level=rng.choice([0, 2, 3, 4, 5]), steps=steps,
                  every=rng.randint(1, min(16, steps)))
    else:
        scene = rng.choice(["drape", "hang", "pull"] if kind == "host" else ["drape", "hang"])
        level = rng.choice([0, 2, 3, 4, 5, 6]) if scene == "hang" else rng.randint(2, 6)
        edges = kind == "host" and scene == "drape"
        top = 256 if edges else 800
        c = _case("", kind, nx=_log(rng, 24, top), ny=_log(rng, 24, top), level=level, bump=bump, scene=scene,
                  radius=0.25 if scene != "drape" else 0.4, edges=edges, steps=1 if edges else rng.randint(1, 4),
                  normals=kind == "frame" and rng.random() < 0.5)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=None)
def _icosphere(level):
    g = (1.0 + math.sqrt(5.0)) / 2.0
    v = np.array([(s * a, t * b, 0.0) for a, b in ((1.0, g),) for s in (-1, 1) for t in (-1, 1)])
    v = np.concatenate([v, np.roll(v, 1, axis=1), np.roll(v, 2, axis=1)])
    v /= np.linalg.norm(v, axis=1, keepdims=True)
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    near = np.abs(d - np.min(d[d > 1e-9])) < 1e-6
    f = np.array([(i, j, k) if np.dot(np.cross(v[j] - v[i], v[k] - v[i]), v[i]) > 0 else (i, k, j)
                  for i in range(12) for j in range(i + 1, 12) for k in range(j + 1, 12)
                  if near[i, j] and near[j, k] and near[i, k]])
    for _ in range(level):
        n = len(v)
        e = np.sort(np.stack([f, np.roll(f, -1, axis=1)], axis=2).reshape(-1, 2), axis=1)
        key, inv = np.unique(e[:, 0] * n + e[:, 1], return_inverse=True)
        mid = v[key // n] + v[key % n]
        v = np.concatenate([v, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        m = n + inv.reshape(-1, 3)  # midpoints of the edges (0,1), (1,2), (2,0) of each face
        f = np.stack([f[:, 0], m[:, 0], m[:, 2], m[:, 0], f[:, 1], m[:, 1], m[:, 2], m[:, 1], f[:, 2],
                      m[:, 0], m[:, 1], m[:, 2]], axis=1).reshape(-1, 3)
    return v, f.astype(np.int32)


def _bumpy(rng, radius, bump):
    """r(direction) of a bumpy sphere."""
    a, ph = rng.normal(size=(4, 3)) * 3.0, rng.uniform(0, 2 * math.pi, 4)
    return lambda d: radius * (1.0 + bump * sum(np.sin(d @ a[i] + ph[i]) for i in range(4)) / 4.0)


def _scene(c, seed, nx=None, ny=None, salt=0):
    """One cloth's problem: grid, constants, state, pins and surface model."""
    rng = np.random.default_rng([seed, salt])
    nx, ny = nx or c["nx"], ny or c["ny"]
    n = max(nx, ny)
    h = 1.0 / (n - 1)
    scale = (h * 31.0) ** 2
    s = types.SimpleNamespace(nx=nx, ny=ny, total_mass=nx * ny / float(n * n), dt=1.0 / c["rate"],
                              substeps=c["substeps"], gravity=(0.0, -9.81, 0.0), contact_offset=DELTA, mt_eps=EPS,
                              mt_t_min=0.0, restitution=RESTITUTION, pin_velocity=(0.0, 0.0, 0.0),
                              ks=tuple(k * scale for k in (500.0, 250.0, 100.0)), kd=(0.5 * scale,) * 3,
                              ks_spring=None, kd_spring=None, mesh_verts=None, mesh_tris=None,
                              wind=types.SimpleNamespace(amp=0.0, dir=(0.0, 0.0, 1.0), udir=(1.0, 0.0, 0.0), freq=0.0,
                                                         kappa=0.0, phase=0.0))
    R = c["radius"]
    # a model's shape is fixed where the grid itself is what a case returns (its size goes with the shape)
    r_of = _bumpy(np.random.default_rng(7) if c["kind"] == "mesh" else rng, R, c["bump"])
    col, row = np.meshgrid(np.arange(nx) * h, np.arange(ny) * h)
    pin = np.zeros((ny, nx), np.uint8)
    vel = np.zeros((ny, nx, 3))
    wave = np.sin(9.0 * col + rng.uniform(0, 6)) * np.sin(7.0 * row + rng.uniform(0, 6))
    if c["scene"] == "hang":
        # vertical, top row pinned, blown along z against a model at (0, -0.6, 0.3): a billow that
        # reaches just past the model's front, held back where the model is
        centre = np.array([0.0, -0.6, 0.3])
        s.origin, s.du, s.dv = (-0.5, 0.0, 0.0), (h, 0.0, 0.0), (0.0, -h, 0.0)
        s.wind = types.SimpleNamespace(amp=2.0, dir=(0.0, 0.0, 1.0), udir=(math.sqrt(0.5), math.sqrt(0.5), 0.0),
                                       freq=1.0, kappa=4.0 * math.pi, phase=float(rng.uniform(0, 2 * math.pi)))
        x, y = col - 0.5, -row
        front = 0.3 - float(r_of(np.array([[0.0, 0.0, -1.0]]))[0])
        z = (front + 0.003) * np.sin(np.minimum(row / 0.6, 1.0) * math.pi / 2) + 2e-4 * wave * np.minimum(row, 0.1)
        d2 = (x - centre[0]) ** 2 + (y - centre[1]) ** 2
        near = d2 < (0.6 * R) ** 2
        if c["level"]:
            back = np.sqrt(np.where(near, R * R - d2, 1.0))
            q = np.stack([x - centre[0], y - centre[1], -back], axis=2)
            rr = r_of((q / np.linalg.norm(q, axis=2, keepdims=True)).reshape(-1, 3)).reshape(ny, nx)
            surf = centre[2] - np.sqrt(np.where(near, rr * rr - np.minimum(d2, 0.9 * rr * rr), 1.0))
            z = np.where(near, np.minimum(z, surf - rng.uniform(0.5, 4.0, (ny, nx)) * DELTA), z)
        pos = np.stack([x, y, z], axis=2)
        vel[..., 2] = 0.2 * np.minimum(row, 0.5) * (1.0 + 0.5 * wave)
        pin[0] = 1
    else:
        # lying on the model: the cloth's centre on its top, straight down the sides from 57 degrees on
        centre = np.zeros(3)
        w, l = (nx - 1) * h, (ny - 1) * h
        s.origin, s.du, s.dv = (-0.5 * w, R, -0.5 * l), (h, 0.0, 0.0), (0.0, 0.0, h)
        u, v = col - 0.5 * w, row - 0.5 * l
        a = np.maximum(np.hypot(u, v), 1e-9)
        th = np.minimum(a / R, 1.0)
        flat = np.stack([u / a, np.zeros_like(a), v / a], axis=2)
        d = np.sin(th)[..., None] * flat
        d[..., 1] += np.cos(th)
        t = np.cos(th)[..., None] * flat
        t[..., 1] -= np.sin(th)
        gap = rng.uniform(0.5, 4.0, (ny, nx)) * DELTA
        pos = (r_of(d.reshape(-1, 3)).reshape(ny, nx) + gap)[..., None] * d + (a - th * R)[..., None] * t
        vel = -0.3 * d * (1.0 + 0.5 * wave)[..., None]
        if c["scene"] == "pull":
            pin[0] = 1
            s.pin_velocity = (0.5, 0.0, 0.0)
        else:
            pin[0, 0] = pin[0, -1] = pin[-1, 0] = pin[-1, -1] = 1
    vel[pin > 0] = 0.0
    s.init_pos = pos.reshape(-1, 3).astype(np.float32)
    s.init_vel = vel.reshape(-1, 3).astype(np.float32)
    s.pinned = pin.reshape(-1)
    if c["level"]:
        mv, mt = _icosphere(c["level"])
        s.mesh_verts = (mv * r_of(mv)[:, None] + centre).astype(np.float32)
        s.mesh_tris = np.roll(mt, int(rng.integers(1, len(mt))), axis=0) if c["kind"] == "mesh" else mt
    if c["kind"] == "rollout":
        typ = np.broadcast_to(np.asarray(TYPE), (ny, nx, 6))[_exists(nx, ny)]
        s.ks_spring = (np.asarray(s.ks)[typ] * rng.uniform(0.8, 1.2, typ.size)).astype(np.float32)
        s.kd_spring = (np.asarray(s.kd)[typ] * rng.uniform(0.8, 1.2, typ.size)).astype(np.float32)
        s.target = (s.init_pos + rng.normal(0.0, 0.02, s.init_pos.shape)).astype(np.float32)
    return s


def _exists(nx, ny):
    """[row, col, direction]: whether the node has that spring."""
    r, q = np.arange(ny)[:, None, None], np.arange(nx)[None, :, None]
    dr, dc = np.asarray(DIRS).T
    return (r + dr < ny) & (q + dc < nx) & (q + dc >= 0)


def _members(c, seed):
    """The cloths of a batch: sides spread evenly over the logarithm of [nx, hi]."""
    k = c["count"]
    sides = [round(c["nx"] * (c["hi"] / c["nx"]) ** (i / max(k - 1, 1))) for i in range(k)]
    return [_scene(dict(c, level=max(2, c["level"] - i % 3)), seed, m, m, 1 + i) for i, m in enumerate(sides)]


def _pinned_copy(a):
    return torch.from_numpy(a).pin_memory().numpy()


def prepare(case, seed):
    c, st = case, types.SimpleNamespace(case=case)
    if c["kind"] == "batch":
        st.batch = P.ClothBatch(_members(c, seed))
        return st
    if c["kind"] == "mesh":
        st.sc = _scene(c, seed)
        st.cloth = P.Cloth(st.sc, mesh=False)
        return st
    st.sc = _scene(c, seed)
    st.cloth = P.Cloth(st.sc, flags=P.capi.CLOTH_FLAG_EDGE_COLLISION if c["edges"] else 0)
    if c["kind"] == "rollout":
        st.rollout = Rollout(st.cloth, c["steps"], c["every"])
        st.args = [torch.tensor(a, device="cuda", requires_grad=True)
                   for a in (st.sc.ks_spring, st.sc.kd_spring, st.sc.init_vel)]
        st.target = torch.tensor(st.sc.target, device="cuda")
    elif c["kind"] == "host":
        st.pos, st.vel = _pinned_copy(st.sc.init_pos), _pinned_copy(st.sc.init_vel)
        st.pos_out, st.vel_out = _pinned_copy(st.sc.init_pos), _pinned_copy(st.sc.init_vel)
    st.views = {}
    return st


class _Planes:
    """Three planes of a cloth's state for torch, which keeps this object, and so the cloth, while it has them."""

    def __init__(self, cloth, ptr, shape, strides):
        self.cloth = cloth
        self.__cuda_array_interface__ = {"shape": shape, "strides": strides, "typestr": "<f4", "data": (ptr, False),
                                         "version": 3}


def _state(st):
    """The cloth's current positions and velocities as [3][row][col] views of its planes."""
    i = st.cloth.info()
    key = i.pos_planes[0]
    if key not in st.views:
        st.views[key] = [torch.as_tensor(_Planes(st.cloth, q, (3, i.ny, i.nx),
                                                 (4 * i.plane_stride, 4 * i.row_pitch, 4)), device="cuda")
                         for q in (i.pos_planes[0], i.vel_planes[0])]
    return st.views[key]


def run(st):
    c = st.case
    if c["kind"] == "mesh":
        st.cloth.set_mesh(st.sc.mesh_verts, st.sc.mesh_tris)
        return st.cloth.grid()
    if c["kind"] == "batch":
        st.batch.step(c["steps"])
        return [st.batch.read(i) for i in range(c["count"])]
    if c["kind"] == "rollout":
        pos, vel = st.rollout(*st.args)
        loss = ((pos - st.target) ** 2).sum(1).mean()
        return [pos.detach(), vel.detach(), *torch.autograd.grad(loss, st.args)]
    if c["kind"] == "host":
        st.cloth.set_state(st.pos, st.vel)
        st.cloth.step(c["steps"])
        return st.cloth.read(out_pos=st.pos_out, out_vel=st.vel_out)
    st.cloth.step(c["steps"])
    out = list(_state(st))
    if c["normals"]:
        out.append(st.cloth.normals())
    return out


def work(case):
    c = case
    tris = 20 * 4 ** c["level"] if c["level"] else 0
    if c["kind"] == "mesh":
        # vertices and triangles in, triangle records (48 B) and about three ids each out
        return {"bytes": tris * (6 + 12 + 48 + 12), "flops": 20 * tris}
    if c["kind"] == "batch":
        k = c["count"]
        nodes = sum(round(c["nx"] * (c["hi"] / c["nx"]) ** (i / max(k - 1, 1))) ** 2 for i in range(k))
        tris = sum(20 * 4 ** max(2, c["level"] - i % 3) for i in range(k))
    else:
        nodes = c["nx"] * c["ny"]
    # one substep of a node: six springs of 38 operations (force, both ends' sums) and 24 for the integration
    flops = 252.0 * nodes * c["steps"] * c["substeps"]
    state = 24 * nodes  # positions and velocities once
    if c["kind"] == "rollout":
        # forward, and a reverse pass of about twice its operations; six springs' ks, kd in and their gradients
        # out, the target in and the start velocities' gradient out
        return {"bytes": 2 * state + (96 + 24) * nodes + 36 * tris, "flops": 3 * flops}
    more = 12 * nodes if c["normals"] else 0
    return {"bytes": 2 * state + more + 36 * tris, "flops": flops + (60 * nodes if c["normals"] else 0)}


# ------------------------------------------------------- the same in 64 bits

def _dot(a, b):
    return (a * b).sum(0)


def _segment_hits(S, E, tri):
    """Hits of the segments S -> E ([n, 3]) with the triangles (v0, e1, e2): (segment, t, r[segment])
    by the extended Moller-Trumbore test.  Pairs come from a hash of the triangles' centres."""
    v0, e1, e2 = tri
    d = E - S
    L = d.norm(dim=1)
    r = d / L.clamp_min(1e-300)[:, None]
    with torch.no_grad():
        ctr = v0 + (e1 + e2) / 3.0
        reach = torch.stack([(p - ctr).norm(dim=1).max() for p in (v0, v0 + e1, v0 + e2)]).max()
        H = float(reach + 0.5 * L.max()) * 1.001 + 1e-9
        lo = ctr.min(dim=0).values - 2 * H
        dim = ((ctr.max(dim=0).values - lo) / H).long() + 3
        cell = ((ctr - lo) / H).long()
        key = (cell[:, 2] * dim[1] + cell[:, 1]) * dim[0] + cell[:, 0]
        key, order = key.sort()
        mid = ((0.5 * (S + E) - lo) / H).floor().long()
        pairs = []
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                q = mid + torch.tensor([0, dy, dz], device=S.device)
                ok = ((q[:, 1:] >= 0) & (q[:, 1:] < dim[1:])).all(1) & (q[:, 0] >= -1) & (q[:, 0] <= dim[0]) & (L >= EPS)
                base = (q[:, 2] * dim[1] + q[:, 1]) * dim[0]
                a = torch.searchsorted(key, base + (q[:, 0] - 1).clamp_min(0))
                b = torch.searchsorted(key, base + (q[:, 0] + 1).clamp(max=int(dim[0]) - 1), right=True)
                cnt = torch.where(ok, (b - a).clamp_min(0), 0)
                seg = torch.repeat_interleave(torch.arange(len(S), device=S.device), cnt)
                k = torch.arange(len(seg), device=S.device) - (cnt.cumsum(0) - cnt)[seg] + a[seg]
                pairs.append((seg, order[k]))
        seg, t = (torch.cat(x) for x in zip(*pairs))

        def test(seg, t):
            h = torch.linalg.cross(r[seg], e2[t])
            a = (e1[t] * h).sum(1)
            f = 1.0 / torch.where(a.abs() < EPS, torch.ones_like(a), a)
            q0 = S[seg] - v0[t]
            u = f * (q0 * h).sum(1)
            q = torch.linalg.cross(q0, e1[t])
            return a, u, f * (r[seg] * q).sum(1), f * (e2[t] * q).sum(1)

        keep = []
        for i in range(0, len(seg), 1 << 22):
            a, u, v, th = test(seg[i:i + (1 << 22)], t[i:i + (1 << 22)])
            keep.append((a.abs() >= EPS) & (u >= 0) & (u <= 1) & (v >= 0) & (u + v <= 1) & (th > 0) &
                        (th < L[seg[i:i + (1 << 22)]]))
        keep = torch.cat(keep) if keep else torch.zeros(0, dtype=torch.bool, device=S.device)
        seg, t = seg[keep], t[keep]
    # t again, with its derivatives where the caller wants them
    h = torch.linalg.cross(r[seg], e2[t])
    q = torch.linalg.cross(S[seg] - v0[t], e1[t])
    th = (e2[t] * q).sum(1) / (e1[t] * h).sum(1)
    return seg, th, r


def _simulate(sc, substeps, x, v, ks=None, kd=None, edges=False):
    """`substeps` substeps in 64 bits from x, v ([3, ny, nx]); ks, kd per spring in canonical order, or per type."""
    f32 = lambda a: torch.tensor(np.asarray(a, np.float32), device="cuda").double()  # noqa: E731
    ny, nx = sc.ny, sc.nx
    du, dv = np.asarray(sc.du, np.float32).astype(float), np.asarray(sc.dv, np.float32).astype(float)
    dt = float(np.float32(sc.dt)) / sc.substeps
    m = float(np.float32(sc.total_mass)) / (nx * ny)
    g = f32(sc.gravity)[:, None, None]
    pin = torch.tensor(sc.pinned.reshape(ny, nx) > 0, device="cuda")
    pv = f32(sc.pin_velocity)[:, None, None]
    w = sc.wind
    amp, kap, fr, ph = (float(np.float32(a)) for a in (w.amp, w.kappa, w.freq, w.phase))
    u32 = np.asarray(w.udir, np.float32).astype(float)
    rows, cols = np.arange(ny)[:, None], np.arange(nx)[None, :]
    phase = torch.tensor(kap * (u32 @ np.asarray(sc.origin, np.float32).astype(float) + rows * (u32 @ dv) +
                                cols * (u32 @ du)) + ph, device="cuda")
    wdir = f32(w.dir)[:, None, None]
    exists = _exists(nx, ny)
    index = np.zeros(exists.shape, np.int64)
    index[exists] = np.arange(int(exists.sum()))
    tri = None
    if sc.mesh_tris is not None:
        V = f32(sc.mesh_verts)
        T = torch.tensor(sc.mesh_tris.astype(np.int64), device="cuda")
        tri = (V[T[:, 0]], V[T[:, 1]] - V[T[:, 0]], V[T[:, 2]] - V[T[:, 0]])
        lo, hi = V.min(0).values - 1e-3, V.max(0).values + 1e-3
    delta, rest = float(np.float32(DELTA)), float(np.float32(RESTITUTION))
    free = (~pin).reshape(-1)
    springs = []
    for k, (dr, dc) in enumerate(DIRS):
        if ny <= dr or nx <= abs(dc):
            continue
        a0, a1 = max(0, -dc), nx - max(0, dc)
        A = (slice(None), slice(0, ny - dr), slice(a0, a1))
        B = (slice(None), slice(dr, ny), slice(a0 + dc, a1 + dc))
        L0 = float(np.linalg.norm(dc * du + dr * dv))
        if ks is None:
            K, D = float(np.float32(sc.ks[TYPE[k]])), float(np.float32(sc.kd[TYPE[k]]))
        else:
            at = torch.tensor(np.ascontiguousarray(index[..., k][A[1:]]), device="cuda")
            K, D = ks[at], kd[at]
        springs.append((A, B, (a0, nx - a1, 0, dr), (a0 + dc, nx - a1 - dc, dr, 0), L0, K, D))
    pad = torch.nn.functional.pad
    for k in range(substeps):
        F = torch.zeros_like(x)
        for A, B, pa, pb, L0, K, D in springs:
            d, e = x[B] - x[A], v[B] - v[A]
            l = _dot(d, d).sqrt()
            f = (K * (l - L0) + D * _dot(e, d) / l) / l * d
            F = F + pad(f, pa) - pad(f, pb)
        acc = F / m + g
        if amp:
            acc = acc + amp * wdir * torch.sin(2 * math.pi * fr * (k * dt) + phase)
        vs = torch.where(pin, pv, v + dt * acc)
        xs = x + dt * vs
        x0, x, v = x, xs, vs
        if tri is None:
            continue
        S0 = x0.reshape(3, -1).T
        E0 = xs.reshape(3, -1).T
        if not edges:
            near = ((torch.maximum(S0, E0) >= lo) & (torch.minimum(S0, E0) <= hi)).all(1) & free
            i = near.nonzero()[:, 0]
            if not len(i):
                continue
            seg, th, r = _segment_hits(S0[i], E0[i], tri)
            K = torch.zeros(len(i), dtype=x.dtype, device="cuda").index_add(0, seg, torch.ones_like(th))
            mean = torch.zeros_like(K).index_add(0, seg, (th - delta).clamp_min(0)) / K.clamp_min(1)
            hit = K > 0
            new = S0[i] + mean[:, None] * r
            j, new = i[hit], new[hit]
        else:
            ids = torch.arange(ny * nx, device="cuda").reshape(ny, nx)
            sums, count = torch.zeros_like(S0), torch.zeros(ny * nx, dtype=x.dtype, device="cuda")
            for (dr, dc), reach in (((0, 1), ((0, 0), (0, 1), (1, 1), (-1, 0))), ((1, 0), ((0, 0), (1, 0), (1, 1), (0, -1))),
                                    ((1, 1), ((0, 0), (1, 1), (1, 0), (0, 1)))):
                a = ids[:ny - dr, :nx - dc].reshape(-1)
                b = ids[dr:, dc:].reshape(-1)
                near = ((torch.maximum(E0[a], E0[b]) >= lo) & (torch.minimum(E0[a], E0[b]) <= hi)).all(1)
                a, b = a[near], b[near]
                if not len(a):
                    continue
                seg, th, r = _segment_hits(E0[a], E0[b], tri)
                p = E0[a][seg] + th[:, None] * r[seg]
                for rr, cc in reach:
                    y, z = a[seg] // nx + rr, a[seg] % nx + cc
                    ok = (y >= 0) & (y < ny) & (z >= 0) & (z < nx)
                    j = (y * nx + z)[ok]
                    q = p[ok] - S0[j]
                    l = q.norm(dim=1, keepdim=True)
                    sums.index_add_(0, j, (l - delta).clamp_min(0) * q / l.clamp_min(1e-300))
                    count.index_add_(0, j, torch.ones_like(l[:, 0]))
            j = ((count > 0) & free).nonzero()[:, 0]
            new = S0[j] + sums[j] / count[j][:, None]
        x = x.reshape(3, -1).index_copy(1, j, new.T).reshape(3, ny, nx)
        v = v.reshape(3, -1).index_copy(1, j, rest * v.reshape(3, -1)[:, j]).reshape(3, ny, nx)
    return x, v


def _normals(x):
    a, b, c, d = x[:, :-1, :-1], x[:, 1:, :-1], x[:, 1:, 1:], x[:, :-1, 1:]
    f, g = torch.linalg.cross(b - a, c - a, dim=0), torch.linalg.cross(c - a, d - a, dim=0)
    pad = torch.nn.functional.pad
    n = (pad(f + g, (0, 1, 0, 1)) + pad(f, (0, 1, 1, 0)) + pad(f + g, (1, 0, 1, 0)) + pad(g, (1, 0, 0, 1)))
    return n / n.norm(dim=0, keepdim=True).clamp_min(1e-300)


def _planes(a, sc):
    return torch.tensor(a, device="cuda").double().T.reshape(3, sc.ny, sc.nx).contiguous()


def _rows(x):
    return x.reshape(3, -1).T.contiguous()


def exact(case, seed):
    c = case
    if c["kind"] == "mesh":
        return None  # whole numbers
    n = c["steps"] * c["substeps"]
    if c["kind"] == "batch":
        out = []
        for sc in _members(c, seed):
            out.append([_rows(q) for q in _simulate(sc, n, _planes(sc.init_pos, sc), _planes(sc.init_vel, sc))])
        return out
    sc = _scene(c, seed)
    x, v = _planes(sc.init_pos, sc), _planes(sc.init_vel, sc)
    if c["kind"] == "rollout":
        ks, kd = (torch.tensor(a, device="cuda").double().requires_grad_() for a in (sc.ks_spring, sc.kd_spring))
        v0 = torch.tensor(sc.init_vel, device="cuda").double().requires_grad_()
        x, v = _simulate(sc, n, x, v0.T.reshape(3, sc.ny, sc.nx), ks, kd)
        pos, vel = _rows(x), _rows(v)
        loss = ((pos - torch.tensor(sc.target, device="cuda").double()) ** 2).sum(1).mean()
        return [pos.detach(), vel.detach(), *torch.autograd.grad(loss, (ks, kd, v0))]
    x, v = _simulate(sc, n, x, v, edges=c["edges"])
    if c["kind"] == "host":
        return [_rows(x), _rows(v)]
    return [x, v] + ([_rows(_normals(x))] if c["normals"] else [])
