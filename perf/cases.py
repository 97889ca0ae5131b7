"""Performance cases of the LiDAR ray caster and its mesh pipeline.

Each case is one call sequence that a program using this package makes, at the
sizes of the package's own workloads:

  cast       fgl.cast: one scan of one or a few environments (a single robot)
  batched    fgl.cast_batched: one step of many environments on one scene
  mixed      fgl.cast_batched over several scenes, sensors, BVH widths and
             minimum ranges (a heterogeneous fleet)
  instances  fgl.cast_batched with moving rigid instances and return points
  host       fgl.cast_batched_host: host poses in, page-locked host returns out
  lbvh       Lbvh.rebuild + Lbvh.cast: a mesh that moves every frame
  density    fgl.gaussian_density with its masks
  mesh       fgl.mesh_from_gaussians: Gaussians to a triangle mesh
  surface    fgl.mesh_from_surface: denoising, TSDF, marching tetrahedra
  effects    fgl.apply_sensor_effects: dropout and range noise on one step

Scenes, Gaussians, poses and surface grids are procedural and follow the seed.
"""

import math

import numpy as np
import torch

import paper_2509_17390_gb300 as fgl

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # the smallest call: one scan of a bare room (latency, one launch)
        {"name": "scan_tiny", "kind": "cast", "envs": 1, "beams": 16, "az": 360, "tris": 108, "range": 100.0},
        # one high-resolution scan of a cluttered indoor scene
        {"name": "scan_indoor", "kind": "cast", "envs": 1, "beams": 32, "az": 1800, "tris": 1_000_000, "range": 120.0},
        # one step of a small training run
        {"name": "step_64", "kind": "batched", "envs": 64, "beams": 16, "az": 360, "tris": 250_000, "range": 120.0,
         "graph": False},
        # one step of a large training run, replayed from a graph: the package's headline workload
        {"name": "walk_4096", "kind": "batched", "envs": 4096, "beams": 16, "az": 360, "tris": 1_000_000,
         "range": 120.0, "graph": True},
        # a fleet on four finely tessellated rooms, with every sensor class
        {"name": "fleet", "kind": "mixed", "envs": 128, "voxel": 0.03, "range": 30.0},
        # a step with four moving objects around each robot, returns as points
        {"name": "moving_objects", "kind": "instances", "envs": 1024, "beams": 16, "az": 360, "tris": 500_000,
         "objects": 4, "range": 120.0},
        # a simulator on the host: poses in and ranges out over the host link
        {"name": "host_1024", "kind": "host", "envs": 1024, "beams": 16, "az": 360, "tris": 250_000, "range": 120.0},
        # a deforming scene: the tree rebuilt, then one scan of each robot
        {"name": "moving_mesh", "kind": "lbvh", "envs": 512, "beams": 16, "az": 360, "tris": 500_000, "range": 120.0},
        # occupancy of a room of Gaussians at a fine grid
        {"name": "occupancy", "kind": "density", "gaussians": 720_000, "room": 5.0, "voxel": 0.025, "tile": 8},
        # a small asset converted as a whole
        {"name": "asset_mesh", "kind": "mesh", "gaussians": 85_000, "room": 2.5, "voxel": 0.05},
        # a large surface grid to a mesh with normals
        {"name": "surface_mesh", "kind": "surface", "room": 6.0, "voxel": 0.02, "denoise": True, "normals": True},
        # sensor effects on one step's returns
        {"name": "effects_1024", "kind": "effects", "envs": 1024, "beams": 16, "az": 360, "drop": 0.05,
         "sigma0": 0.01, "sigma1": 0.001},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cast", "batched", "batched", "mixed", "instances", "host", "lbvh", "density", "mesh",
                       "surface", "effects"])
    c = {"kind": kind}
    if kind in ("cast", "batched", "instances", "host", "lbvh", "effects"):
        c["beams"] = rng.choice([16, 32, 64, 128]) if rng.random() < 0.6 else rng.randint(5, 100)
        c["az"] = rng.choice([360, 512, 1024, 1800, 2048]) if rng.random() < 0.6 else rng.randint(91, 2048)
        most = {"cast": 8, "batched": 4096, "instances": 1024, "host": 1024, "lbvh": 512, "effects": 4096}[kind]
        rays = {"cast": 500_000, "batched": 20_000_000, "instances": 5_000_000, "host": 5_000_000,
                "lbvh": 3_000_000, "effects": 20_000_000}[kind]
        c["envs"] = _log_int(rng, 1, max(1, min(most, rays // (c["beams"] * c["az"]))))
    if kind in ("cast", "batched", "instances", "host", "lbvh"):
        most = 1_000_000 if kind in ("cast", "batched") else 500_000
        c["tris"] = _log_int(rng, 300, most)
        c["range"] = rng.choice([10.0, 30.0, 100.0, 120.0])
    if kind == "batched":
        c["graph"] = rng.random() < 0.5
    if kind == "mixed":
        c.update(envs=_log_int(rng, 4, 128), voxel=round(rng.uniform(0.03, 0.08), 3), range=30.0)
    if kind == "instances":
        c["objects"] = rng.randint(1, 6)
    if kind == "density":
        c.update(gaussians=_log_int(rng, 3_000, 400_000), room=round(rng.uniform(1.5, 4.0), 2),
                 voxel=round(rng.uniform(0.03, 0.06), 4), tile=rng.choice([8, 8, 4]))
    if kind == "mesh":
        c.update(gaussians=_log_int(rng, 3_000, 200_000), room=round(rng.uniform(1.5, 4.0), 2),
                 voxel=round(rng.uniform(0.035, 0.06), 4))
    if kind == "surface":
        c.update(room=round(rng.uniform(1.5, 6.0), 2), voxel=round(rng.uniform(0.02, 0.06), 4),
                 denoise=rng.random() < 0.7, normals=rng.random() < 0.5)
    if kind == "effects":
        c.update(drop=round(rng.uniform(0.0, 0.2), 3), sigma0=rng.choice([0.0, 0.01, 0.03]), sigma1=rng.choice([0.0, 0.001]))
    return c


# ---------------------------------------------------------------------------
# procedural meshes
# ---------------------------------------------------------------------------


def _indexed(soup):
    """Triangle soup [n, 3, 3] to (verts, tris) with equal corners shared."""
    v, inv = np.unique(soup.reshape(-1, 3), axis=0, return_inverse=True)
    return v, inv.reshape(-1, 3).astype(np.int64)


def _unit_box(n):
    """The surface of [0, 1]^3, every face split n x n, with shared corners."""
    g = np.arange(n + 1)
    quads = []
    for a in range(3):
        b, c = (a + 1) % 3, (a + 2) % 3
        for side in (0, n):
            p = np.zeros((n + 1, n + 1, 3), np.int64)
            p[..., a] = side
            p[..., b] = g[:, None]
            p[..., c] = g[None, :]
            q = [p[:-1, :-1], p[1:, :-1], p[1:, 1:], p[:-1, 1:]]
            order = ((0, 1, 2), (0, 2, 3)) if side else ((0, 2, 1), (0, 3, 2))
            quads += [np.stack([q[i] for i in o], -2).reshape(-1, 3) for o in order]
    soup = np.concatenate(quads)
    key, inv = np.unique((soup[:, 0] * (n + 1) + soup[:, 1]) * (n + 1) + soup[:, 2], return_inverse=True)
    v = np.stack([key // (n + 1) ** 2, key // (n + 1) % (n + 1), key % (n + 1)], 1) / n
    return v, inv.reshape(-1, 3)


def _unit_sphere(level):
    """An icosphere of 20 * 4^level triangles."""
    g = (1 + 5 ** 0.5) / 2
    v = np.array([(-1, g, 0), (1, g, 0), (-1, -g, 0), (1, -g, 0), (0, -1, g), (0, 1, g), (0, -1, -g), (0, 1, -g),
                  (g, 0, -1), (g, 0, 1), (-g, 0, -1), (-g, 0, 1)], float)
    f = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                  (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5),
                  (2, 4, 11), (6, 2, 10), (8, 6, 7), (9, 8, 1)])
    s = (v / np.linalg.norm(v, axis=1, keepdims=True))[f]
    for _ in range(level):
        a, b, c = s[:, 0], s[:, 1], s[:, 2]
        ab, bc, ca = (m / np.linalg.norm(m, axis=1, keepdims=True) for m in (a + b, b + c, c + a))
        s = np.concatenate([np.stack(t, 1) for t in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return _indexed(s)


def _placed(unit, offset, size):
    """Copies of a unit mesh, copy k at offset[k] + size[k] * unit."""
    uv, ut = unit
    v = offset[:, None, :] + size[:, None, :] * uv[None]
    t = ut[None] + (np.arange(len(offset)) * len(uv))[:, None, None]
    return v.reshape(-1, 3), t.reshape(-1, 3)


def _merged(parts):
    at = np.cumsum([0] + [len(v) for v, _ in parts])
    v = np.concatenate([p[0] for p in parts]).astype(np.float32)
    t = np.concatenate([p[1] + a for p, a in zip(parts, at)]).astype(np.int32)
    return np.ascontiguousarray(v), np.ascontiguousarray(t)


def _indoor(rng, tris):
    """About `tris` triangles: a closed room with boxes (tris <= 2,000), or
    cluttered with icospheres and subdivided boxes in equal object counts of
    the 20 x 15 x 4 m scene.  Returns (verts, tris, room, objects), objects
    the boxes' (lo, hi) rows that robots stay out of."""
    small = tris <= 2_000
    room = np.array([10.0, 8.0, 3.0]) if small else np.array([20.0, 15.0, 4.0])
    parts = [_placed(_unit_box(1), np.zeros((1, 3)), room[None])]
    if small:
        n = max(1, (tris - 12) // 12)
        size = rng.uniform(0.2, 1.5, (n, 3))
        lo = rng.uniform(0, 1, (n, 3)) * (room - size)
        lo[:, 2] = 0.0
        parts.append(_placed(_unit_box(1), lo, size))
        return (*_merged(parts), room, np.concatenate([lo, lo + size], 1))
    ns, nb = max(1, int(0.002 * tris)), max(1, int(0.000834 * tris))
    r = np.clip(0.3 * np.exp(0.5 * rng.standard_normal(ns)), 0.05, 1.5)[:, None]
    c = r + rng.uniform(0, 1, (ns, 3)) * (room - 2 * r)
    size = rng.uniform(0.2, 1.5, (nb, 3))
    lo = rng.uniform(0, 1, (nb, 3)) * (room - size)
    parts += [_placed(_unit_sphere(2), c, np.repeat(r, 3, 1)), _placed(_unit_box(6), lo, size)]
    return (*_merged(parts), room, np.concatenate([np.concatenate([c - r, c + r], 1), np.concatenate([lo, lo + size], 1)]))


def _scanned_room(rng, room, voxel):
    """A room as a level-set mesh of spacing `voxel` has it: an uneven floor,
    walls and objects of triangles of about that edge."""
    room = np.asarray(room, float)
    parts, objects = [], []
    shell = _unit_box(max(1, int(round(room.max() / voxel))))
    v = shell[0] * room
    v = v + rng.uniform(-0.25, 0.25, v.shape) * voxel
    parts.append((v, shell[1]))
    for _ in range(4):
        size = rng.uniform(0.3, 0.25 * room.min() + 0.3, 3)
        lo = np.r_[rng.uniform(0, 1, 2) * (room[:2] - size[:2]), 0.0]
        v, t = _placed(_unit_box(max(1, int(round(size.max() / voxel)))), lo[None], size[None])
        parts.append((v + rng.uniform(-0.25, 0.25, v.shape) * voxel, t))
        objects.append(np.r_[lo, lo + size])
    return (*_merged(parts), room, np.array(objects))


def _poses(rng, n, room, objects, margin=0.3, tilt=0.35):
    """float32 [n, 3, 4] poses at free places of the room: any heading, up to
    `tilt` radians of lean."""
    p, box = np.empty((0, 3)), torch.from_numpy(objects).cuda()
    for _ in range(200):
        q = margin + rng.uniform(0, 1, (max(256, 2 * n), 3)) * (room - 2 * margin)
        x = torch.from_numpy(q).cuda()[:, None]
        inside = ((x > box[:, :3] - 0.05) & (x < box[:, 3:] + 0.05)).all(2).any(1)
        p = np.concatenate([p, q[~inside.cpu().numpy()]])[:n]
        if len(p) == n:
            break
    if len(p) < n:  # nearly no free place: inside an object then
        p = np.concatenate([p, margin + rng.uniform(0, 1, (n - len(p), 3)) * (room - 2 * margin)])
    yaw, lean, way = rng.uniform(0, 2 * np.pi, n), rng.uniform(0, tilt, n), rng.uniform(0, 2 * np.pi, n)
    return np.ascontiguousarray(np.concatenate([_rotations(yaw, lean, way), p[:, :, None]], 2), np.float32)


def _rotations(yaw, lean, way):
    """Rz(yaw) after a turn by `lean` about the horizontal axis at angle `way`."""
    x, y, c, s = np.cos(way), np.sin(way), np.cos(lean), np.sin(lean)
    k, z = 1 - c, np.zeros_like(yaw)
    T = np.stack([np.stack([c + x * x * k, x * y * k, y * s], -1), np.stack([x * y * k, c + y * y * k, -x * s], -1),
                  np.stack([-y * s, x * s, c], -1)], -2)
    Z = np.stack([np.stack([np.cos(yaw), -np.sin(yaw), z], -1), np.stack([np.sin(yaw), np.cos(yaw), z], -1),
                  np.stack([z, z, z + 1], -1)], -2)
    return Z @ T


# beams -> the elevation span of that class of spinning sensor
_SPAN = {16: (-15.0, 15.0), 32: (-16.0, 15.0), 64: (-24.9, 2.0), 128: (-22.5, 22.5)}


def _grid_angles(beams, az):
    lo, hi = _SPAN.get(beams, (-20.0, 15.0))
    E, A = np.meshgrid(np.deg2rad(np.linspace(lo, hi, beams)), 2 * np.pi * np.arange(az) / az, indexing="ij")
    return E.reshape(-1).astype(np.float32), A.reshape(-1).astype(np.float32), beams, az


def _rosette_angles(n, phase):
    """A non-repetitive rose curve of 35 degrees around the forward axis."""
    t = np.arange(n) * 1e-3
    w = 2 * np.pi * 61.0
    rho, psi = np.deg2rad(35.0) * np.sin(w * t + phase), w / ((1 + 5 ** 0.5) / 2) * t
    el, az = np.arcsin(np.sin(rho) * np.sin(psi)), np.arctan2(np.sin(rho) * np.cos(psi), np.cos(rho))
    return el.astype(np.float32), az.astype(np.float32), 1, n


# ---------------------------------------------------------------------------
# procedural Gaussians and surface grids
# ---------------------------------------------------------------------------


def _gaussian_room(rng, n, side):
    """n Gaussians on the floor, walls and furniture of an open-topped room of
    side x 0.8 side x 0.5 side metres."""
    L = side * np.array([1.0, 0.8, 0.5])
    rects = [([0, 0, 0], [L[0], L[1], 0]), ([0, 0, 0], [0, L[1], L[2]]), ([L[0], 0, 0], L), ([0, 0, 0], [L[0], 0, L[2]]),
             ([0, L[1], 0], L)]
    for _ in range(3):
        size = rng.uniform(0.15, 0.3, 3) * side * np.array([1, 1, 0.8])
        lo = np.r_[rng.uniform(0.1, 0.9, 2) * (L[:2] - size[:2]), 0.0]
        for a in range(3):
            for at in (lo[a], lo[a] + size[a]):
                l, h = lo.copy(), lo + size
                l[a] = h[a] = at
                rects.append((l, h))
    lo, hi = np.array([r[0] for r in rects], float), np.array([r[1] for r in rects], float)
    e = np.sort(hi - lo, 1)
    area = e[:, 1] * e[:, 2]
    k = rng.choice(len(rects), n, p=area / area.sum())
    mu = lo[k] + rng.uniform(0, 1, (n, 3)) * (hi[k] - lo[k])
    scale = np.clip(0.045 * np.exp(0.75 * rng.standard_normal((n, 3))), 0.01, 0.2)
    quat = rng.standard_normal((n, 4))
    return [np.ascontiguousarray(a, np.float32) for a in (mu, scale, quat, rng.uniform(0.3, 1.0, n))], L


def _grid(L, voxel, margin):
    return (-margin, -margin, -margin), tuple(int(math.ceil((x + 2 * margin) / voxel)) for x in L)


def _room_grid(case):
    side = case["room"]
    return _grid(side * np.array([1.0, 0.8, 0.5]), case["voxel"], 0.75 if case["kind"] != "density" else 0.3)


def _surface_grid(case, seed):
    """u8 [nz, ny, nx] one-to-two-voxel surfaces of a room with spheres and
    boxes, a few stray voxels among them."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    origin, (nx, ny, nz) = _room_grid(case)
    h, L = case["voxel"], case["room"] * np.array([1.0, 0.8, 0.5])
    ax = [torch.arange(n, device="cuda", dtype=torch.float32) * h + (0.5 * h + origin[0]) for n in (nx, ny, nz)]
    Z, Y, X = ax[2][:, None, None], ax[1][None, :, None], ax[0][None, None, :]

    def box(lo, hi):
        d = [torch.maximum(lo[a] - P, P - hi[a]) for a, P in enumerate((X, Y, Z))]
        return torch.maximum(torch.maximum(d[0], d[1]), d[2])

    d = box((0, 0, 0), (L[0], L[1], 2 * L[2]))
    s = (d.abs() <= 0.75 * h) & (Z <= L[2])
    for _ in range(6):
        size = rng.uniform(0.1, 0.25, 3) * case["room"]
        lo = np.r_[rng.uniform(0.05, 0.95, 2) * (L[:2] - size[:2]), 0.0]
        s |= box(lo, np.minimum(lo + size, L)).abs() <= 0.75 * h
        r = rng.uniform(0.05, 0.12) * case["room"]
        c = r + rng.uniform(0, 1, 3) * (L - 2 * r)
        s |= (((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2).sqrt() - r).abs() <= 0.75 * h
    s |= torch.rand(s.shape, generator=gen, device="cuda") < 2e-4
    return s.to(torch.uint8).contiguous(), origin


# ---------------------------------------------------------------------------
# what a program has in hand
# ---------------------------------------------------------------------------


class _State:
    def __init__(self, **k):
        self.__dict__.update(k)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _ray_inputs(case, seed):
    """The host inputs of a ray-casting case: meshes, angles and poses."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "mixed":
        rooms = [(3.0, 2.5, 1.5), (4.5, 3.5, 2.0), (5.0, 4.0, 2.5), (6.0, 5.0, 3.0)]
        scenes = [_scanned_room(rng, r, case["voxel"]) for r in rooms]
        angles = [_grid_angles(*g) for g in ((16, 360), (16, 2048), (32, 1800), (64, 1024), (128, 512), (128, 2048))]
        angles.append(_rosette_angles(20_000, rng.uniform(0, 6.28)))
        per = [(np.arange((case["envs"] + 3 - k) // 4) * 5 + 2 * k) % len(angles) for k in range(4)]
        items = []
        for k, s in enumerate(scenes):
            for a in np.unique(per[k]):
                near = 0.3 if a % 3 == 2 else 0.0
                items.append((k, int(a), _poses(rng, int(np.sum(per[k] == a)), s[2], s[3], 0.25, 0.05), near))
        return [s[:2] for s in scenes], angles, items
    v, t, room, objects = _indoor(rng, case["tris"])
    P = _poses(rng, case["envs"], room, objects)
    return [(v, t)], [_grid_angles(case["beams"], case["az"])], [(0, 0, P, 0.0)]


def _objects(case, seed, P):
    """The moving objects: meshes in their own frames and, around each robot,
    their poses [envs, objects, 3, 4]."""
    rng = np.random.default_rng(seed + 1)
    n, k = len(P), case["objects"]
    one = np.zeros((1, 3))
    meshes = [_merged([_placed(_unit_sphere(3), one, one + 0.3)]),
              _merged([_placed(_unit_box(4), one - [0.4, 0.3, 0.3], one + [0.8, 0.6, 0.6])]),
              _merged([_placed(_unit_box(4), one - 0.25, one + 0.5)]),
              _merged([_placed(_unit_box(3), one - [0.1, 0.1, 0.9], one + [0.2, 0.2, 1.8])])]
    ang, far = rng.uniform(0, 2 * np.pi, (n, k)), rng.uniform(0.6, 1.2, (n, k))
    at = P[:, None, :, 3] + np.stack([far * np.cos(ang), far * np.sin(ang), rng.uniform(-0.2, 0.2, (n, k))], -1)
    R = _rotations(rng.uniform(0, 2 * np.pi, (n, k)), np.zeros((n, k)), np.zeros((n, k)))
    return [meshes[i % 4] for i in range(k)], np.ascontiguousarray(np.concatenate([R, at[..., None]], -1), np.float32)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("density", "mesh"):
        (mu, scale, quat, alpha), _ = _gaussian_room(np.random.default_rng(seed), case["gaussians"], case["room"])
        origin, dims = _room_grid(case)
        st = _State(case=case, g=[_dev(a) for a in (mu, scale, quat, alpha)], origin=origin, dims=dims)
        if kind == "mesh":
            st.mesh = _mesh_buffers(case, dims)
        return st
    if kind == "surface":
        surf, origin = _surface_grid(case, seed)
        return _State(case=case, surf=surf, origin=origin, mesh=_mesh_buffers(case, surf.shape))
    if kind == "effects":
        t, i = _returns(case, seed)
        return _State(case=case, seed=seed, range0=t, tri0=i, range=torch.empty_like(t), tri=torch.empty_like(i))
    meshes, angles, items = _ray_inputs(case, seed)
    sensors = [fgl.Sensor(*a) for a in angles]
    if kind == "lbvh":
        v, t = meshes[0]
        v, t = _dev(v), _dev(t)
        return _State(case=case, tree=fgl.Lbvh(v, t), verts=v, tris=t, sensor=sensors[0], poses=_dev(items[0][2]))
    # in a mixed batch one scene is held as a 4-wide tree
    scenes = [fgl.Scene(v, t, width=4 if k == 1 else 8) for k, (v, t) in enumerate(meshes)]
    st = _State(case=case, scenes=scenes, sensors=sensors)
    if kind == "cast":
        st.poses = _dev(items[0][2])
        return st
    pin = kind == "host"
    st.items, st.outs = [], []
    for k, a, P, near in items:
        n = len(P) * sensors[a].n_rays
        out = [torch.empty(n, dtype=d, pin_memory=True) if pin else torch.empty(n, dtype=d, device="cuda")
               for d in (torch.float32, torch.int32)]
        poses = torch.from_numpy(P).pin_memory() if pin else _dev(P)
        extra = None
        if kind == "instances":
            parts, at = _objects(case, seed, P)
            st.parts = [fgl.Scene(*m) for m in parts]
            out += [torch.empty((n, 3), dtype=torch.float32, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda")]
            extra = {"instances": st.parts, "instance_poses": _dev(at), "points": out[2], "out_instance": out[3]}
        st.items.append((scenes[k], sensors[a], poses, case["range"], out[0], out[1], near, extra))
        st.outs.append(out)
    if not pin:
        st.stream = torch.cuda.Stream() if case.get("graph") else None
        st.opts = fgl.BatchOpts(use_graph=1) if case.get("graph") else None
        st.arr = fgl.make_items(st.items)
    return st


def _mesh_buffers(case, dims):
    """The program's own vertex, triangle and normal buffers, with room to spare
    (zeros past the mesh)."""
    cells = (case["room"] / case["voxel"]) ** 2
    n = int(150 * cells) + 20_000 if case["kind"] == "mesh" else int(60 * cells + 0.01 * float(np.prod(dims))) + 1_000
    out = [torch.zeros((n, 3), dtype=torch.float32, device="cuda"), torch.zeros((2 * n, 3), dtype=torch.int32, device="cuda")]
    return out + ([torch.zeros((n, 3), dtype=torch.float32, device="cuda")] if case.get("normals") else [])


def _keep(buffers, mesh):
    for b, m in zip(buffers, mesh):
        b[:len(m)].copy_(m)
    return buffers


def _returns(case, seed):
    """Returns of one step: three quarters hits, the rest misses."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = case["envs"] * case["beams"] * case["az"]
    t = 0.3 + 20.0 * torch.rand(n, generator=gen, device="cuda") ** 2
    hit = torch.rand(n, generator=gen, device="cuda") < 0.75
    i = torch.randint(0, 1_000_000, (n,), generator=gen, device="cuda", dtype=torch.int32)
    return torch.where(hit, t, torch.full_like(t, 100.0)), torch.where(hit, i, torch.full_like(i, -1))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------


def run(st):
    case = st.case
    kind = case["kind"]
    if kind == "cast":
        return list(fgl.cast(st.scenes[0], st.sensors[0], st.poses, case["range"]))
    if kind == "host":
        fgl.cast_batched_host(st.items)
        return st.outs
    if kind in ("batched", "mixed", "instances"):
        if st.stream is None:
            fgl.cast_batched(st.items, arr=st.arr)
            return st.outs
        # a graph needs a stream of its own; the caller's stream waits for the step
        main = torch.cuda.current_stream()
        st.stream.wait_stream(main)
        fgl.cast_batched(st.items, st.opts, stream=st.stream, arr=st.arr)
        main.wait_stream(st.stream)
        return st.outs
    if kind == "lbvh":
        st.tree.rebuild(st.verts, st.tris)
        return list(st.tree.cast(st.sensor, st.poses, case["range"]))
    if kind == "density":
        return list(fgl.gaussian_density(*st.g, st.origin, case["voxel"], st.dims, tile=case["tile"])[:3])
    if kind == "mesh":
        return list(_keep(st.mesh, fgl.mesh_from_gaussians(*st.g, st.origin, case["voxel"], st.dims)))
    if kind == "surface":
        *mesh, phi = fgl.mesh_from_surface(st.surf, st.origin, case["voxel"], sigma=0.5 * case["voxel"] if case["denoise"] else None,
                                           normals=case["normals"], capacity=(len(st.mesh[0]), len(st.mesh[1])))
        return [*_keep(st.mesh, mesh), phi]
    # the effects work in place: each step's returns arrive fresh
    st.range.copy_(st.range0)
    st.tri.copy_(st.tri0)
    fgl.apply_sensor_effects(st.range, st.tri, case["envs"], seed=st.seed, step=3, drop_prob=case["drop"], sigma0=case["sigma0"],
                             sigma1=case["sigma1"], max_range=100.0)
    return [st.range, st.tri]


def work(case):
    """Bytes: inputs once, outputs once.  Flops of a ray: one 8-wide node test a
    level of an 8-ary tree and one triangle test; of a voxel row: its Gaussian
    terms, at the mean extent of the scale distribution."""
    kind = case["kind"]
    if kind in ("cast", "batched", "mixed", "instances", "host", "lbvh"):
        if kind == "mixed":  # mean rays of the six grids and the rosette
            rays, tris = case["envs"] * 72_000, 500.0 / case["voxel"] ** 2
        else:
            rays, tris = case["envs"] * case["beams"] * case["az"], case["tris"]
        out = 24 if kind == "instances" else 8
        levels = max(1.0, math.log(max(tris, 8)) / math.log(8))
        build = 200 * tris if kind == "lbvh" else 0
        seen = tris if kind == "lbvh" else min(tris, rays)
        return {"bytes": rays * out + case["envs"] * 48 + 18 * seen + 4 * 12 * tris * (kind == "lbvh"),
                "flops": rays * (96 * levels + 60) + build}
    if kind == "effects":
        n = case["envs"] * case["beams"] * case["az"]
        return {"bytes": 32 * n, "flops": 60 * n}  # the fresh copy in and out, then the pass in and out
    _, (nx, ny, nz) = _room_grid(case)
    vox = nx * ny * nz
    if kind == "surface":
        return {"bytes": 11 * vox + 100 * (case["room"] / case["voxel"]) ** 2, "flops": 20 * vox}
    h, n = case["voxel"], case["gaussians"]
    terms = n * ((0.36 + case.get("tile", 8) * h) / h) ** 3
    return {"bytes": 44 * n + (6 if kind == "density" else 17) * vox, "flops": 12 * terms}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------


def exact(case, seed):
    kind = case["kind"]
    if kind == "mesh":  # its vertices' number and order hang on thresholds that 64 bits may cross elsewhere
        return None
    if kind == "density":
        (mu, scale, quat, alpha), _ = _gaussian_room(np.random.default_rng(seed), case["gaussians"], case["room"])
        origin, dims = _room_grid(case)
        return [_density64(mu, scale, quat, alpha, origin, case["voxel"], dims, case["tile"]), None, None]
    if kind == "surface":
        surf, origin = _surface_grid(case, seed)
        v, nrm, phi = _mesh64(surf != 0, origin, case["voxel"], 0.5 * case["voxel"] if case["denoise"] else None, case["normals"])
        out = [b.double() if b.is_floating_point() else None for b in _mesh_buffers(case, surf.shape)]
        for b, m in zip(out[::2], (v, nrm)):
            b[:len(m)] = m
        return [*out, phi]
    if kind == "effects":
        return [_effects64(case, seed), None]
    meshes, angles, items = _ray_inputs(case, seed)
    pairs = sum(len(P) * len(angles[a][0]) * len(meshes[k][1]) for k, a, P, _ in items)
    if pairs > 1.2e11:
        return None
    outs = []
    for k, a, P, near in items:
        parts = _objects(case, seed, P) if kind == "instances" else ([], np.zeros((len(P), 0, 3, 4)))
        t, pts = _cast64(meshes[k], angles[a], P, near, case["range"], *parts)
        outs.append([t, None, pts, None] if kind == "instances" else [t, None])
    return outs[0] if kind in ("cast", "lbvh") else outs


def _cast64(mesh, angles, P, near, far, parts, at):
    """Nearest hit of every ray by testing every triangle: signed volumes of the
    ray with the triangle's edges, seen from the sensor."""
    el, az = (torch.from_numpy(x).cuda().double() for x in angles[:2])
    d0 = torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin()], 1)
    ts, ps = [], []
    for e in range(len(P)):
        pose = torch.from_numpy(P[e]).cuda().double()
        tri = [torch.from_numpy(mesh[0]).cuda().double()[torch.from_numpy(mesh[1]).cuda().long()]]
        for (v, t), M in zip(parts, at[e]):
            M = torch.from_numpy(M).cuda().double()
            tri.append((torch.from_numpy(v).cuda().double() @ M[:, :3].T + M[:, 3])[torch.from_numpy(t).cuda().long()])
        A, B, C = (torch.cat(tri) - pose[:, 3]).unbind(1)
        vol = (A * torch.cross(B, C, dim=1)).sum(1)
        N = [torch.cross(x, y, dim=1).T.contiguous() for x, y in ((C, B), (A, C), (B, A))]
        d = d0 @ pose[:, :3].T
        best = torch.full((len(d),), float(far), dtype=torch.float64, device="cuda")
        rows = max(1, (1 << 26) // len(A))
        for s in range(0, len(d), rows):
            U, V, W = (d[s:s + rows] @ n for n in N)
            det = U + V + W
            hit = (torch.minimum(torch.minimum(U, V), W) >= 0) | (torch.maximum(torch.maximum(U, V), W) <= 0)
            t = -vol / det
            t = torch.where(hit & (det != 0) & (t > 0) & (t >= near), t, best[s:s + rows, None])
            best[s:s + rows] = torch.minimum(best[s:s + rows], t.min(1).values)
        p = pose[:, 3] + best[:, None] * d
        p[best >= far] = float("nan")
        ts.append(best)
        ps.append(p)
    return torch.cat(ts), torch.cat(ps)


def _density64(mu, scale, quat, alpha, origin, h, dims, B):
    """Sum over the candidates of each voxel's tile; which tiles a Gaussian is a
    candidate of is a float32 decision of the interface, so it is taken so."""
    f = np.float32
    w, x, y, z = (quat / np.sqrt(((quat[:, 0] ** 2 + quat[:, 1] ** 2) + quat[:, 2] ** 2) + quat[:, 3] ** 2)[:, None]).T
    one, two = f(1), f(2)
    R = np.stack([np.stack([one - two * (y * y + z * z), two * (x * y - w * z), two * (x * z + w * y)], -1),
                  np.stack([two * (x * y + w * z), one - two * (x * x + z * z), two * (y * z - w * x)], -1),
                  np.stack([two * (x * z - w * y), two * (y * z + w * x), one - two * (x * x + y * y)], -1)], -2)
    q = R * scale[:, None, :]
    e = f(3) * np.sqrt((q[..., 0] ** 2 + q[..., 1] ** 2) + q[..., 2] ** 2)
    o, cell = np.array(origin, f), f(B) * f(h)
    tiles = np.array([-(-n // B) for n in dims])
    lo = np.maximum(np.floor((mu - e - o) / cell), 0).astype(int)
    hi = np.minimum(np.floor((mu + e - o) / cell), tiles - 1).astype(int)
    n = np.prod(np.maximum(hi - lo + 1, 0), 1)
    g = np.repeat(np.arange(len(mu)), n)
    i = np.arange(len(g)) - np.repeat(np.cumsum(n) - n, n)
    ext = (hi - lo + 1)[g]
    t = lo[g] + np.stack([i % ext[:, 0], i // ext[:, 0] % ext[:, 1], i // (ext[:, 0] * ext[:, 1])], 1)
    # the inverse covariance from the unrounded rotation
    qd = torch.from_numpy(quat).cuda().double()
    w, x, y, z = (qd / qd.norm(dim=1, keepdim=True)).unbind(1)
    Rd = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z), 1 - 2 * (x * x + z * z),
                      2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    Q = Rd / torch.from_numpy(scale).cuda().double()[:, None, :]
    md, a2 = torch.from_numpy(mu).cuda().double(), torch.from_numpy(alpha).cuda().double() ** 2
    hd = float(f(h))
    od = torch.from_numpy(o).cuda().double()
    idx = torch.arange(B ** 3, device="cuda")
    inside = (torch.stack([idx % B, idx // B % B, idx // (B * B)], 1).double() + 0.5) * hd
    out = torch.zeros((int(np.prod(tiles)), B ** 3), dtype=torch.float64, device="cuda")
    gd, td = torch.from_numpy(g).cuda(), torch.from_numpy(t).cuda()
    for s in range(0, len(g), 1 << 17):
        gs, tt = gd[s:s + (1 << 17)], td[s:s + (1 << 17)]
        p = (od + tt.double() * (B * hd) - md[gs])[:, None, :] + inside
        r = torch.einsum("nvi,nij->nvj", p, Q[gs])
        term = a2[gs, None] * torch.exp(-0.5 * (r * r).sum(2))
        out.index_add_(0, (tt[:, 2] * int(tiles[1]) + tt[:, 1]) * int(tiles[0]) + tt[:, 0], term)
    out = out.view(tiles[2], tiles[1], tiles[0], B, B, B).permute(0, 3, 1, 4, 2, 5).reshape(tiles[2] * B, tiles[1] * B, tiles[0] * B)
    return out[:dims[2], :dims[1], :dims[0]].contiguous()


def _faces(p, op):
    """op over the six face neighbours of a grid padded by one."""
    n = [p[2:, 1:-1, 1:-1], p[:-2, 1:-1, 1:-1], p[1:-1, 2:, 1:-1], p[1:-1, :-2, 1:-1], p[1:-1, 1:-1, 2:], p[1:-1, 1:-1, :-2]]
    r = n[0]
    for x in n[1:]:
        r = op(r, x)
    return r


def _mesh64(surf, origin, h, sigma, normals, trunc=0.06):
    """(vertices, normals or None, phi) of a surface grid."""
    hd, td = float(np.float32(h)), float(np.float32(trunc))
    if sigma:
        sv = float(np.float32(sigma)) / hd
        R = int(math.ceil(3 * sv))
        w = torch.exp(-torch.arange(-R, R + 1, device="cuda").double() ** 2 / (2 * sv * sv))
        w /= w.sum()
        b = surf.double()
        for axis in range(3):
            pad = [0] * 6
            pad[2 * (2 - axis)] = pad[2 * (2 - axis) + 1] = R
            p = torch.nn.functional.pad(b, pad)
            b = sum(w[k] * p.narrow(axis, k, b.shape[axis]) for k in range(2 * R + 1))
        surf = b >= 0.5
    pad = (1, 1, 1, 1, 1, 1)
    free = ~surf
    out = torch.zeros_like(surf)
    last = -1
    while True:  # the frame's component of the free voxels
        for _ in range(16):
            out |= free & _faces(torch.nn.functional.pad(out, pad, value=True), torch.logical_or)
        now = int(out.sum())
        if now == last:
            break
        last = now
    other = torch.nn.functional.pad(surf.to(torch.int8), pad, value=-1)
    here = surf.to(torch.int8)
    n = [other[2:, 1:-1, 1:-1], other[:-2, 1:-1, 1:-1], other[1:-1, 2:, 1:-1], other[1:-1, :-2, 1:-1], other[1:-1, 1:-1, 2:], other[1:-1, 1:-1, :-2]]
    m = torch.zeros_like(surf)
    for x in n:
        m |= (x >= 0) & (x != here)
    layers = int(math.ceil(td / hd))
    dist = torch.full(surf.shape, td, dtype=torch.float64, device="cuda")
    dist[m] = min(0.5 * hd, td)
    for p in range(1, layers + 1):
        grown = m | _faces(torch.nn.functional.pad(m, pad), torch.logical_or)
        dist[grown & ~m] = min((p + 0.5) * hd, td)
        m = grown
    phi = torch.where(out, dist, -dist)
    inside = phi < 0
    nz, ny, nx = phi.shape
    cross = torch.zeros((*phi.shape, 7), dtype=torch.bool, device="cuda")
    for t in range(1, 8):
        dx, dy, dz = t & 1, (t >> 1) & 1, (t >> 2) & 1
        cross[:nz - dz, :ny - dy, :nx - dx, t - 1] = inside[:nz - dz, :ny - dy, :nx - dx] != inside[dz:, dy:, dx:]
    k, j, i, t = cross.nonzero().unbind(1)
    del cross
    t = t + 1
    step = torch.stack([t & 1, (t >> 1) & 1, (t >> 2) & 1], 1)
    kb, jb, ib = k + step[:, 2], j + step[:, 1], i + step[:, 0]
    fa, fb = phi[k, j, i], phi[kb, jb, ib]
    tau = (0.0 - fa) / (fb - fa)
    o = torch.tensor([float(np.float32(x)) for x in origin], dtype=torch.float64, device="cuda")
    v = o + (torch.stack([i, j, k], 1).double() + 0.5) * hd + (tau * hd)[:, None] * step.double()
    if not normals:
        return [v, None, phi]

    def grad(a):
        g = []
        for axis, n_ax in ((2, nx), (1, ny), (0, nz)):
            up, dn = [x.clone() for x in a], [x.clone() for x in a]
            up[axis] = (a[axis] + 1).clamp(max=n_ax - 1)
            dn[axis] = (a[axis] - 1).clamp(min=0)
            span = (up[axis] - dn[axis]).double() * hd
            g.append((phi[tuple(up)] - phi[tuple(dn)]) / span)
        return torch.stack(g, 1)

    nrm = (1 - tau)[:, None] * grad((k, j, i)) + tau[:, None] * grad((kb, jb, ib))
    length = nrm.norm(dim=1, keepdim=True)
    return [v, torch.where(length > 0, nrm / length, torch.zeros_like(nrm)), phi]


def _effects64(case, seed):
    """Philox-4x32-10 words, dropout, then Box-Muller noise on the kept hits."""
    t, tri = _returns(case, seed)
    rays = case["beams"] * case["az"]
    n = torch.arange(t.numel(), device="cuda")
    M = 0xFFFFFFFF

    def mul(a, b):  # 32 x 32 -> (low, high) in int64 halves
        lo, hi = a * (b & 0xFFFF), a * (b >> 16)
        mid = (lo >> 16) + (hi & M)
        full_hi = ((lo >> 16) + hi) >> 16
        return ((mid << 16) | (lo & 0xFFFF)) & M, full_hi & M

    c = [n % rays, n // rays, torch.full_like(n, 3), torch.zeros_like(n)]
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        l0, h0 = mul(c[0], 0xD2511F53)
        l1, h1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    f32 = lambda x: float(np.float32(x))  # noqa: E731
    u0, u1, u2 = (c[0] >> 8).double() / 2 ** 24, ((c[1] >> 8) + 1).double() / 2 ** 24, (c[2] >> 8).double() / 2 ** 24
    t = t.double()
    noise = torch.sqrt(-2 * torch.log(u1)) * torch.cos(2 * math.pi * u2)
    kept = (t + (f32(case["sigma0"]) + f32(case["sigma1"]) * t) * noise).clamp(0.0, 100.0)
    kept = torch.where(u0 < f32(case["drop"]), torch.full_like(t, 100.0), kept)
    return torch.where(tri >= 0, kept, t)
