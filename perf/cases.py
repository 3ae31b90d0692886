"""What a program that uses this framework has it do, as cases that can be timed and compared.

The cases are the fusion calls of the C ABI through its Python binding, on views of the
synthetic room (0.5-4 m deep, Kinect noise, 5 % dropout), and the read-out that follows them:

  track     one frame into a map that already holds the blocks it sees: the steady state of a
            camera that moves through a known place. `sync`: the default call, which waits and
            returns the status; otherwise the caller goes on at once.
  stages    the same with allocation and integration as two kernels (fuse mode 0).
  scan      an emptied volume, a run of frames, and the map in key order: a new session.
  batch     one frame for each of many sessions in one call.
  stream    frames in pinned host memory, fused in order into one map.
  mesh      the surface of a map, its triangles in the order of their cells.

Where the order of blocks matters to the result (pool indices are given out as blocks are
claimed), the map is laid out by the program beforehand -- it owns the volume's memory -- or the
blocks are put in key order at the end. Everything is on the current CUDA device.
"""
import functools
import math

import numpy as np
import torch

from paper_2608_08287_gb300 import synth, tsdf

DEV = "cuda"
ROOM_SEED = 20261204          # the room of the repository's own frames
EMPTY = -1                    # the empty key as int64
AXIS = 1 << 20                # bias of a packed block coordinate


def _case(name, kind, width, height, voxel, band, **more):
    c = dict(name=name, kind=kind, width=width, height=height, voxel=voxel, band=band,
             colour=True, sync=False, load=0.0, frames=1)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: a 160x120 camera at 1 cm, waiting for each frame's status
        _case("track_160x120_sync", "track", 160, 120, 0.01, 4, sync=True),
        # a 320x240 camera at 5 mm; half of the GPU's threads have work
        _case("track_320x240", "track", 320, 240, 0.005, 4),
        # the headline workload of the benchmark: 640x480 at 5 mm, colour
        _case("track_640x480", "track", 640, 480, 0.005, 4),
        # the same camera when the table has filled up to the load of a whole orbit
        _case("track_640x480_full_table", "track", 640, 480, 0.005, 4, load=0.88),
        # depth only, a wide band, the largest image
        _case("track_1280x720_depth_wide", "track", 1280, 720, 0.005, 8, colour=False),
        # odd sizes, and a truncation of three voxels, which has no compiled band
        _case("track_423x237_band3", "track", 423, 237, 0.0075, 3),
        # a wide truncation of a coarse map, again without a compiled band
        _case("track_637x477_band6", "track", 637, 477, 0.01, 6, sync=True),
        # allocation and integration as separate passes, as the paper has them
        _case("stages_640x480", "stages", 640, 480, 0.005, 4),
        # a new session: everything that it sees has to be allocated
        _case("scan_640x480_x8", "scan", 640, 480, 0.005, 4, frames=8),
        # many sessions at once, cameras of three sizes
        _case("batch_24_sessions", "batch", 640, 480, 0.005, 4, frames=24),
        # a recorded sequence from host memory, copies and fusion overlapping
        _case("stream_640x480_x12", "stream", 640, 480, 0.005, 4, frames=12),
        # the surface of a room's map
        _case("mesh_640x480", "mesh", 640, 480, 0.005, 4),
    ]


def draw(rng):
    kind = rng.choice(["track"] * 5 + ["stages", "scan", "batch", "stream", "mesh"])
    top = {"track": 1280, "stages": 800}.get(kind, 640)
    width = int(round(math.exp(rng.uniform(math.log(96), math.log(top)))))
    height = max(48, int(width * rng.uniform(0.5, 0.75)))
    if rng.random() < 0.5:  # half of the cameras have whole tiles
        width, height = width // 16 * 16, height // 16 * 16
    voxel = rng.choice([0.005, 0.0075, 0.01, 0.02])
    band = rng.choice([2, 3, 4, 4, 4, 4, 5, 6, 8])
    c = dict(kind=kind, width=width, height=height, voxel=voxel, band=band,
             colour=rng.random() < 0.75, sync=rng.random() < 0.3, load=0.0, frames=1)
    if kind == "track" and rng.random() < 0.2:
        c["load"] = round(rng.uniform(0.5, 0.88), 3)
    if kind in ("scan", "stream"):
        c["frames"] = rng.randint(3, 8)
    if kind == "batch":
        c["frames"] = rng.randint(2, 20)
    return c


# ----------------------------------------------------------------------------
# views of the room, rendered on the GPU
# ----------------------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def _prims():
    return synth.room_prims(ROOM_SEED)


def _hits(o, d, p):
    """Ray parameter of primitive p for rays o + s d (s is the camera depth); inf for none."""
    inf = float("inf")
    if isinstance(p, synth.Plane):
        n = torch.tensor(p.n, dtype=torch.float64, device=DEV)
        s = (p.c - o @ n) / (d @ n)
        return torch.where(s > 1e-9, s, inf)
    if isinstance(p, synth.Sphere):
        oc = o - torch.tensor(p.centre, dtype=torch.float64, device=DEV)
        a, b, c = (d * d).sum(1), d @ oc, oc @ oc - p.r * p.r
        q = b * b - a * c
        s = (-b - q.clamp(min=0).sqrt()) / a
        return torch.where((q >= 0) & (s > 1e-9), s, inf)
    lo, hi = (torch.tensor(x, dtype=torch.float64, device=DEV) for x in (p.lo, p.hi))
    t1, t2 = (lo - o) / d, (hi - o) / d
    near, far = torch.minimum(t1, t2).amax(1), torch.maximum(t1, t2).amin(1)
    return torch.where((near > 1e-9) & (far >= near), near, inf)


def _camera(width, height):
    s = width / 640.0
    return np.array([525.0 * s, 525.0 * s, (width - 1) / 2.0, (height - 1) / 2.0], np.float32)


def _view(width, height, colour, seed, at):
    """Frame `at` of the orbit that `seed` starts: depth, colour or None, intrinsics, pose."""
    first = np.random.RandomState(seed & 0x7FFFFFFF).randint(0, 300)
    intr = _camera(width, height)
    pose = synth.orbit_pose(first + at, ROOM_SEED + 1).astype(np.float32)
    fx, fy, cx, cy = (float(x) for x in intr)
    v, u = torch.meshgrid(torch.arange(height, device=DEV, dtype=torch.float64),
                          torch.arange(width, device=DEV, dtype=torch.float64), indexing="ij")
    ray = torch.stack([(u.reshape(-1) - cx) / fx, (v.reshape(-1) - cy) / fy,
                       torch.ones(width * height, device=DEV, dtype=torch.float64)], 1)
    P = torch.from_numpy(pose.astype(np.float64)).to(DEV)
    o, d = P[:3, 3], ray @ P[:3, :3].T
    z = torch.stack([_hits(o, d, p) for p in _prims()])
    z, what = z.min(0)
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1009 + at) & 0x7FFFFFFFFFFF)
    sigma = 0.0012 + 0.0019 * (z - 0.4) ** 2
    z = z + sigma * torch.randn(z.shape, generator=g, device=DEV, dtype=torch.float64)
    kept = torch.rand(z.shape, generator=g, device=DEV) >= 0.05
    depth = torch.where(kept & torch.isfinite(z) & (z > 0), z, 0.0).float().view(height, width)
    rgb = None
    if colour:
        albedo = torch.tensor([p.albedo for p in _prims()], device=DEV)
        jitter = torch.randint(-12, 13, (width * height, 3), generator=g, device=DEV)
        rgb = (albedo[what] + jitter).clamp(0, 255).to(torch.uint8).view(height, width, 3)
    return depth.contiguous(), rgb, intr, pose


# ----------------------------------------------------------------------------
# the maps that the cameras move through
# ----------------------------------------------------------------------------
def _pack(b):
    """Sortable key of block coordinates (n, 3) int64, in the order x, y, z."""
    return ((b[:, 0] + AXIS) << 42) | ((b[:, 1] + AXIS) << 21) | (b[:, 2] + AXIS)


def _unpack(key):
    m = (1 << 21) - 1
    return torch.stack([((key >> 42) & m) - AXIS, ((key >> 21) & m) - AXIS, (key & m) - AXIS], 1)


def _points(view):
    """Depth, world position and unit ray of a view's valid points, in 64 bits."""
    depth, _, intr, pose = view
    fx, fy, cx, cy = (float(x) for x in intr)
    h, w = depth.shape
    d = depth.reshape(-1).double()
    at = torch.nonzero(torch.isfinite(d) & (d > 0)).reshape(-1)
    d = d[at]
    rx, ry = ((at % w).double() - cx) / fx, (torch.div(at, w, rounding_mode="floor").double() - cy) / fy
    R = torch.from_numpy(pose[:3, :3].astype(np.float64)).to(DEV)
    t = torch.from_numpy(pose[:3, 3].astype(np.float64)).to(DEV)
    ray = torch.stack([rx, ry, torch.ones_like(rx)], 1)
    return (ray * d[:, None]) @ R.T + t, (ray / ray.norm(dim=1, keepdim=True)) @ R.T


def _blocks_seen(view, voxel, band):
    """Keys of the blocks that a view's bands reach, with those a hair beside them."""
    p, n = _points(view)
    found = []
    for k in range(-band, band + 1):
        x = (p + (k * voxel) * n) / voxel
        lo, hi = torch.floor((x - 0.01) / 8).long(), torch.floor((x + 0.01) / 8).long()
        key = torch.unique(torch.cat([_pack(lo), _pack(hi)]))
        mixed = (lo != hi).sum(1) > 1  # near an edge or a corner of its block
        lo, hi = lo[mixed], hi[mixed]
        for c in range(1, 7):
            take = torch.tensor([(c >> j) & 1 for j in range(3)], device=DEV, dtype=torch.bool)
            key = torch.cat([key, _pack(torch.where(take, hi, lo))])
        found.append(torch.unique(key))
    return torch.unique(torch.cat(found))


def _pow2(n):
    return 1 << max(1, int(n - 1).bit_length())


@functools.lru_cache(maxsize=64)
def _view_size(width, height, voxel, band):
    """The most blocks that one of four views around the orbit sees."""
    intr = _camera(width, height)
    return max(len(_blocks_seen(_view(width, height, False, 0, at), voxel, band))
               for at in (0, 75, 150, 225))


def _map_size(case, width=None, height=None, views=1):
    """(blocks, table slots) of the map of a case, the same for every seed. With `load`, the
    table is filled that far; otherwise it is the next power of two above twice the blocks."""
    w, h = width or case["width"], height or case["height"]
    own = _view_size(w, h, case["voxel"], case["band"])
    if case["load"]:
        slots = _pow2(2 * own)
        return max(int(1.5 * own), int(case["load"] * slots)), slots
    n = int((1.4 + 0.2 * views) * own) + 64
    return n, _pow2(2 * n + 1)


def _map_keys(case, seed, width=None, height=None, views=1):
    """Keys of a map's blocks in pool order: what the camera sees in its `views` frames (every
    fourth of its orbit), and other parts of the orbit up to the map's size."""
    w, h = width or case["width"], height or case["height"]
    n, _ = _map_size(case, w, h, views)

    def seen(at):
        return _blocks_seen(_view(w, h, False, seed, at), case["voxel"], case["band"])

    own = have = torch.unique(torch.cat([seen(4 * i) for i in range(views)]))
    at = 4 * views - 4
    while len(have) < n:
        at += 6
        have = torch.unique(torch.cat([have, seen(at)]))
    others = have[~torch.isin(have, own)][:max(0, n - len(own))]
    keys = torch.unique(torch.cat([own, others]))
    if len(keys) != n:
        raise RuntimeError("%d blocks seen, the map has %d" % (len(keys), n))
    return keys


def _place(keys, slots):
    """Table slot of every key, by linear probing from its home slot."""
    b = _unpack(keys).cpu().numpy().astype(np.uint32)
    home = ((b[:, 0] * np.uint32(73856093)) ^ (b[:, 1] * np.uint32(19349669))
            ^ (b[:, 2] * np.uint32(83492791))).astype(np.int64) & (slots - 1)
    taken = np.zeros(slots, bool)
    slot = np.full(len(home), -1, np.int64)
    left, s = np.arange(len(home)), home.copy()
    while len(left):
        free = np.nonzero(~taken[s])[0]
        _, first = np.unique(s[free], return_index=True)
        won = free[first]
        slot[left[won]] = s[won]
        taken[s[won]] = True
        stay = np.ones(len(left), bool)
        stay[won] = False
        left, s = left[stay], (s[stay] + 1) & (slots - 1)
    return torch.from_numpy(slot).to(DEV)


class _Map:
    """A volume in memory that the program owns, and views of its sums."""

    def __init__(self, case, pool, slots, keys=None):
        pool = min(pool, slots)
        nbytes = tsdf.tsdf_volume_bytes(slots, pool)
        self.memory = torch.empty(nbytes, dtype=torch.uint8, device=DEV)
        self.vol = tsdf.Volume(case["voxel"], case["voxel"] * case["band"], slots, pool,
                               memory=self.memory)
        lay = self.vol.layout()

        def part(at, size, dtype):
            return self.memory[at:at + size].view(dtype)

        self.sums = part(lay.voxel_sums_offset, pool * 8192, torch.float32).view(pool, 512, 4)
        self.blue = part(lay.blue_sums_offset, pool * 2048, torch.float32).view(pool, 512)
        self.coords = part(lay.coords_offset, pool * 12, torch.int32).view(pool, 3)
        if keys is not None:  # the blocks of the map: pool index i is keys[i]
            n = len(keys)
            slot = _place(keys, slots)
            table = part(lay.table_offset, slots * 16, torch.int64).view(slots, 2)
            table[slot, 0] = keys
            table.view(torch.int32)[slot, 2] = torch.arange(n, device=DEV, dtype=torch.int32)
            self.coords[:n] = _unpack(keys).int()
            part(0, 4, torch.int32)[0] = n
            self.sums, self.blue = self.sums[:n], self.blue[:n]

    def state(self, colour):
        return {"sums": self.sums, "blue": self.blue} if colour else {"sums": self.sums}


def _sessions(case):
    """Sizes of a batch's cameras: a third each of the full, the half and the quarter size."""
    w, h = case["width"], case["height"]
    return [(max(16, w >> (i % 3)), max(12, h >> (i % 3))) for i in range(case["frames"])]


def _call(view):
    """A view as a call takes it: its arrays, and its camera as the binding's structs."""
    depth, rgb, intr, pose = view
    return depth, rgb, tsdf.intrinsics(intr), tsdf.pose_struct(pose)


def _frames_of(case, seed):
    """The frames that a pass fuses (every fourth of the orbit)."""
    return [_view(case["width"], case["height"], case["colour"], seed, 4 * i)
            for i in range(case["frames"])]


def _mesh_samples(case, seed, keys):
    """(tsdf sum, weight) of every voxel of a map seen from one camera, as float32. Every seed
    has its own distances and weights, and the same sides of the surface: as many triangles."""
    depth, _, intr, pose = _view(case["width"], case["height"], False, 0, 0)
    h, w = depth.shape
    fx, fy, cx, cy = (float(x) for x in intr)
    R = torch.from_numpy(pose[:3, :3].astype(np.float64)).to(DEV)
    t = torch.from_numpy(pose[:3, 3].astype(np.float64)).to(DEV)
    tau = case["voxel"] * case["band"]
    l = torch.arange(512, device=DEV)
    local = torch.stack([l & 7, (l >> 3) & 7, l >> 6], 1)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed & 0x7FFFFFFF)
    out = []
    for part in torch.split(keys, 4096):
        x = (((_unpack(part) * 8)[:, None] + local[None]).reshape(-1, 3).double() + 0.5) * case["voxel"]
        c = (x - t) @ R
        u = torch.floor(fx * c[:, 0] / c[:, 2] + cx + 0.5)
        v = torch.floor(fy * c[:, 1] / c[:, 2] + cy + 0.5)
        inside = (c[:, 2] > 0) & (u >= 0) & (u < w) & (v >= 0) & (v < h)
        q = torch.where(inside, v * w + u, 0.0).long()
        d = torch.where(inside, depth.reshape(-1)[q].double(), 0.0)
        off = (d - c[:, 2]) / tau
        seen = (d > 0) & (off >= -1.0) & (off <= 1.0)
        off = off * (0.5 + 0.5 * torch.rand(off.shape, generator=g, device=DEV, dtype=torch.float64))
        weight = torch.randint(1, 9, seen.shape, generator=g, device=DEV).float() * seen
        out.append(torch.stack([off.float() * weight, weight], 1))
    return torch.cat(out).view(-1, 512, 2)


# ----------------------------------------------------------------------------
# prepare, run
# ----------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("track", "stages"):
        n, slots = _map_size(case)
        m = _Map(case, n + 1024, slots, _map_keys(case, seed))
        if kind == "stages":
            m.vol.set_option("fuse_mode", 0)
        view = _call(_view(case["width"], case["height"], case["colour"], seed, 0))
        return {"case": case, "map": m, "view": view}
    if kind == "scan":
        pool = _map_size(case, views=case["frames"])[0]
        m = _Map(case, pool, _pow2(2 * pool + 1))
        result = {"coords": torch.zeros_like(m.coords), "sums": torch.zeros_like(m.sums)}
        if case["colour"]:
            result["blue"] = torch.zeros_like(m.blue)
        return {"case": case, "map": m, "views": [_call(v) for v in _frames_of(case, seed)],
                "result": result}
    if kind == "batch":
        maps, items = [], []
        for i, (w, h) in enumerate(_sessions(case)):
            n, slots = _map_size(case, w, h)
            maps.append(_Map(case, n + 256, slots, _map_keys(case, seed + 31 * i, w, h)))
            items.append((maps[-1].vol.handle,
                          *_call(_view(w, h, case["colour"], seed + 31 * i, 0))))
        return {"case": case, "maps": maps, "items": items, "frames": tsdf.make_frames(items),
                "batch": tsdf.Batch(case["frames"])}
    if kind == "stream":
        n, slots = _map_size(case, views=case["frames"])
        m = _Map(case, n + 1024, slots, _map_keys(case, seed, views=case["frames"]))
        host = [(m.vol.handle, d.cpu().pin_memory(), c.cpu().pin_memory() if c is not None else None,
                 i, p) for d, c, i, p in (_call(v) for v in _frames_of(case, seed))]
        return {"case": case, "map": m, "host": host, "frames": tsdf.make_host_frames(host)}
    n, slots = _map_size(case)
    keys = _map_keys(case, 0)
    m = _Map(case, n, slots, keys)
    m.sums[..., :2] = _mesh_samples(case, seed, keys)
    room = 220 * n
    return {"case": case, "map": m, "room": room,
            "tris": torch.empty(room, 9, device=DEV),
            "cells": torch.empty(room, 4, device=DEV, dtype=torch.int32),
            "count": torch.zeros(1, device=DEV, dtype=torch.int32)}


def _ok(status):
    if status != "OK":
        raise RuntimeError(status)


def _in_key_order(m, n, result):
    """The first n blocks of a volume in the order of their coordinates, in the program's arrays."""
    c = m.coords[:n]
    b = c.long()
    order = torch.argsort((b[:, 0] << 42) + (b[:, 1] << 21) + b[:, 2])
    torch.index_select(c, 0, order, out=result["coords"][:n])
    torch.index_select(m.sums, 0, order, out=result["sums"][:n])
    if "blue" in result:
        torch.index_select(m.blue, 0, order, out=result["blue"][:n])
    return {"blocks": n, **result}


def _cell_order(c):
    """Triangles by the x, y, z of their cells and their place in them: the packed cells in
    order, and the order."""
    key = c[:, 0].long().mul_(1 << 18).add_(c[:, 1]).mul_(1 << 18).add_(c[:, 2]).mul_(16).add_(c[:, 3])
    return torch.sort(key)


def run(state):
    case = state["case"]
    kind, colour = case["kind"], case["colour"]
    if kind in ("track", "stages"):
        m = state["map"]
        depth, rgb, intr, pose = state["view"]
        _ok(m.vol.fuse(depth, intr, pose, rgb, sync=case["sync"]))
        return m.state(colour)
    if kind == "scan":
        m = state["map"]
        _ok(m.vol.reset())
        for depth, rgb, intr, pose in state["views"]:
            _ok(m.vol.fuse(depth, intr, pose, rgb, sync=False))
        _ok(m.vol.status())
        return _in_key_order(m, m.vol.block_count(), state["result"])
    if kind == "batch":
        _ok(tsdf.tsdf_fuse_batch_async(state["batch"].handle, state["frames"]))
        return [m.state(colour) for m in state["maps"]]
    if kind == "stream":
        _ok(tsdf.tsdf_fuse_frames_host(state["frames"])[0])
        return state["map"].state(colour)
    _ok(tsdf.tsdf_extract_mesh_async(state["map"].vol.handle, state["tris"], state["cells"],
                                     state["room"], state["count"]))
    n = int(state["count"])
    cells, order = _cell_order(state["cells"][:n])
    return {"tris": torch.gather(state["tris"], 0, order[:, None].expand(-1, 9)), "cells": cells}


# ----------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------
def _f(a):
    return a.double() if isinstance(a, torch.Tensor) else float(a)


def _fma(a, b, c):
    return (_f(a) * _f(b) + _f(c)).float()


def _mul(a, b):
    return (_f(a) * _f(b)).float()


def _add(a, b):
    return (_f(a) + _f(b)).float()


def _div(a, b):
    return (_f(a) / _f(b)).float()


def _contributions(view, voxel, band):
    """The voxels that a frame's points reach: which are taken is decided in float32, in the
    order of operations that the framework fixes; the values are computed in 64 bits. Returns
    (block key, local index, tsdf, pixel) of each."""
    depth, _, intr, pose = view
    f32 = np.float32
    v, tau = f32(voxel), f32(voxel * band)
    fx, fy, cx, cy = (f32(x) for x in intr)
    h, w = depth.shape
    flat = depth.reshape(-1)
    px = torch.nonzero(torch.isfinite(flat) & (flat > 0)).reshape(-1)
    d = flat[px]
    rx = _div(_add((px % w).float(), -cx), fx)
    ry = _div(_add(torch.div(px, w, rounding_mode="floor").float(), -cy), fy)
    n = torch.sqrt(_fma(rx, rx, _fma(ry, ry, 1.0)).double()).float()
    R, t = pose[:3, :3], pose[:3, 3]
    cp = (_mul(rx, d), _mul(ry, d), d)
    cd = (_div(rx, n), _div(ry, n), (1.0 / n.double()).float())
    P, D = [], []
    for i in range(3):
        P.append(_fma(float(R[i, 2]), cp[2], _fma(float(R[i, 1]), cp[1], _fma(float(R[i, 0]), cp[0], float(t[i])))))
        D.append(_fma(float(R[i, 2]), cd[2], _fma(float(R[i, 1]), cd[1], _mul(float(R[i, 0]), cd[0]))))

    def fma32(a, b, c):
        return f32(np.float64(a) * np.float64(b) + np.float64(c))

    half = [fma32(f32(0.5), v, -t[i]) for i in range(3)]
    A = [[f32(v * R[i, j]) for i in range(3)] for j in range(3)]
    b = [fma32(R[2, j], half[2], fma32(R[1, j], half[1], f32(R[0, j] * half[0]))) for j in range(3)]
    inv_v = f32(1.0) / v
    R64, t64, v64 = pose[:3, :3].astype(np.float64), pose[:3, 3].astype(np.float64), float(v)
    out, last = [], None
    for k in range(2 * band + 1):
        tk = f32(f32(k - band) * v)
        q = [torch.floor(_mul(_fma(float(tk), D[i], P[i]), inv_v)) for i in range(3)]
        fresh = torch.ones_like(px, dtype=torch.bool)
        if last is not None:
            fresh = (q[0] != last[0]) | (q[1] != last[1]) | (q[2] != last[2])
        last = q
        c = [_fma(float(A[j][2]), q[2], _fma(float(A[j][1]), q[1], _fma(float(A[j][0]), q[0], float(b[j]))))
             for j in range(3)]
        iz = (1.0 / c[2].double()).float()
        qu = torch.floor(_add(_fma(float(fx), _mul(c[0], iz), float(cx)), 0.5))
        qv = torch.floor(_add(_fma(float(fy), _mul(c[1], iz), float(cy)), 0.5))
        ok = fresh & (c[2] > 0) & (qu >= 0) & (qu < w) & (qv >= 0) & (qv < h)
        at = torch.where(ok, qv.double() * w + qu.double(), 0.0).long()
        d2 = torch.where(ok, flat[at], 0.0)
        ok &= torch.isfinite(d2) & (d2 > 0) & (_add(d2, -c[2]) >= -float(tau))
        i = torch.nonzero(ok).reshape(-1)
        g = torch.stack([x[i].long() for x in q], 1)
        centre = (g.double() + 0.5) * v64 - torch.from_numpy(t64).to(DEV)
        z = centre @ torch.from_numpy(R64[:, 2].copy()).to(DEV)
        value = ((d[i].double() - z) / float(tau)).clamp(-1.0, 1.0)
        lo = g & 7
        out.append((_pack(g >> 3), lo[:, 0] | (lo[:, 1] << 3) | (lo[:, 2] << 6), value, px[i]))
    return [torch.cat(x) for x in zip(*out)]


def _sums(view, voxel, band, keys, sums, blue):
    """Adds a frame to sums (n, 512, 4) and blue (n, 512) of the blocks `keys` (sorted)."""
    key, local, value, px = _contributions(view, voxel, band)
    at = torch.searchsorted(keys, key) * 512 + local
    rgb = view[1]
    colour = rgb.reshape(-1, 3)[px].double() if rgb is not None else value.new_zeros(len(px), 3)
    sums.view(-1, 4).index_add_(0, at, torch.cat([value[:, None], torch.ones_like(value)[:, None],
                                                  colour[:, :2]], 1))
    blue.view(-1).index_add_(0, at, colour[:, 2].contiguous())


def _exact_maps(views, case, keys):
    sums = torch.zeros(len(keys), 512, 4, device=DEV, dtype=torch.float64)
    blue = torch.zeros(len(keys), 512, device=DEV, dtype=torch.float64)
    for view in views:
        _sums(view, case["voxel"], case["band"], keys, sums, blue)
    return {"sums": sums, "blue": blue} if case["colour"] else {"sums": sums}


TETS = ((0, 1, 3, 7), (0, 1, 7, 5), (0, 2, 7, 3), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 7, 6))


def _tet_triangles(inside):
    """Triangles (three edges as pairs of the tetrahedron's corners 0-3) for a 4-bit mask of its
    inside corners, wound towards the outside."""
    lone = ((0, 1, 2, 3), (1, 0, 3, 2), (2, 0, 1, 3), (3, 0, 2, 1))
    pair = {3: (0, 1, 2, 3), 5: (0, 2, 3, 1), 6: (1, 2, 0, 3), 9: (0, 3, 1, 2), 10: (1, 3, 2, 0),
            12: (2, 3, 0, 1)}
    n = bin(inside).count("1")
    if n in (0, 4):
        return []
    if n == 2:
        a, b, c, d = pair[inside]
        return [((a, c), (a, d), (b, d)), ((a, c), (b, d), (b, c))]
    a, b, c, d = lone[(inside if n == 1 else 15 - inside).bit_length() - 1]
    return [((a, b), (a, c), (a, d)) if n == 1 else ((a, b), (a, d), (a, c))]


def _exact_mesh(case, seed):
    keys = _map_keys(case, 0)
    s = _mesh_samples(case, seed, keys).double()
    v = float(np.float32(case["voxel"]))
    mean = torch.where(s[..., 1] > 0, s[..., 0] / s[..., 1], float("nan"))
    blocks = _unpack(keys)
    tile = torch.full((len(keys), 9, 9, 9), float("nan"), device=DEV, dtype=torch.float64)  # z, y, x
    grid = mean.view(-1, 8, 8, 8)
    for c in range(8):
        step = torch.tensor([c & 1, (c >> 1) & 1, c >> 2], device=DEV)
        want = _pack(blocks + step)
        at = torch.searchsorted(keys, want).clamp(max=len(keys) - 1)
        there = keys[at] == want
        to = tuple(slice(8, 9) if (c >> j) & 1 else slice(0, 8) for j in (2, 1, 0))
        of = tuple(slice(0, 1) if (c >> j) & 1 else slice(0, 8) for j in (2, 1, 0))
        part = grid[at][(slice(None), *of)]
        tile[(slice(None), *to)] = torch.where(there[:, None, None, None], part, float("nan"))
    val = torch.stack([tile[:, (c >> 2):(c >> 2) + 8, ((c >> 1) & 1):((c >> 1) & 1) + 8,
                            (c & 1):(c & 1) + 8].reshape(-1) for c in range(8)], 1)
    cube = torch.nonzero(~torch.isnan(val).any(1)).reshape(-1)
    val = val[cube]
    l = cube % 512
    base = blocks[cube // 512] * 8 + torch.stack([l & 7, (l >> 3) & 7, l >> 6], 1)
    tris, cells = [], []
    for t, tet in enumerate(TETS):
        mask = sum((val[:, c] < 0).long() << j for j, c in enumerate(tet))
        for m in range(1, 15):
            at = torch.nonzero(mask == m).reshape(-1)
            for k, tri in enumerate(_tet_triangles(m)):
                corners = []
                for a, b in tri:
                    a, b = tet[a], tet[b]
                    lo, hi = (a, b) if a & b == a else (b, a)
                    f = val[at, lo] / (val[at, lo] - val[at, hi])
                    for j in range(3):
                        p = base[at, j].double() + ((lo >> j) & 1) + 0.5
                        corners.append((p + f * (((hi >> j) & 1) - ((lo >> j) & 1))) * v)
                tris.append(torch.stack(corners, 1))
                cells.append(torch.cat([base[at], torch.full((len(at), 1), 2 * t + k, device=DEV)], 1))
    tris, c = torch.cat(tris), torch.cat(cells)
    cells, order = _cell_order(c)
    return {"tris": tris[order], "cells": cells}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("track", "stages"):
        view = _view(case["width"], case["height"], case["colour"], seed, 0)
        return _exact_maps([view], case, _map_keys(case, seed))
    if kind == "stream":
        return _exact_maps(_frames_of(case, seed), case, _map_keys(case, seed, views=case["frames"]))
    if kind == "batch":
        return [_exact_maps([_view(w, h, case["colour"], seed + 31 * i, 0)], case,
                            _map_keys(case, seed + 31 * i, w, h))
                for i, (w, h) in enumerate(_sessions(case))]
    if kind == "scan":
        views = _frames_of(case, seed)
        keys = torch.unique(torch.cat([_contributions(v, case["voxel"], case["band"])[0] for v in views]))
        room = _map_size(case, views=case["frames"])[0] - len(keys)
        out = {"coords": _unpack(keys).int(), **_exact_maps(views, case, keys)}
        return {"blocks": len(keys),
                **{k: torch.cat([x, x.new_zeros(room, *x.shape[1:])]) for k, x in out.items()}}
    return _exact_mesh(case, seed)


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _fusion_work(views, case):
    """Bytes and operations of fusing frames into one map: the images, a table entry for each
    block, and every voxel that a frame touches read and written once; the walk of a point's band
    (about 60 operations a sample) and five additions a contribution."""
    b = f = 0.0
    for view in views:
        depth, rgb = view[0], view[1]
        key, local, _, _ = _contributions(view, case["voxel"], case["band"])
        touched = len(torch.unique(key * 512 + local))
        b += depth.numel() * (7 if rgb is not None else 4) + len(torch.unique(key)) * 16
        b += touched * 2 * (20 if rgb is not None else 8)
        points = int((torch.isfinite(depth) & (depth > 0)).sum())
        f += points * (2 * case["band"] + 1) * 60 + len(key) * (5 if rgb is not None else 2)
    return b, f


def work(case):
    kind, seed = case["kind"], 1
    if kind == "batch":
        views = [_view(w, h, case["colour"], seed + 31 * i, 0)
                 for i, (w, h) in enumerate(_sessions(case))]
    elif kind == "mesh":
        keys = _map_keys(case, 0)
        c = _exact_mesh(case, seed)["cells"]
        # the blocks' sums and coordinates read; triangles and cells written, then put in order
        return {"bytes": float(len(keys) * (512 * 16 + 16) + len(c) * (52 + 52 + 44)),
                "flops": float(len(keys) * 512 * 8 + len(c) * 60)}
    else:
        views = _frames_of(case, seed)
    b, f = _fusion_work(views, case)
    if kind == "scan":  # the map comes out in key order: each block read and written once more
        n = len(torch.unique(torch.cat([_contributions(v, case["voxel"], case["band"])[0] for v in views])))
        b += 2 * n * (512 * (20 if case["colour"] else 16) + 12)
    return {"bytes": float(b), "flops": float(f)}
