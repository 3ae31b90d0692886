"""Surface extraction on made-up voxel sums, cube by cube: random signs over a
cluster of blocks (every inside mask of a cube occurs, across block faces, edges
and corners), with unobserved voxels, absent blocks and NaN sums left out of the
surface. Against a plain statement of marching tetrahedra in 64 bits: the same
triangles by name, vertices on the same edges, normals towards positive values.

Vertices: t = v_lo / (v_lo - v_hi) is one float32 subtraction and division of
means with 2^-24 relative error, so t is off by at most 4 * 2^-24 and a
coordinate by that times the 1 cm edge plus 2^-23 of its size (below 0.5 m):
3e-8 + 6e-8 < 1e-7.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2608_08287_gb300 import tsdf
from test_gpu_parity import _built  # noqa: F401

pytestmark = pytest.mark.gpu

V = np.float32(0.01)
TETS = ((0, 1, 3, 7), (0, 1, 7, 5), (0, 2, 7, 3), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 7, 6))


def made_volume(blocks, sums, slots):
    """A volume holding the given blocks (n, 3) and sums (n, 512, 4)."""
    n = len(blocks)
    mem = torch.empty(tsdf.tsdf_volume_bytes(slots, n), dtype=torch.uint8, device="cuda")
    vol = tsdf.Volume(float(V), 4 * float(V), slots, n, memory=mem)
    lay = vol.layout()
    table = np.full((slots, 2), -1, np.int64)
    for i, b in enumerate(blocks):
        s = tsdf.tsdf_block_slot(int(b[0]), int(b[1]), int(b[2]), slots)
        while table[s, 0] != -1:
            s = (s + 1) % slots
        table[s, 0] = tsdf.tsdf_block_key(int(b[0]), int(b[1]), int(b[2]))
        table[s, 1] = (-1 << 32) | i
    for at, a in ((lay.table_offset, table), (lay.coords_offset, blocks.astype(np.int32)),
                  (lay.voxel_sums_offset, sums.astype(np.float32)),
                  (0, np.array([n], np.uint32))):
        b = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1).copy()).cuda()
        mem[at:at + len(b)] = b
    return vol, mem


@pytest.mark.parametrize("hidden,nan", [(0.0, 0.0), (0.05, 0.0), (0.4, 0.02)])
@pytest.mark.parametrize("origin", [(0, 0, 0), (-1, 2, -2)])
def test_cubes(hidden, nan, origin):
    rs = np.random.RandomState(int(100 * hidden) + origin[1])
    side = 3
    every = np.array([(x, y, z) for x in range(side) for y in range(side) for z in range(side)])
    kept = every[rs.permutation(len(every))[:len(every) - 4]]
    mean = rs.uniform(-1, 1, (8 * side,) * 3)               # x, y, z
    seen = rs.uniform(0, 1, mean.shape) >= hidden
    bad = rs.uniform(0, 1, mean.shape) < nan
    weight = rs.randint(1, 6, mean.shape)
    there = np.zeros(mean.shape, bool)
    sums = np.zeros((len(kept), 512, 4), np.float32)
    l = np.arange(512)
    for i, b in enumerate(kept):
        gx, gy, gz = 8 * b[0] + (l & 7), 8 * b[1] + ((l >> 3) & 7), 8 * b[2] + (l >> 6)
        there[gx, gy, gz] = True
        w = np.where(seen[gx, gy, gz], weight[gx, gy, gz], 0)
        sums[i, :, 0] = np.where(bad[gx, gy, gz], np.nan, np.float32(mean[gx, gy, gz]) * w)
        sums[i, :, 1] = w
    mean = np.float32(np.float32(mean) * weight.astype(np.float32)) / weight.astype(np.float32)
    ok = there & seen & ~bad
    vol, mem = made_volume(kept + np.array(origin), sums, 1 << 9)
    tris, cells, _ = vol.extract_mesh()
    vol.close()
    want = {}
    edge = 8 * side
    for x, y, z in np.argwhere(ok[:-1, :-1, :-1]):
        c = [(x + (k & 1), y + ((k >> 1) & 1), z + (k >> 2)) for k in range(8)]
        if max(max(p) for p in c) >= edge or not all(ok[p] for p in c):
            continue
        f = [float(mean[p]) for p in c]
        for t, tet in enumerate(TETS):
            n_in = sum(f[k] < 0 for k in tet)
            cuts = [(a, b) for i, a in enumerate(tet) for b in tet[i + 1:] if (f[a] < 0) != (f[b] < 0)]
            pts = []
            for a, b in cuts:
                r = f[a] / (f[a] - f[b])
                pa, pb = np.array(c[a], float) + 0.5, np.array(c[b], float) + 0.5
                pts.append((pa + r * (pb - pa) + 8 * np.array(origin)) * float(V))
            up = np.array([c[k] for k in tet if f[k] >= 0], float)
            down = np.array([c[k] for k in tet if f[k] < 0], float)
            for k in range(0 if n_in in (0, 4) else (2 if n_in == 2 else 1)):
                name = (*(int(g) + 8 * o for g, o in zip((x, y, z), origin)), 2 * t + k)
                want[name] = (np.array(pts), up.mean(0) - down.mean(0) if n_in in (1, 2, 3) else None)
    got = {tuple(int(q) for q in cell): tri for cell, tri in zip(cells, tris)}
    assert len(got) == len(cells)
    assert set(got) == set(want)
    for name, tri in got.items():
        pts, up = want[name]
        d = np.abs(tri[:, None].astype(np.float64) - pts[None]).max(2)
        assert (d.min(1) <= 1e-7).all()
        a = np.cross(tri[1].astype(np.float64) - tri[0], tri[2].astype(np.float64) - tri[0])
        assert a @ up > -1e-10
