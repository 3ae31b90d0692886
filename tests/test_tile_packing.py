"""The tile kernel's packed voxels and directory tags in plain integers (CPU):
words of a band's samples are equal exactly when their voxels are, and the
local index, the block tag and the key rebuilt from the tag are those of the
voxel, over the whole range that the kernel packs."""
import numpy as np

MAGIC = 0x4B400000
BIAS = 1 << 20
M32 = (1 << 32) - 1


def word(g):
    b = (g + MAGIC).astype(np.int64)
    return (b[..., 0] + (b[..., 1] << 10) + (b[..., 2] << 20)) & M32


def test_packed_voxels_and_tags():
    rs = np.random.RandomState(0)
    n = 20000
    lim = 1 << 22
    g0 = rs.randint(-lim + 40, lim - 40, (n, 3))          # a point's first voxel
    g0[:200] = rs.choice([-lim + 40, lim - 41, -1, 0, 7, 8], (200, 3))
    g = g0[:, None] + np.arange(34)[None, :, None] * rs.choice([-1, 0, 1], (n, 1, 3))
    tile = (g0 >> 3) + rs.randint(-500, 501, (n, 3))      # the tile's base block
    aligned = (g0 + MAGIC) & ~7
    base = (aligned[:, 0] - 512) + ((aligned[:, 1] - 512) << 10) + ((aligned[:, 2] - 512) << 20)
    p = (word(g) - base[:, None]) & M32
    same = (g[:, 1:] == g[:, :-1]).all(2)
    assert np.array_equal(p[:, 1:] == p[:, :-1], same)
    local = (((p & 0x00701C07) * ((1 << 14) + (1 << 7) + 1) & M32) >> 14) & 511
    assert np.array_equal(local, (g[..., 0] & 7) | ((g[..., 1] & 7) << 3) | ((g[..., 2] & 7) << 6))
    block = (p >> 3) & 0x07F1FC7F
    assert (block != 0).all()
    dd = ((aligned - (MAGIC - 8 * BIAS)) >> 3) - (tile + BIAS)
    delta = (dd[:, 0] + 448) + ((dd[:, 1] + 448) << 10) + ((dd[:, 2] + 1984) << 20)
    tag = (block + delta[:, None]) & M32
    assert (tag != M32).all()
    back = np.stack([tag & 1023, (tag >> 10) & 1023, tag >> 20], 2) - np.array([512, 512, 2048])
    assert np.array_equal(back + tile[:, None], g >> 3)


def test_floor_by_directed_addition():
    """x + 1.5 * 2^23 rounded down is the floor, for every float within 2^22."""
    rs = np.random.RandomState(1)
    x = np.concatenate([rs.uniform(-2.0 ** 22, 2.0 ** 22, 100000), rs.uniform(-4, 4, 100000),
                        np.float32(10.0) ** rs.uniform(-40, 6, 1000), [-2.0 ** 22, 0.0, -0.0, -1e-45]])
    x = np.float32(x)
    x = x[np.abs(x) <= 2 ** 22]
    exact = x.astype(np.longdouble) + np.longdouble(12582912.0)
    down = exact.astype(np.float32)
    down = np.where(down.astype(np.longdouble) > exact, np.nextafter(down, np.float32(-np.inf)), down)
    # (the sum of a tiny x needs more bits than a long double has: its floor decides)
    tiny = (np.abs(x) < 1e-10) & (x < 0)
    down = np.where(tiny, np.float32(12582911.0), down)
    assert np.array_equal(down.view(np.uint32).astype(np.int64) - MAGIC, np.floor(x).astype(np.int64))
