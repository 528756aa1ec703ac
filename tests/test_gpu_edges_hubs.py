"""Vertices of many half-edges in the bucket form of the edge lists: where a
list passes from a thread to a warp (32), to the CTA's bitmap (128), beyond
what shared memory holds (3,968) and beyond what a rank counts (65,535);
neighbours spread over several passes of the bitmap (126,976 ids each), hubs
that share a block of 256 vertices, the number of them that sends the call to
the sort, and large meshes, whose first try (four launches) leaves hubs to a
second.  Against numpy's sorted unique pairs; the route by the launches."""
import numpy as np
import pytest

from tests.test_gpu_edges import api, fan, reference  # noqa: F401

pytestmark = pytest.mark.gpu
RNG = np.random.default_rng(21)


def shuffled(T):
    """The triangles in any order, corners rotated, a tenth of them twice."""
    T = np.concatenate([T, T[RNG.integers(0, len(T), max(len(T) // 10, 1))]])
    T = T[RNG.permutation(len(T))]
    return np.take_along_axis(T, (np.arange(3) + RNG.integers(0, 3, (len(T), 1))) % 3, 1)


def sphere(lon, lat=5):
    """Rings of lon vertices between two poles, a pole first and last."""
    ring = 1 + np.arange(lat * lon).reshape(lat, lon)
    a, b = ring[:-1], ring[1:]
    an, bn = np.roll(a, -1, 1), np.roll(b, -1, 1)
    quads = [np.stack([a, b, bn], -1).reshape(-1, 3), np.stack([a, bn, an], -1).reshape(-1, 3)]
    top = np.stack([np.zeros(lon, int), ring[0], np.roll(ring[0], -1)], 1)
    end = np.stack([np.full(lon, 1 + lat * lon), np.roll(ring[-1], -1), ring[-1]], 1)
    return np.concatenate([top, *quads, end])


def hubs(n, k, spread):
    """n hubs 0 .. n - 1 of k triangles each over `spread` other ids."""
    o = n + RNG.integers(0, spread, (n * k, 2))
    return np.concatenate([np.repeat(np.arange(n), k)[:, None], o], 1)


LISTS = {f"fan_{k}": (fan(k), 4) for k in (15, 16, 17, 63, 64, 65, 128, 1983, 1984, 1985, 15000)}
LISTS |= {f"mixed_{k}": (shuffled(fan(k)), 4) for k in (17, 60, 300, 3000, 15000)}
LISTS |= {f"sphere_{k}": (sphere(k), 4) for k in (20, 100, 1000, 3000)}
LISTS |= {
    "spread_1000": (hubs(1, 1000, 290_000), 4), "spread_100": (hubs(3, 100, 100_000), 4),
    "hubs_60": (hubs(60, 17, 4000), 4), "hubs_8": (hubs(8, 200, 900), 4), "hubs_5": (hubs(5, 700, 4000), 4),
    "too_many": (hubs(256, 17, 4000), 0), "too_many_hubs": (hubs(30, 1000, 4000), 0),
    "large": (sphere(16, 3200), 4), "large_17": (sphere(17, 3000), 8), "large_hub": (sphere(1000, 60), 8),
    "large_fan": (np.concatenate([sphere(40, 1600), 70_000 + fan(40_000)]), 0),
    "fan_32768": (fan(32768), 0), "fan_70000": (fan(70000), 0),
}


@pytest.mark.parametrize("name", sorted(LISTS))
def test_hubs(api, name):  # noqa: F811
    import torch
    T, launches = LISTS[name]  # 0: the sort's
    T = T.astype(np.int32)
    nv = int(T.max()) + 1
    ref = reference(T)
    tris = torch.tensor(T, device="cuda:0")
    ctx = api.Context()
    ctx.hfcr_reserve(nv, len(T), 16)
    for cap in (3 * len(T), len(ref)):
        out = torch.full((cap, 2), -7, dtype=torch.int32, device="cuda:0")
        n0 = api.hfcr_launch_count()
        n = ctx.hfcr_build_edges(tris, nv, out)
        n0 = api.hfcr_launch_count() - n0
        assert n0 == launches or (launches == 0 and n0 > 8)
        got = out.cpu().numpy()
        assert n == len(ref) and np.array_equal(got[:n], ref)
        assert (got[n:] == -7).all()
    ctx.close()
