"""Edge lists by buckets of the smaller vertex, and where the radix sort takes
over: valences around the bucket limit of 128, a block of 256 vertices around
what its shared memory holds (4,096 half-edges), fans, repeated and degenerate
triangles, isolated vertices, more vertices than reserved, short output
buffers, and the sort's own change from ranks to passes at 8,192 keys.  Against numpy's sorted unique pairs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2081_gb300 import api as a
    a.lib()
    return a


def reference(T):
    e = np.concatenate([T[:, [0, 1]], T[:, [1, 2]], T[:, [2, 0]]]).astype(np.int64)
    return np.unique(np.sort(e, 1), axis=0)


def fan(k):
    """k triangles around vertex 0: 0 is the smaller vertex of 2 k half-edges."""
    i = np.arange(1, k + 1)
    return np.stack([np.zeros(k, int), i, i % k + 1], 1)


def dense(rng, nv, per):
    """Triangles whose smallest vertex runs over all nv vertices `per` times."""
    a = np.repeat(np.arange(nv), per)
    return np.stack([a, nv + rng.integers(0, 500, len(a)), nv + 500 + rng.integers(0, 500, len(a))], 1)


RNG = np.random.default_rng(3)
LISTS = {
    "one": np.array([[2, 0, 1]]),
    "degenerate": np.array([[0, 0, 0], [1, 1, 2], [2, 1, 1], [3, 4, 5], [5, 4, 3]]),
    "fan_64": fan(64), "fan_65": fan(65), "fan_5000": fan(5000),
    # three keys a triangle into the sort: 8,190 by ranks, 8,193 by passes
    "fan_2730": fan(2730), "fan_2731": fan(2731),
    "random": RNG.integers(0, 900, (3000, 3)),
    "dense_7": dense(RNG, 300, 7), "dense_8": dense(RNG, 256, 8), "dense_9": dense(RNG, 600, 9),
    "dense_60": dense(RNG, 300, 60),
    "sparse_ids": RNG.integers(0, 200_000, (257, 3)),
    "scan_edge": np.stack([np.arange(4095), np.arange(4095) + 1, np.full(4095, 4096)], 1),
}


@pytest.mark.parametrize("name", sorted(LISTS))
@pytest.mark.parametrize("reserve", ["vertices", "few"])
def test_edges(api, name, reserve):
    import torch
    T = LISTS[name].astype(np.int32)
    nv = int(T.max()) + 1 + (5 if name == "random" else 0)
    ctx = api.Context()
    ctx.hfcr_reserve(nv if reserve == "vertices" else 1, len(T), 16)
    ref = reference(T)
    tris = torch.tensor(T, device="cuda:0")
    for rep in range(2):
        for cap in (3 * len(T) + 4, len(ref)):
            out = torch.full((cap, 2), -7, dtype=torch.int32, device="cuda:0")
            n = ctx.hfcr_build_edges(tris, nv, out)
            got = out.cpu().numpy()
            assert n == len(ref) and np.array_equal(got[:n], ref)
            assert (got[n:] == -7).all()
    with pytest.raises(api.HfcrError):
        ctx.hfcr_build_edges(tris, nv - 6 if name == "random" else nv - 1, out)
    ctx.close()
