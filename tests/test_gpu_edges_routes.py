"""Each mesh of a call takes its own route to its edge list: a mesh that the
buckets give up on (a hub of more half-edges than they count) does not send
the other one to the sort; and a short list over many vertex ids goes to the
sort, which does not pass over the ids.  By the launches of the calls."""
import numpy as np
import pytest

from tests.gpu_util import detect, dev_mesh
from tests.test_gpu_edges import api, fan, reference  # noqa: F401
from tests.test_gpu_hierarchy import soup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hub", ["A", "B"])
def test_a_hub_beside_an_ordinary_mesh(api, hub):  # noqa: F811
    k = 40_000
    phi = 2 * np.pi * np.arange(k) / k
    V = np.concatenate([[[0.5, 0.5, 2.0]], np.stack([0.5 + np.cos(phi), 0.5 + np.sin(phi), 0 * phi - 0.5], 1)])
    rng = np.random.default_rng(11)
    meshes = [(V, fan(k).astype(np.int32)), soup(rng, 300, 0.3)]
    if hub == "B":
        meshes.reverse()
    count, rec = {}, {}
    for own in ("", "A", "B", "AB"):  # the meshes whose lists the call derives
        A, PA = dev_mesh(api, *meshes[0], True, np.float32, edges="A" not in own)
        B, PB = dev_mesh(api, *meshes[1], True, np.float32, edges="B" not in own)
        ctx = api.Context(bvh_rebuild_interval=1000)
        ctx.hfcr_reserve(k + 1, k, 1 << 20)
        detect(ctx, A, B, 1 << 20)  # builds the hierarchies and the traversal orders
        n0 = api.hfcr_launch_count()
        rec[own] = detect(ctx, A, B, 1 << 20)[2]
        count[own] = api.hfcr_launch_count() - n0
        ctx.close()
    assert len(rec[""]) > 0 and all(np.array_equal(r, rec[""]) for r in rec.values())
    assert count["AB"] - count[""] == (count["A"] - count[""]) + (count["B"] - count[""])


@pytest.mark.parametrize("nt,line", [(100, 300_000), (2730, 300_000), (2731, 1_013_655), (9000, 1_045_000)])
def test_many_ids_few_triangles(api, nt, line):  # noqa: F811
    import torch
    rng = np.random.default_rng(nt)
    for nv in (line, line + 1):
        T = rng.integers(0, nv, (nt, 3)).astype(np.int32)
        T[0, 0], T[1, 1] = nv - 1, 0
        ref = reference(T)
        ctx = api.Context()
        ctx.hfcr_reserve(nv, nt, 16)
        out = torch.full((3 * nt, 2), -7, dtype=torch.int32, device="cuda:0")
        n0 = api.hfcr_launch_count()
        n = ctx.hfcr_build_edges(torch.tensor(T, device="cuda:0"), nv, out)
        n0 = api.hfcr_launch_count() - n0
        got = out.cpu().numpy()
        assert n == len(ref) and np.array_equal(got[:n], ref) and (got[n:] == -7).all()
        assert (n0 == 4) == (nv == line)
        ctx.close()
