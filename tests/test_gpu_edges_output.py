"""Where hfcr_build_edges puts its list: an output that starts at an odd
multiple of 4 bytes (an int32_t * promises no more), with room for every
possible edge or for just the ones there are, and outputs that a failing call
must leave as they were.  By buckets, by the sort that a vertex of more half-
edges than a bucket takes, and by the sort of more vertices than reserved."""
import numpy as np
import pytest

from tests.test_gpu_edges import api, fan, reference  # noqa: F401

pytestmark = pytest.mark.gpu


def mesh(name):
    T = fan(400) if name == "fan" else np.random.default_rng(5).integers(0, 700, (900, 3))
    return T.astype(np.int32), int(T.max()) + 1


@pytest.mark.parametrize("name", ["random", "fan"])
@pytest.mark.parametrize("reserve", ["vertices", "few"])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_output_at_any_int(api, name, reserve, shift):  # noqa: F811
    import torch
    T, nv = mesh(name)
    ref = reference(T)
    tris = torch.tensor(T, device="cuda:0")
    ctx = api.Context()
    ctx.hfcr_reserve(nv if reserve == "vertices" else 1, len(T), 16)
    for cap in (3 * len(T), len(ref)):
        buf = torch.full((2 * cap + 8,), -7, dtype=torch.int32, device="cuda:0")
        out = buf[shift:shift + 2 * cap].view(cap, 2)
        assert out.data_ptr() % 8 == 4 * (shift % 2)
        n = ctx.hfcr_build_edges(tris, nv, out)
        got = buf.cpu().numpy()
        assert n == len(ref) and np.array_equal(got[shift:shift + 2 * n].reshape(n, 2), ref)
        assert (got[:shift] == -7).all() and (got[shift + 2 * n:] == -7).all()
    ctx.close()


@pytest.mark.parametrize("name", ["random", "fan"])
@pytest.mark.parametrize("reserve", ["vertices", "few"])
def test_failing_call_leaves_the_output(api, name, reserve):  # noqa: F811
    import torch
    T, nv = mesh(name)
    T[len(T) // 2, 1] = nv + 3
    tris = torch.tensor(T, device="cuda:0")
    ctx = api.Context()
    ctx.hfcr_reserve(nv if reserve == "vertices" else 1, len(T), 16)
    out = torch.full((3 * len(T), 2), -7, dtype=torch.int32, device="cuda:0")
    with pytest.raises(api.HfcrError) as e:
        ctx.hfcr_build_edges(tris, nv, out)
    assert e.value.status == api.HFCR_ERR_ARG
    assert (out.cpu().numpy() == -7).all()
    ctx.close()


@pytest.mark.parametrize("name", ["random", "fan"])
def test_output_over_the_triangles(api, name):  # noqa: F811
    """The list may replace the triangles it is made from."""
    import torch
    T, nv = mesh(name)
    ref = reference(T)
    buf = torch.zeros((3 * len(T), 2), dtype=torch.int32, device="cuda:0")
    tris = buf.view(-1)[:3 * len(T)].view(-1, 3)
    tris.copy_(torch.tensor(T))
    ctx = api.Context()
    ctx.hfcr_reserve(nv, len(T), 16)
    n = ctx.hfcr_build_edges(tris, nv, buf)
    assert n == len(ref) and np.array_equal(buf[:n].cpu().numpy(), ref)
    ctx.close()
