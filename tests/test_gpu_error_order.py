"""Which error a call reports when a mesh has several faults: positions that
are not finite or out of range come before an index out of range, whether the
edge lists are the caller's or derived by the call."""
import numpy as np
import pytest

from tests.gpu_util import dev_mesh, torch_dev
from tests.test_gpu_edges import api  # noqa: F401

pytestmark = pytest.mark.gpu

V = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], float)
T = np.array([[0, 2, 1], [0, 1, 3], [1, 2, 3], [0, 3, 2]], np.int32)


def scene(api, fault, edges):  # noqa: F811
    A, _ = dev_mesh(api, V, T, True, np.float32, edges=edges)
    B, _ = dev_mesh(api, V + 0.25, T, True, np.float32, edges=edges)
    if "index" in fault:
        A.tris[2, 1] = 9
    if "nan" in fault:
        B.y[3] = float("nan")
    if "range" in fault:
        A.z[1] = 2.0 ** 39
    return A, B


@pytest.mark.parametrize("edges", [False, True])
@pytest.mark.parametrize("fault,code", [("index", "ARG"), ("index nan", "NONFINITE"), ("index range", "RANGE"),
                                        ("index range nan", "NONFINITE"), ("nan", "NONFINITE")])
def test_positions_before_indices(api, fault, code, edges):  # noqa: F811
    import torch
    A, B = scene(api, fault, edges)
    ctx = api.Context()
    ctx.hfcr_reserve(4, 4, 64)
    out = torch.zeros((64, 4), dtype=torch.int32, device=torch_dev())
    for call in (lambda: ctx.hfcr_detect(A, B, out), lambda: ctx.hfcr_resolve(A, B, 1e-3, 4),
                 lambda: ctx.hfcr_autotune(A, B)):
        with pytest.raises(api.HfcrError) as e:
            call()
        assert e.value.status == getattr(api, "HFCR_ERR_" + code)
    ctx.close()
