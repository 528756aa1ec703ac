"""The float64 solver of the zones that the float32 runs leave above the target,
staged in shared memory, at the sizes where it can go wrong: one row, a warp's
edge, the threads with rows (255 to 257) and with vertices (479 to 481), the
most rows it takes (1,024) and more, fans (every row shares the hub), rows
sharing x0 (blocks of up to four) and inverse masses.  One refinement round
leaves every zone above a relative residual of 1e-12, so every zone is solved
again.  Against the float64 oracle, at the float64 solvers' tolerance."""
import numpy as np
import pytest

import oracle
from gpu_util import dev_mesh, rel_err, respond

pytestmark = pytest.mark.gpu

TOL_DX = 1e-9

# faces of each fan, faces of each strip, rows per x0
SYSTEMS = {
    "small": ([], [1, 2, 31, 32, 33, 64], 1),
    "threads": ([], [255, 256, 257, 479, 480, 481], 1),
    "limit": ([], [1023, 1024, 1025], 1),
    "fans": ([8, 60, 120, 300], [5], 1),
    "blocks": ([], [9, 40, 500], 2),
}


@pytest.mark.parametrize("masses", [False, True], ids=["unit", "masses"])
@pytest.mark.parametrize("name", SYSTEMS)
def test_rescued_zones_against_oracle(name, masses):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2081_gb300 import api
    fans, strips, share = SYSTEMS[name]
    rng = np.random.default_rng(len(name))
    V, T = [], []
    for i, n in enumerate(fans):
        base, t = len(V), 2 * np.pi * np.arange(n) / n
        V += [(0.0, 3.0 * i, 0.0)] + [(np.cos(x), 3.0 * i + np.sin(x), 0.0) for x in t]
        T += [(base, base + 1 + j, base + 1 + (j + 1) % n) for j in range(n)]
    for i, n in enumerate(strips):
        base, L = len(V), (n + 1) // 2
        V += [(0.1 * c, -1.0 - 0.5 * i + 0.1 * j, 0.0) for c in range(L + 1) for j in range(2)]
        quads = [((base + 2 * c, base + 2 * c + 2, base + 2 * c + 1),
                  (base + 2 * c + 1, base + 2 * c + 2, base + 2 * c + 3)) for c in range(L)]
        T += [t for q in quads for t in q][:n]
    VB = np.array(V) + rng.uniform(-0.002, 0.002, (len(V), 3))
    TB = np.array(T, np.int32)
    k = len(TB)
    x0 = np.arange(k) // share
    VA = np.array([VB[TB[x0 == v]].mean(axis=(0, 1)) for v in range(x0[-1] + 1)])
    VA = np.concatenate([VA + np.array([0.0, 0.0, -0.02]), VA[-1:] + 1.0, VA[-1:] + 2.0])
    TA = np.array([[0, 1, 2]], np.int32)
    wA, wB = (rng.uniform(0.5, 2.0, len(v)).astype(np.float32) if masses else None for v in (VA, VB))
    A, PA = dev_mesh(api, VA, TA, False, np.float64, inv_mass=wA)
    B, PB = dev_mesh(api, VB, TB, True, np.float64, inv_mass=wB)
    st = np.zeros((k, 4), np.int32)
    st[:, 1] = x0
    st[:, 2] = np.arange(k)
    ctx = api.Context(max_refine=1, max_cg_iters=2000)
    ctx.hfcr_reserve(max(len(VA), len(VB)), max(len(TB), 1), 1 << 14)
    g, info = respond(ctx, A, B, torch.tensor(st, device="cuda:0"), k, 1e-4, len(VA), len(VB), np.float64)
    assert info.converged and info.n_stencils == k and info.rel_residual <= 1e-12
    w = np.concatenate([wA, wB]).astype(np.float64) if masses else None
    rA, rB, _, _ = oracle.respond(st[:, :3].astype(np.uint32), PA, TA, PB, TB, 1e-4, w)
    assert rel_err(g, np.concatenate([rA, rB])) <= TOL_DX
