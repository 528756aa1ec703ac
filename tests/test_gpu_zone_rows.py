"""The zone solver by rows at the sizes where it can go wrong, against the
float64 oracle: one warp's edge (31 to 33 rows), the half and whole CTA's row
counts (255 to 257, 512, 1,023 to 1,025, 1,536 and 1,537), zones whose matrix
does not fit shared memory (a fan: every row shares the hub, so a matrix of n
rows has n^2 entries) and, with block_switch_iters=1, the hand-over of a large
zone to the blocks.  Every row has its own x0, so the systems are positive
definite with condition numbers below ~n / 9; the tolerance is the other
solver tests'."""
import numpy as np
import pytest

import oracle
from gpu_util import dev_mesh, rel_err, respond

pytestmark = pytest.mark.gpu

TOL_DX = 1e-6


def strip(n, y0, base):
    """n faces of a strip (the last one dropped when n is odd)."""
    L = (n + 1) // 2
    V = [(0.1 * i, y0 + 0.1 * j, 0.0) for i in range(L + 1) for j in range(2)]
    T = []
    for i in range(L):
        a = base + 2 * i
        T += [(a, a + 2, a + 1), (a + 1, a + 2, a + 3)]
    return V, T[:n]


def fan(n, y0, base):
    """n faces around one hub."""
    t = 2 * np.pi * np.arange(n) / n
    V = [(0.0, y0, 0.0)] + [(np.cos(x), y0 + np.sin(x), 0.0) for x in t]
    return V, [(base, base + 1 + i, base + 1 + (i + 1) % n) for i in range(n)]


CASES = {
    "warp_edge": ([("s", n) for n in (1, 2, 31, 32, 33, 31, 32, 33)], 48),
    "half_edge": ([("s", n) for n in (64, 255, 256, 257, 256)], 48),
    "cta_edge": ([("s", n) for n in (511, 512, 513, 1023, 1024, 1025)], 48),
    "rows_limit": ([("s", n) for n in (1536, 1537)], 48),
    "fan_small": ([("f", n) for n in (8, 24, 32, 60, 80, 90)], 48),
    "fan_dense": ([("f", n) for n in (120, 256, 400)], 48),
    "fan_large": ([("f", 1200)], 48),
    "hand_over": ([("s", n) for n in (1024, 1300, 1536)], 1),
    "no_blocks": ([("s", n) for n in (300, 1300)], 0),
}


@pytest.mark.parametrize("name", CASES)
def test_rows_solver_against_oracle(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2081_gb300 import api
    zones, switch = CASES[name]
    rng = np.random.default_rng(len(name))
    V, T = [], []
    for i, (kind, n) in enumerate(zones):
        v, t = (strip if kind == "s" else fan)(n, 3.0 * i, len(V))
        V += v
        T += t
    VB = np.array(V) + rng.uniform(-0.002, 0.002, (len(V), 3))
    TB = np.array(T, np.int32)
    k = len(TB)
    VA = VB[TB].mean(axis=1) + np.array([0.0, 0.0, -0.02]) + rng.uniform(-0.005, 0.005, (k, 3))
    TA = np.array([[0, 1, 2]], np.int32)
    if k < 3:
        VA = np.concatenate([VA, VA[-1:] + 1.0])
    A, PA = dev_mesh(api, VA, TA, False, np.float32)
    B, PB = dev_mesh(api, VB, TB, True, np.float32)
    st = np.zeros((k, 4), np.int32)
    st[:, 1] = np.arange(k)
    st[:, 2] = np.arange(k)
    ctx = api.Context(block_switch_iters=switch)
    ctx.hfcr_reserve(max(len(VA), len(VB)), max(len(TA), len(TB)), 1 << 14)
    g, info = respond(ctx, A, B, torch.tensor(st, device="cuda:0"), k, 1e-4, len(VA), len(VB), np.float32)
    assert info.converged and info.n_stencils == k and info.rel_residual <= 1e-12
    rA, rB, _, sol = oracle.respond(st[:, :3].astype(np.uint32), PA, TA, PB, TB, 1e-4)
    assert sol.n_zones == len(zones)
    assert rel_err(g, np.concatenate([rA, rB])) <= TOL_DX
