"""The setup of up to 4,096 stencils in one CTA (setup_path 0) against the
sequence of kernels (setup_path 1), at the sizes where it can go wrong: one
stencil, the CTA's thread count and its multiples, its limit and the first
size above; vertex lists of 16, 17, 128 and 129 entries and of hundreds
(fans: the hub is in every row); runs of rows sharing x0 longer than a group;
one zone and thousands; inverse masses.  Sums over a list and over a zone's
rows have the same order on both paths, so the displacements are the same
bits."""
import numpy as np
import pytest

from gpu_util import dev_mesh, respond

pytestmark = pytest.mark.gpu

# faces of each fan, faces of each strip, rows per x0
SYSTEMS = {
    "one": ([], [1], 1),
    "two_zones": ([], [1, 1], 1),
    "threads": ([], [1023], 1),
    "threads_even": ([], [512, 512], 1),
    "threads_odd": ([], [1000, 25], 1),
    "single_rows": ([], [1] * 2049, 1),
    "limit_less_one": ([], [15] * 273, 1),
    "limit": ([], [16] * 256, 1),
    "above": ([], [16] * 256 + [1], 1),
    "lists": ([8, 16, 17, 32, 128, 129], [40], 1),
    "long_lists": ([400, 700, 129], [7] * 20, 1),
    "shared_x0": ([12], [9, 14, 200], 7),
    "pairs_x0": ([], [300, 2, 1, 500], 2),
}


@pytest.mark.parametrize("masses", [False, True], ids=["unit", "masses"])
@pytest.mark.parametrize("name", SYSTEMS)
def test_paths_identical(name, masses):
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
    perm = rng.permutation(len(V))                  # vertex ids in no particular order
    VB = (np.array(V) + rng.uniform(-0.002, 0.002, (len(V), 3)))[np.argsort(perm)]
    TB = perm[np.array(T)].astype(np.int32)
    k = len(TB)
    x0 = np.arange(k) // share
    VA = np.array([VB[TB[x0 == v]].mean(axis=(0, 1)) for v in range(x0[-1] + 1)] if share > 1
                  else VB[TB].mean(axis=1)) + np.array([0.0, 0.0, -0.02])
    VA = np.concatenate([VA, VA[-1:] + 1.0, VA[-1:] + 2.0])
    wA, wB = (rng.uniform(0.5, 2.0, len(v)) if masses else None for v in (VA, VB))
    A, _ = dev_mesh(api, VA, np.array([[0, 1, 2]], np.int32), False, np.float32, inv_mass=wA)
    B, _ = dev_mesh(api, VB, TB, True, np.float32, inv_mass=wB)
    st = np.zeros((k, 4), np.int32)
    st[:, 1] = x0
    st[:, 2] = np.arange(k)
    got = []
    for path in (0, 1):
        ctx = api.Context(setup_path=path)
        ctx.hfcr_reserve(max(len(VA), len(VB)), max(len(TB), 1), 1 << 14)
        g, info = respond(ctx, A, B, torch.tensor(st, device="cuda:0"), k, 1e-4, len(VA), len(VB),
                          np.float32)
        got.append((g, info.cg_iters, info.n_touched, info.n_stencils))
        ctx.close()
    assert got[0][1:] == got[1][1:] and got[0][3] == k
    assert np.isfinite(got[0][0]).all() and np.array_equal(got[0][0], got[1][0])
