"""Impact zones around a hub, a vertex that is in every row: where the zone's
matrix by rows fits, where it is rejected before its rows are merged, and in
every size class of zones, alone and among others.  Both setups give the same
bits, and the displacement is the oracle's."""
import numpy as np
import pytest

import oracle
from tests import test_gpu_setup_cta as base
from tests.gpu_util import dev_mesh, rel_err, respond
from tests.test_gpu_solver import api  # noqa: F401

pytestmark = pytest.mark.gpu

SYSTEMS = {f"fan_{n}": ([n], [], 1) for n in (31, 33, 60, 85, 120, 255, 257, 700, 1030, 1600)}
SYSTEMS |= {"fans": ([60, 61, 100, 300], [50], 1), "fan_shared_x0": ([200], [], 3), "fan_beside_large": ([400], [1100], 1)}


@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_paths_identical(name, monkeypatch):
    monkeypatch.setattr(base, "SYSTEMS", SYSTEMS)
    base.test_paths_identical(name, True)


@pytest.mark.parametrize("n", [40, 120, 300, 1100])
def test_fan_against_the_oracle(api, n):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    t = 2 * np.pi * np.arange(n) / n
    VB = np.concatenate([[[0, 0, 0]], np.stack([np.cos(t), np.sin(t), 0 * t], 1)]) + rng.uniform(-0.002, 0.002, (n + 1, 3))
    i = np.arange(n)
    TB = np.stack([0 * i, 1 + i, 1 + (i + 1) % n], 1).astype(np.int32)
    VA = np.concatenate([VB[TB].mean(1) - [0, 0, 0.02], [[3, 0, 0], [4, 0, 0], [3, 1, 0]]])
    A, PA = dev_mesh(api, VA, np.array([[n, n + 1, n + 2]], np.int32), False, np.float32)
    B, PB = dev_mesh(api, VB, TB, True, np.float32)
    st = np.zeros((n, 4), np.int32)
    st[:, 1] = st[:, 2] = i
    ctx = api.Context()
    ctx.hfcr_reserve(max(len(VA), len(VB)), n, 1 << 12)
    g, info = respond(ctx, A, B, torch.tensor(st, device="cuda:0"), n, 1e-4, len(VA), len(VB), np.float32)
    rA, rB, _, _ = oracle.respond(st[:, :3].astype(np.uint32), PA, np.array([[n, n + 1, n + 2]], np.int32), PB, TB, 1e-4)
    r = np.concatenate([rA, rB])
    assert info.rel_residual <= 1e-12
    assert rel_err(g, r) <= 1e-6
    ctx.close()
