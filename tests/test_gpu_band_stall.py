"""Bands on which the pipelined CG's float32 recurrences stall above their
tolerance and would then grow: a constant displacement spread over wide bands,
and over bands that end at an open border of the mesh (no fixed far side).
The field against the oracle's direct solve, the same again in a second call;
and a constant field costs about what a rough one does on the same band."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev_mesh
from tests.test_gpu_band import strip
from tests.test_gpu_diffusion import FIELD_TOL, _gpu_diffuse, api  # noqa: F401

pytestmark = pytest.mark.gpu


def field(kind, n, moved):
    dx = np.zeros((n, 3))
    m = len(moved)
    if kind == "const":
        dx[moved] = [1e-2, -2e-3, 5e-6]
    elif kind == "ramp":
        dx[moved] = np.linspace(0.1, 1, m)[:, None] * [1e-2, -3e-3, 7e-2]
    else:
        dx[moved] = np.random.default_rng(n).normal(size=(m, 3)) * 1e-2
    return dx


@pytest.mark.parametrize("kind", ["const", "ramp"])
@pytest.mark.parametrize("R,nx,rows,at", [(8, 300, 21, 10), (8, 950, 21, 10), (7, 700, 19, 9), (6, 300, 13, 6),
                                          (8, 100, 17, 8), (4, 1000, 9, 4), (3, 2000, 7, 3), (5, 200, 6, 0)])
def test_stalling_bands(api, R, nx, rows, at, kind):  # noqa: F811
    V, T = strip(rows, nx)
    moved = np.arange(at * nx, (at + 1) * nx)
    dx = field(kind, len(V), moved)
    M, _ = dev_mesh(api, V, T, False, np.float32, edges=True)
    ctx = api.Context()
    ctx.hfcr_reserve(len(V), len(T), 16)
    got = _gpu_diffuse(api, ctx, M, dx, R)
    ref = oracle.diffuse(dx, oracle.edges(T), R)
    scale = np.abs(dx).max(0)
    assert (np.abs(got - ref).max(0) <= FIELD_TOL * scale).all()
    assert np.array_equal(got, _gpu_diffuse(api, ctx, M, dx, R))
    ctx.close()


@pytest.mark.parametrize("tol", [1e-4, 1e-7, 1e-12, 1e-14])
def test_other_tolerances(api, tol):  # noqa: F811
    """An open band to looser and tighter residuals, down to where a round
    reduces little and the plain form goes on from the pipelined one's field."""
    V, T = strip(9, 400)
    dx = field("const", len(V), np.arange(4 * 400, 5 * 400))
    M, _ = dev_mesh(api, V, T, False, np.float32, edges=True)
    ctx = api.Context(diffuse_tol=tol)
    ctx.hfcr_reserve(len(V), len(T), 16)
    got = _gpu_diffuse(api, ctx, M, dx, 4)
    ref = oracle.diffuse(dx, oracle.edges(T), 4)
    # |error| <= |A^-1| |r|: the band of 4 open rows has |A^-1| < 30, and |b| <=
    # 2 sqrt(2 nx) times the displacement of a moved vertex
    bound = 30 * (tol * 2 * np.sqrt(2 * 400) + 1e-14) * np.abs(dx).max(0)
    assert (np.abs(got - ref).max(0) <= bound).all()
    ctx.close()


def test_a_constant_field_is_not_slow(api):  # noqa: F811
    import torch
    R, nx = 8, 950
    V, T = strip(2 * R + 5, nx)
    M, _ = dev_mesh(api, V, T, False, np.float32, edges=True)
    ctx = api.Context()
    ctx.hfcr_reserve(len(V), len(T), 16)
    ms = {}
    for kind in ("rough", "const"):
        new = torch.tensor(field(kind, len(V), np.arange((R + 2) * nx, (R + 3) * nx)).T.copy(), device="cuda:0")
        x, t = new.clone(), []
        for _ in range(10):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            x.copy_(new)
            e[0].record()
            ctx.hfcr_diffuse(M, x, R)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        ms[kind] = min(t)
    ctx.close()
    assert ms["const"] < 1.8 * ms["rough"]
