"""The band CG's cluster kernels where they change over: bands of just 256
vertices per CTA and one more, the pipelined kernel's 960 per CTA and 15,360
in all and beyond, its 8 rings and beyond, vertices of more neighbours than
their codes hold.  Against the oracle's direct solve."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import dev_mesh
from tests.test_gpu_diffusion import FIELD_TOL, _gpu_diffuse, api  # noqa: F401

pytestmark = pytest.mark.gpu


def strip(rows, nx):
    """rows x nx grid, each quad split along a diagonal."""
    i, j = np.meshgrid(np.arange(rows), np.arange(nx), indexing="ij")
    V = np.stack([j.ravel() * 0.01, i.ravel() * 0.01, np.zeros(rows * nx)], 1)
    a = (i[:-1, :-1] * nx + j[:-1, :-1]).ravel()
    T = np.concatenate([np.stack([a, a + 1, a + nx + 1], 1), np.stack([a, a + nx + 1, a + nx], 1)])
    return V, T.astype(np.int32)


def check(api, V, T, moved, R, band=None):  # noqa: F811
    rng = np.random.default_rng(len(V) + R)
    dx = np.zeros((len(V), 3))
    dx[moved] = rng.normal(size=(len(moved), 3)) * 1e-2
    M, _ = dev_mesh(api, V, T, False, np.float32, edges=True)
    ctx = api.Context()
    ctx.hfcr_reserve(len(V), len(T), 16)
    got = _gpu_diffuse(api, ctx, M, dx, R)
    ref = oracle.diffuse(dx, oracle.edges(T), R)
    if band is not None:
        assert np.count_nonzero(np.any(ref != 0, axis=1) & ~np.any(dx != 0, axis=1)) == band
    assert np.abs(got - ref).max() <= FIELD_TOL * np.abs(dx).max()
    assert np.array_equal(got, _gpu_diffuse(api, ctx, M, dx, R))  # the same again
    ctx.close()


@pytest.mark.parametrize("R,nx", [(1, 1), (1, 127), (1, 128), (1, 129), (2, 240), (2, 241), (8, 240),
                                  (8, 960), (8, 961), (9, 100), (30, 60)])
def test_band_sizes(api, R, nx):  # noqa: F811
    if nx == 1:     # a single band vertex on either side: a strip of two columns, one moved vertex
        V, T = strip(3, 2)
        check(api, V, T, np.array([2, 3]), 1, 4)
        return
    rows = 2 * R + 5
    V, T = strip(rows, nx)
    check(api, V, T, np.arange((R + 2) * nx, (R + 3) * nx), R, 2 * R * nx)


@pytest.mark.parametrize("k", [7, 8, 9, 300])
def test_many_neighbours(api, k):  # noqa: F811
    """A hub of k neighbours inside the band (8 codes are kept per vertex),
    the moved vertex on its rim, a second fan around that."""
    rim = np.arange(1, k + 1)
    out = rim + k
    nxt = np.roll(rim, -1)
    T = np.concatenate([np.stack([np.zeros(k, int), rim, nxt], 1), np.stack([rim, out, nxt], 1),
                        np.stack([nxt, out, np.roll(out, -1)], 1)]).astype(np.int32)
    phi = 2 * np.pi * np.arange(k) / k
    V = np.concatenate([np.zeros((1, 3)), np.stack([np.cos(phi), np.sin(phi), 0 * phi], 1),
                        2 * np.stack([np.cos(phi), np.sin(phi), 0 * phi], 1)])
    for R in (1, 2, 8):
        check(api, V, T, np.array([1]), R)
