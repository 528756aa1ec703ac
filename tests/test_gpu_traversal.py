"""The two phases of the traversal where they can go wrong: a warp's pending
visits beyond its shared memory, the leaf list beyond its capacity, few and
odd numbers of edges, and orientation signs that only the integer stages
decide.  Pairs against the exact brute-force oracle; narrow
tests against the number of overlapping boxes."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import detect, dev_mesh
from tests.test_gpu_hierarchy import api, overlaps, soup  # noqa: F401

pytestmark = pytest.mark.gpu


def check(api, VA, TA, VB, TB, dtype, cap=1 << 17, tris=0, **kw):
    A, PA = dev_mesh(api, VA, TA, False, dtype)
    B, PB = dev_mesh(api, VB, TB, True, dtype)
    ctx = api.Context(**kw)
    ctx.hfcr_reserve(max(len(VA), len(VB)), max(len(TA), len(TB), tris), cap)
    _, n, got, st = detect(ctx, A, B, cap)
    ref = oracle.detect(PA, TA, False, PB, TB, True)
    assert np.array_equal(got, ref.rec)
    assert st.narrow_tests == overlaps(PA, oracle.edges(TA), PB, TB, dtype)
    ctx.close()
    return n, st


@pytest.mark.parametrize("variant", range(9))
def test_long_edges_over_many_faces(api, variant):  # noqa: F811
    """Edges as long as the scene: every warp's stack outgrows shared memory
    (with room in the leaf list for all of their candidates)."""
    rng = np.random.default_rng(7)
    VA, TA = soup(rng, 90, 1.0)
    VB, TB = soup(rng, 6000, 0.05)
    n, st = check(api, VA, TA, VB, TB, np.float32, tris=1 << 20, traverse_variant=variant)
    assert n > 0 and st.narrow_tests < 3 << 20


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_more_leaves_than_the_list_holds(api, dtype):  # noqa: F811
    """Every edge's box overlaps almost every face's: more (edge, leaf)
    candidates than three per reserved triangle."""
    rng = np.random.default_rng(8)
    VA, TA = soup(rng, 70, 1.5)
    VB, TB = soup(rng, 70, 1.5)
    n, st = check(api, VA, TA, VB, TB, dtype)
    assert st.narrow_tests > 3 * 70


@pytest.mark.parametrize("nt", [1, 2, 11, 43])
def test_few_edges(api, nt):  # noqa: F811
    rng = np.random.default_rng(9 + nt)
    VA, TA = soup(rng, nt, 0.7)
    VB, TB = soup(rng, 700, 0.2)
    check(api, VA, TA, VB, TB, np.float32)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("f32_filter", [True, False])
def test_signs_beyond_the_float64_filter(api, dtype, f32_filter):  # noqa: F811
    """Segment ends on the planes of the triangles, moved by multiples of tiny
    amounts (2^-20 to 2^-140 of the coordinates), and ends exactly on them."""
    rng = np.random.default_rng(10)
    VB, TB = soup(rng, 60, 1.0)
    VB = np.round(VB * 64) / 64                   # planes through grid points
    VB[::3, 2] = VB[1::3, 2] = VB[2::3, 2] = np.round(rng.uniform(-8, 8, 60)) / 8
    ends = []
    for f in range(60):
        a, b, c = VB[3 * f:3 * f + 3]
        for _ in range(4):
            s, t = np.sort(rng.integers(0, 65, 2)) / 64.0
            on = a * s + b * (t - s) + c * (1 - t)      # exact on the grid
            eps = rng.choice([0.0, 2.0 ** -20, 2.0 ** -44, 2.0 ** -60, 2.0 ** -100, 2.0 ** -140]) * rng.choice([-1, 1])
            far = on + np.array([rng.integers(-4, 5) / 8, rng.integers(-4, 5) / 8, rng.choice([-1, 1]) / 4])
            p = on.copy()
            if on[2] == 0.0:
                p[2] = eps                              # representable beside 0 only
            ends.append([p, far, far + np.array([0.25, 0.5, 0.125])])
    VA = np.array(ends).reshape(-1, 3)
    TA = np.arange(len(VA), dtype=np.int32).reshape(-1, 3)
    n, st = check(api, VA, TA, VB, TB, dtype, f32_filter=f32_filter)
    assert st.exact_fallbacks > 0
