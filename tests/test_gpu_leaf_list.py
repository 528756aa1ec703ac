"""The list of overlapping boxes between the two phases of a traversal, of
max(6 max_tris, 12 max_pairs) entries: just full, one too many and many too
many, in single pairs and batches and every variant of the walk.  Pairs against
the exact brute-force oracle; narrow tests against the number of overlapping
boxes.  And what an overflow may cost: layers that lie on one another in
float64, where testing one edge's leaves by one thread took five times as
long."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import detect, dev_mesh, torch_dev
from tests.test_gpu_hierarchy import api, overlaps, soup  # noqa: F401

pytestmark = pytest.mark.gpu


def run(api, A, B, max_verts, max_tris, pairs, segs=None, **kw):  # noqa: F811
    import torch
    ctx = api.Context(**kw)
    ctx.hfcr_reserve(max_verts, max_tris, pairs)
    if segs is None:
        _, n, got, st = detect(ctx, A, B, pairs)
    else:
        out = torch.zeros((pairs, 4), dtype=torch.int32, device=torch_dev())
        n, st = ctx.hfcr_detect_batch(A, B, segs, out, stats=True)
        got = out[:n].cpu().numpy().astype(np.uint32)
    ctx.close()
    return got, st


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("variant", [0, 4, 8])
def test_list_just_full_and_beyond(api, dtype, variant):  # noqa: F811
    rng = np.random.default_rng(31)
    VA, TA = soup(rng, 200, 1.5)
    VB, TB = soup(rng, 600, 0.03)
    A, PA = dev_mesh(api, VA, TA, False, dtype)
    B, PB = dev_mesh(api, VB, TB, True, dtype)
    ref = oracle.detect(PA, TA, False, PB, TB, True)
    N = overlaps(PA, oracle.edges(TA), PB, TB, dtype)
    fits = -(-N // 12)
    assert N > 6 * len(TB) and len(ref.rec) < fits // 2
    for pairs in (fits, fits - 1, len(ref.rec)):
        got, st = run(api, A, B, len(VB), len(TB), pairs, traverse_variant=variant)
        assert np.array_equal(got, ref.rec)
        assert st.narrow_tests == N


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_batch_beyond_the_list(api, dtype):  # noqa: F811
    import torch
    rng = np.random.default_rng(32)
    va, ta, vb, tb, segs, ref, N = [], [], [], [], [[0, 0, 0, 0]], [], 0
    for size in (1, 40, 3, 25):
        V, T = soup(rng, 10 * size, 1.5)
        W, U = soup(rng, 30 * size, 0.03)
        a, f, b, g = segs[-1]
        V, W = V.astype(dtype), W.astype(dtype)
        rec = oracle.detect(V.astype(float), T, False, W.astype(float), U, True).rec.astype(np.int64)
        rec[:, 1:3] += a
        rec[:, 3] += g
        ref.append(rec)
        N += overlaps(V.astype(float), oracle.edges(T), W.astype(float), U, dtype)
        va.append(V), vb.append(W), ta.append(T + a), tb.append(U + b)
        segs.append([a + len(V), f + len(T), b + len(W), g + len(U)])
    cat = [np.concatenate(x) for x in (va, ta, vb, tb)]
    ref = np.concatenate(ref)
    A, _ = dev_mesh(api, cat[0], cat[1], False, dtype)
    B, _ = dev_mesh(api, cat[2], cat[3], True, dtype)
    table = torch.tensor(segs, dtype=torch.int32, device=torch_dev())
    assert N > max(6 * len(cat[3]), 12 * (len(ref) + 1))
    got, st = run(api, A, B, len(cat[2]), len(cat[3]), len(ref) + 1, table)
    assert np.array_equal(got.astype(np.int64), ref)
    assert st.narrow_tests == N


def layer(rng, n, turn, jitter):
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    x, y = j.ravel() / (n - 1) - 0.5, i.ravel() / (n - 1) - 0.5
    x, y = x * np.cos(turn) - y * np.sin(turn), x * np.sin(turn) + y * np.cos(turn)
    V = np.stack([x, y, 0.3 * np.sin(4 * x) * np.cos(3 * y)], 1) + rng.uniform(-jitter, jitter, (n * n, 3)) / n
    a = (i[:-1, :-1] * n + j[:-1, :-1]).ravel()
    return V, np.concatenate([np.stack([a, a + 1, a + n + 1], 1), np.stack([a, a + n + 1, a + n], 1)]).astype(np.int32)


def test_overflow_of_conforming_layers_is_not_slow(api):  # noqa: F811
    import torch
    rng = np.random.default_rng(33)
    VA, T = layer(rng, 300, 0.0, 0.15)
    VB, _ = layer(rng, 300, 0.2, 0.15)
    VB[:, 2] += 0.15 / 300
    A, _ = dev_mesh(api, VA, T, False, np.float64, edges=True)
    B, _ = dev_mesh(api, VB, T, True, np.float64)
    ms, rec = {}, {}
    for room in (True, False):
        ctx = api.Context()
        pairs = 1 << 18 if room else max(len(rec[True]), 1)
        ctx.hfcr_reserve(len(VA), (16 if room else 1) * len(T), pairs)
        _, _, rec[room], st = detect(ctx, A, B, pairs)
        assert (st.narrow_tests > max(6 * len(T), 12 * pairs)) == (not room)
        out = torch.zeros((pairs, 4), dtype=torch.int32, device=torch_dev())
        t = []
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            ctx.hfcr_detect(A, B, out)
            e[1].record()
            torch.cuda.synchronize()
            t.append(e[0].elapsed_time(e[1]))
        ms[room] = min(t)
        ctx.close()
    assert np.array_equal(rec[True], rec[False])
    assert ms[False] < 2.5 * ms[True]
