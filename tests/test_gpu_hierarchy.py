"""Hierarchy refit on face counts around its block size (one CTA refits 512
leaves, the nodes that span blocks are merged by a second kernel): the pairs
against the exact brute-force oracle, and the number of narrow-phase tests,
which is the number of (edge, face) pairs whose float32 boxes overlap whatever
the tree, before and after the vertices move (the kept tree refitted)."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import detect, dev_mesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_2081_gb300 import api as a
    a.lib()
    return a


def soup(rng, n, size):
    """n triangles of edge length about `size` in the box [-1, 1]^3, signs mixed."""
    c = rng.uniform(-1, 1, (n, 1, 3))
    return (c + rng.uniform(-size, size, (n, 3, 3))).reshape(-1, 3), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def box32(P, idx, dtype):
    p = P[idx].astype(dtype)
    lo, hi = p.min(1), p.max(1)
    if dtype == np.float64:   # rounded outward, as the tree's boxes are
        l32, h32 = lo.astype(np.float32), hi.astype(np.float32)
        lo = np.where(l32 > lo, np.nextafter(l32, np.float32(-np.inf)), l32)
        hi = np.where(h32 < hi, np.nextafter(h32, np.float32(np.inf)), h32)
    return lo, hi


def overlaps(PE, E, PF, F, dtype):
    if len(F) == 1:
        return len(E)          # a tree of one leaf is tested outright
    el, eh = box32(PE, E, dtype)
    fl, fh = box32(PF, F, dtype)
    n = 0
    for i in range(0, len(E), 256):
        n += int(((el[i:i + 256, None] <= fh) & (eh[i:i + 256, None] >= fl)).all(2).sum())
    return n


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("nf", [1, 2, 3, 511, 512, 513, 1024, 1025, 2900])
def test_refit_block_edges(api, nf, dtype):
    rng = np.random.default_rng(nf)
    VA, TA = soup(rng, 150, 0.5)
    VB, TB = soup(rng, nf, 0.1)
    A, _ = dev_mesh(api, VA, TA, False, dtype)
    B, _ = dev_mesh(api, VB, TB, True, dtype)
    EA = oracle.edges(TA)
    ctx = api.Context()
    ctx.hfcr_reserve(len(VA) + len(VB), max(len(TA), nf), 1 << 16)
    for step in range(3):
        PA = np.stack([t.cpu().numpy() for t in (A.x, A.y, A.z)], 1).astype(np.float64)
        PB = np.stack([t.cpu().numpy() for t in (B.x, B.y, B.z)], 1).astype(np.float64)
        _, n, got, st = detect(ctx, A, B)
        ref = oracle.detect(PA, TA, False, PB, TB, True)
        assert np.array_equal(got, ref.rec), step
        assert st.narrow_tests == overlaps(PA, EA, PB, TB, dtype), step
        for t in (B.x, B.y, B.z):   # every face elsewhere, on both sides of 0
            t.copy_(t.roll(3 * (nf // 2)) * (-0.8 if step else 0.9))
    ctx.close()


def test_refit_block_edges_in_a_batch(api):
    """Trees of 1 to 1,500 faces back to back, so that they begin and end
    anywhere in the refit's blocks."""
    import torch
    rng = np.random.default_rng(5)
    sizes = [1, 511, 2, 512, 700, 33, 1500, 1, 290]
    segs, VA, TA, VB, TB = [[0, 0, 0, 0]], [], [], [], []
    for nf in sizes:
        va, ta = soup(rng, 40, 0.5)
        vb, tb = soup(rng, nf, 0.12)
        s = segs[-1]
        VA.append(va), TA.append(ta + s[0]), VB.append(vb), TB.append(tb + s[2])
        segs.append([s[0] + len(va), s[1] + len(ta), s[2] + len(vb), s[3] + len(tb)])
    VA, TA, VB, TB = (np.concatenate(x) for x in (VA, TA, VB, TB))
    A, PA = dev_mesh(api, VA, TA, False, np.float32)
    B, PB = dev_mesh(api, VB, TB, True, np.float32)
    dsegs = torch.tensor(segs, dtype=torch.int32, device="cuda:0")
    out = torch.zeros((1 << 16, 4), dtype=torch.int32, device="cuda:0")
    ctx = api.Context()
    ctx.hfcr_reserve(max(len(VA), len(VB)), max(len(TA), len(TB)), 1 << 16)
    for step in range(2):
        PB = np.stack([t.cpu().numpy() for t in (B.x, B.y, B.z)], 1).astype(np.float64)
        n, st = ctx.hfcr_detect_batch(A, B, dsegs, out, stats=True)
        rec, tests = [], 0
        for a, b in zip(segs[:-1], segs[1:]):
            ta, tb = TA[a[1]:b[1]], TB[a[3]:b[3]]
            r = oracle.detect(PA, ta, False, PB, tb, True).rec.astype(np.int64)
            r[:, 3] += a[3]
            rec.append(r)
            tests += overlaps(PA, oracle.edges(ta), PB, tb, np.float32)
        rec = np.concatenate(rec)
        rec = rec[np.lexsort((rec[:, 3], rec[:, 2], rec[:, 1], rec[:, 0]))]
        assert np.array_equal(out[:n].cpu().numpy().astype(np.int64), rec), step
        assert st.narrow_tests == tests, step
        for t in (B.x, B.y, B.z):
            t.mul_(-0.9)
