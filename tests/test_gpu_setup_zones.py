"""Both setups of up to 4,096 stencils on one large zone, where the zone's
vertices are numbered differently: at the sizes where the zone solver changes
(1,024 rows: the large-zone launch; 1,536: the last by rows; beyond what one
SM's shared memory holds: the cluster, which shares the vertices out by
number), up to the limit of 4,096, and with the blocks taking over after one
iteration.  The displacements are the same bits."""
import pytest

from tests import test_gpu_setup_cta as base

pytestmark = pytest.mark.gpu

SIZES = [1024, 1025, 1536, 1537, 2300, 4095, 4096]
base_systems = dict(base.SYSTEMS)


@pytest.mark.parametrize("switch", [48, 1])
@pytest.mark.parametrize("masses", [False, True], ids=["unit", "masses"])
@pytest.mark.parametrize("rows", SIZES)
def test_one_zone(rows, masses, switch, monkeypatch):
    from paper_1409_2081_gb300 import api
    context = api.Context
    monkeypatch.setattr(api, "Context", lambda **kw: context(block_switch_iters=switch, **kw))
    monkeypatch.setattr(base, "SYSTEMS", {**base_systems, "zone": ([], [rows], 1)})
    base.test_paths_identical("zone", masses)


@pytest.mark.parametrize("switch", [48, 1])
def test_a_large_zone_among_others(switch, monkeypatch):
    from paper_1409_2081_gb300 import api
    context = api.Context
    monkeypatch.setattr(api, "Context", lambda **kw: context(block_switch_iters=switch, **kw))
    monkeypatch.setattr(base, "SYSTEMS", {"mixed": ([130, 20], [1300, 300, 40, 1200] + [5] * 30, 2)})
    base.test_paths_identical("mixed", True)


# more groups than a few warps take eight at a time: of one row, of several, mixed
@pytest.mark.parametrize("masses", [False, True], ids=["unit", "masses"])
@pytest.mark.parametrize("strips,share", [([17] * 242, 1), ([4200], 1), ([9000], 1), ([5000], 2), ([6000], 7), ([5001], 5),
                                          ([3000, 40, 3000], 3), ([1] * 9000, 1)])
def test_many_groups(strips, share, masses, monkeypatch):
    monkeypatch.setattr(base, "SYSTEMS", {"groups": ([], strips, share)})
    base.test_paths_identical("groups", masses)
