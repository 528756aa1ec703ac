"""The adjacency lists' sort where its form changes: vertices of 8, 9, 16 and 17
neighbours (registers, twice as many, in place), against the oracle's direct
solve of the field that uses them."""
import pytest

from tests.test_gpu_band import test_many_neighbours as many_neighbours
from tests.test_gpu_diffusion import api  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 8, 9, 15, 16, 17, 18])
def test_list_lengths(api, k):  # noqa: F811
    many_neighbours(api, k)
