"""Sizes at which two kernels' tiles and groups end, beside those of their own
test files: the network's tiles of 16 samples, and batches whose last
reduction group holds one item."""

import pytest

from test_gpu_batched_groups import _check, bt  # noqa: F401 (bt is a fixture)
from test_gpu_mlp_tiles import M, test_values_and_gradient_at_tile_edges as _network  # noqa: F401 (M is a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,H,n", [(5, 8, 15), (17, 64, 16), (32, 63, 17), (17, 64, 16 * 608 + 1)])
def test_network_tiles_of_16(M, D, H, n):  # noqa: F811
    _network(M, D, H, n)


@pytest.mark.parametrize("items", [21, 31])  # groups of 5 and 6
def test_last_group_of_one_item(bt, items):  # noqa: F811
    K = 1024 * (items - 1) + 700
    _check(bt, [(0, False, 3, 2, K), (0, True, 5, 7, K), (0, False, 20, 13, K)], 10 << 8)
