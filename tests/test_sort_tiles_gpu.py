"""The device sort at the edges of its two tile sizes -- 2,048 pairs up to 2^20 of
them, 4,096 above -- through the merge of result records, against numpy."""
import pytest

pytestmark = pytest.mark.gpu

import test_sort_sizes_gpu as sizes  # noqa: E402


@pytest.mark.parametrize("n", [10_239, 10_240, 10_241, (1 << 20) - 1, 1 << 20, (1 << 20) + 1])
@pytest.mark.parametrize("cells", [3, 1 << 20], ids=["few", "many"])
def test_merge_at_tile_edges(n, cells):
    sizes.test_merge_of_records_equals_numpy(n, cells)
