"""The text-position sweep when many warps' rows outgrow the smallest row
buffers at about the same time, while other warps take tasks: every warp stops
as a whole and the sweep is run again with larger buffers.  Tasks of one
injected row and of the default size, one entry per cell as the oracle's."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1208_0274_gb300 import ae  # noqa: E402


@pytest.mark.parametrize("segment", [0, 1, 33])
def test_many_warps_outgrow_their_rows(segment):
    rng = np.random.default_rng(segment)
    T = iid_text(40_000, DNA, [0.25] * 4, rng)
    q = iid_text(1_200, DNA, [0.25] * 4, rng)
    for s in range(1_000, 39_000, 2_000):      # twenty homologs: rows of hundreds of entries at low gap costs
        T[s:s + 300] = q[100 + s // 100:400 + s // 100]
    sch = Scheme(2, -3, -2, -1)
    idx = ae.ae_index_build(T, ae.AE_DNA)
    got, _ = ae.ae_search(idx, [q], sch, 40, options=ae.make_options(leaf_wide_rows=0, leaf_capacity=64,
                                                                   leaf_segment=segment))
    st = ae.ae_last_stats()
    idx.close()
    assert st["leaf_sweeps"] > 1 and st["leaf_max_width"] > 64
    i, j, s = oracle.sw_hits(T, q, sch, 40)
    assert np.array_equal(got["text_end"], i) and np.array_equal(got["query_end"], j) and np.array_equal(got["score"], s)
