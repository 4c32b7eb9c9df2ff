"""Sweep walks that never leave their warp (two row entries per lane): a homolog
whose row grows past every chunk edge of 64 entries and shrinks again, injected
rows merged on the way, with tier counting, without block walks and in the
no-allocation entry point.  Results against the oracle."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text, mutate

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1208_0274_gb300 import ae  # noqa: E402


@pytest.mark.parametrize("L,div,scheme", [(130, 0.0, (1, -3, -5, -2)), (400, 0.06, (1, -3, -5, -2)),
                                          (250, 0.04, (1, -3, -2, -2))])
def test_warp_walks(L, div, scheme):
    rng = np.random.default_rng(L)
    T = iid_text(9_000, DNA, [0.25] * 4, rng)
    q = np.concatenate([iid_text(33, DNA, [0.25] * 4, rng), mutate(T[4_000:4_000 + L], DNA, [0.25] * 4, div, div / 5, rng),
                        iid_text(200, DNA, [0.25] * 4, rng)])
    sch, H = Scheme(*scheme), 16
    i, j, s = oracle.sw_hits(T, q, sch, H)
    idx = ae.ae_index_build(T, ae.AE_DNA)
    for opts in (dict(leaf_wide_rows=0), dict(tier_stats=1), dict(leaf_wide_rows=0, leaf_capacity=64, leaf_delay=0)):
        got, _ = ae.ae_search(idx, [q], sch, H, options=ae.make_options(**opts))
        st = ae.ae_last_stats()
        assert st["leaf_max_width"] > 64 and st["leaf_wide_walks"] == 0
        if "tier_stats" in opts:
            assert sum(st["entries_tier"]) == st["entries"]
        assert np.array_equal(got["text_end"], i) and np.array_equal(got["query_end"], j) and np.array_equal(got["score"], s)
    d = torch.from_numpy(q).cuda()
    out = torch.zeros((i.size + 1, 4), dtype=torch.int32, device="cuda")
    status, counts = ae.ae_search_device_static(idx, d.data_ptr(), np.array([0, q.size]), sch, H, out.data_ptr(), i.size + 1)
    idx.close()
    assert status == ae.AE_OK and int(counts[0]) == i.size
    got = out[:i.size].cpu().numpy().view(ae.HIT_DTYPE).reshape(-1)
    assert np.array_equal(got["text_end"], i) and np.array_equal(got["query_end"], j) and np.array_equal(got["score"], s)
