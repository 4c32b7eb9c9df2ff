"""The device sort at the edges of its forms -- one block up to 8,192 pairs,
tiles of 4,096 above -- through the merge of result records, against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


@pytest.mark.parametrize("n", [1, 2, 31, 1_023, 8_191, 8_192, 8_193, 12_288, 12_289, 100_003])
@pytest.mark.parametrize("cells", [3, 1 << 20], ids=["few", "many"])
def test_merge_of_records_equals_numpy(n, cells):
    rng = np.random.default_rng(n)
    nq, text, m = 5, 1 << 20, 3_000
    hits = np.zeros(n, dtype=ae.HIT_DTYPE)
    hits["text_end"] = rng.integers(0, min(cells, text), size=n)
    hits["query_end"] = rng.integers(0, min(cells, m), size=n)
    hits["score"] = rng.integers(1, 1_000, size=n)
    qid = rng.integers(0, nq, size=n).astype(np.int32)
    d_hits = torch.from_numpy(hits.view(np.uint8).copy()).cuda()
    d_qid = torch.from_numpy(qid).cuda()
    d_out = torch.zeros(n * 16, dtype=torch.uint8, device="cuda")
    counts, total = ae.ae_hits_merge(d_hits.data_ptr(), d_qid.data_ptr(), n, nq, text, m, d_out.data_ptr())
    order = np.lexsort((-hits["score"], hits["query_end"], hits["text_end"], qid))
    h, q = hits[order], qid[order]
    first = np.ones(n, dtype=bool)
    first[1:] = (q[1:] != q[:-1]) | (h["text_end"][1:] != h["text_end"][:-1]) | (h["query_end"][1:] != h["query_end"][:-1])
    want = h[first]
    got = d_out.cpu().numpy().view(ae.HIT_DTYPE)[:total]
    assert total == want.size and np.array_equal(got, want)
    assert np.array_equal(counts, np.bincount(q[first], minlength=nq))
