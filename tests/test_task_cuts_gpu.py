"""Where the sweep's tasks are cut: the longest walk of a task stays within the
span that a task may cover and a row's life beyond it, also where injections
follow each other without a gap (a tandem repeat with one copy in the query),
and each query of a batch is cut by its own injections (one dense query among
many short ones).  Results against the oracle."""
import numpy as np
import pytest

from workloads import BLOSUM62, DNA, PROTEIN, PROTEIN_BG, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1208_0274_gb300 import ae  # noqa: E402

P4 = [0.25] * 4
SCH = Scheme(1, -3, -5, -2)


def _same(got, counts, T, qs, which, sch, H, alphabet):
    at = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    for q in which:
        part = got[at[q]:at[q + 1]]
        i, j, s = oracle.sw_hits(T, qs[q], sch, H, alphabet=alphabet)
        assert np.array_equal(part["text_end"], i) and np.array_equal(part["query_end"], j)
        assert np.array_equal(part["score"], s)


@pytest.mark.parametrize("m,copies,segment", [(613, 3_000, 0), (613, 3_000, 1), (250, 900, 0), (250, 900, 500)])
def test_tandem_repeat_is_walked_in_spans(m, copies, segment):
    rng = np.random.default_rng(m)
    word = iid_text(171, DNA, P4, rng)
    rep = np.concatenate([word] * copies)
    hit = rng.random(rep.size) < 0.12
    rep[hit] = np.frombuffer(DNA, np.uint8)[rng.integers(0, 4, size=int(hit.sum()))]
    T = np.concatenate([iid_text(2_000, DNA, P4, rng), rep, iid_text(2_000, DNA, P4, rng)])
    q = iid_text(m, DNA, P4, rng)
    q[40:211] = word
    idx = ae.ae_index_build(T, ae.AE_DNA)
    got, counts = ae.ae_search(idx, [q], SCH, 25, options=ae.make_options(leaf_segment=segment))
    st = ae.ae_last_stats()
    idx.close()
    # a task covers less than two spans of two to four query lengths (at least 1,024 positions); a
    # row past the last injection lives while its score lasts: m letters matched, m / 2 of gap
    span = max(1_024, 4 << (m.bit_length() - 1))
    assert st["leaf_max_steps"] <= 2 * span + m + m // 2
    assert got.size > 0
    _same(got, counts, T, [q], [0], SCH, 25, DNA)


@pytest.mark.parametrize("where", [0, 150, 300])
def test_dense_query_among_short_ones(where):
    rng = np.random.default_rng(where)
    T = iid_text(20_000, PROTEIN, PROTEIN_BG, rng)
    qs = [iid_text(14, PROTEIN, PROTEIN_BG, rng) for _ in range(300)]
    qs[7] = T[12_000:12_012].copy()
    big = iid_text(2_500, PROTEIN, PROTEIN_BG, rng)
    big[500:700] = T[7_000:7_200]
    qs.insert(where, big)
    sch, H = Scheme(gap_open=-11, gap_extend=-1, matrix=BLOSUM62), 45
    idx = ae.ae_index_build(T, ae.AE_PROTEIN)
    ae.ae_search(idx, [big], sch, H)
    st1 = ae.ae_last_stats()
    got, counts = ae.ae_search(idx, qs, sch, H)
    st = ae.ae_last_stats()
    idx.close()
    # dense by itself (more than one injection for four positions), not on average
    assert st1["injections"] > T.size / 4 and st["injections"] < T.size * len(qs) / 4
    # its tasks are those it has alone; the short queries' walks are no longer than a span
    assert st["leaf_max_steps"] <= st1["leaf_max_steps"] + 1_024 + 64
    _same(got, counts, T, qs, [0, 7, 8, where, 300], sch, H, PROTEIN)
