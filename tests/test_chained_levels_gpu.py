"""Trie levels launched in a row, each taking its place in the leaf, injection
and hit arrays from the counters of the levels before it: several levels of one
chain write all three.  Against the same levels launched one at a time (a
workspace limit switches the chains off) and the oracle: equal results and
equal counters."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_1208_0274_gb300 import ae  # noqa: E402


# texts of `copies` mutated copies of a word, whose substrings stay in the trie with
# hits for many levels while single occurrences leave it at every level
@pytest.mark.parametrize("copies,m,H,opts", [
    (2, 33, 8, {}),
    (5, 200, 10, dict(leaf_delay=0)),
    (40, 150, 12, dict(leaf_delay=3)),
    (40, 700, 14, dict(int16_limit=20)),
])
def test_chained_levels_equal_single_levels(copies, m, H, opts):
    rng = np.random.default_rng(copies + m)
    word = iid_text(400, DNA, [0.25] * 4, rng)
    T = np.concatenate([word] * copies)
    hit = rng.random(T.size) < 0.02
    T[hit] = np.frombuffer(DNA, np.uint8)[rng.integers(0, 4, size=int(hit.sum()))]
    q = iid_text(m, DNA, [0.25] * 4, rng)
    L = min(m - 3, 300)
    q[2:2 + L] = word[50:50 + L]
    sch = Scheme(1, -3, -5, -2)
    idx = ae.ae_index_build(T, ae.AE_DNA)
    got = []
    for limit in (1 << 34, 0):
        hits, counts = ae.ae_search(idx, [q, q[:m // 2]], sch, H, options=ae.make_options(workspace_limit=limit, **opts))
        st = ae.ae_last_stats()
        # the trie's entries (those of the sweep depend on the order of rows injected at one position)
        got.append((hits, counts, [st["entries"] - st["entries_leaf"]] +
                    [st[k] for k in ("triples", "nodes", "injections", "levels", "levels_int16", "reroutes")]))
    idx.close()
    assert got[0][2] == got[1][2]
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    i, j, s = oracle.sw_hits(T, q, sch, H)
    part = got[1][0][:int(got[1][1][0])]
    assert part.size > 0
    assert np.array_equal(part["text_end"], i) and np.array_equal(part["query_end"], j) and np.array_equal(part["score"], s)
