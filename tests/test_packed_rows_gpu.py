"""The packed row layout where it can go wrong: rows that end at, before and
after a 32-entry chunk, rows open over many chunks (moved from region to
region), long gap runs, hits inside the trie, rows leaving at once, and the
int32 route taking over a packed frontier.  On texts of repeated words, whose
trie keeps long rows at great depth, against the general row kernel: equal
results and equal counters."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


def _words(n, word, rng, mut):
    words = [iid_text(word, DNA, [0.25] * 4, rng) for _ in range(12)]
    out = np.concatenate([words[int(i)] for i in rng.integers(0, 12, size=n // word + 1)])[:n]
    hit = rng.random(n) < mut
    out[hit] = np.frombuffer(DNA, np.uint8)[rng.integers(0, 4, size=int(hit.sum()))]
    return out


# (text, query lengths, word length, mutation rate, scheme, H, options)
CASES = [
    (3_000, (31, 32, 33), 40, 0.0, (1, -3, -5, -2), 12, {}),
    (60_000, (64, 65, 2_000), 50, 0.01, (1, -3, -5, -2), 40, {}),
    (60_000, (1, 500, 1_500), 30, 0.02, (1, -3, -2, -2), 35, dict(leaf_delay=0)),
    (40_000, (1_200,), 60, 0.005, (2, -3, -4, -1), 60, dict(leaf_delay=14)),
    (40_000, (900, 40), 45, 0.01, (1, -3, -5, -2), 30, dict(int16_limit=25)),
    (60_000, (6_000,), 400, 0.08, (1, -4, -5, -2), 25, dict(leaf_delay=3)),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_packed_rows_equal_general_rows(case):
    n, ms, word, mut, sch, H, opts = CASES[case]
    rng = np.random.default_rng(case)
    T = _words(n, word, rng, mut)
    qs = [np.concatenate([T[s:s + m] for s in [int(rng.integers(0, n - m))]]) for m in ms]
    idx = ae.ae_index_build(T, ae.AE_DNA)
    got = []
    for general in (1, 0):
        hits, counts = ae.ae_search(idx, qs, Scheme(*sch), H, options=ae.make_options(general_rows=general, **opts))
        st = ae.ae_last_stats()
        # the trie's entries (those of the sweep depend on the order of rows injected at one position)
        got.append((hits, counts, [st["entries"] - st["entries_leaf"]] +
                    [st[k] for k in ("triples", "nodes", "injections", "reroutes")]))
    idx.close()
    assert got[0][0].size > 0
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
    assert got[0][2] == got[1][2]
