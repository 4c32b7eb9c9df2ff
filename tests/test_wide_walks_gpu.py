"""Sweep walks continued on a block, where they can go wrong: rows around the
block's 512 threads and past its shared memory, buffers grown from a small odd
capacity, several homologs of several queries in one task, injections merged
into a walked row, and homologs running into the text's or a sequence's end.
Results must equal those of the warp walks alone."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text, mutate

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402

P = [0.25] * 4


# (homolog lengths, divergence, H, scheme, options)
@pytest.mark.parametrize("lengths,div,H,scheme,opts", [
    ((300, 40, 700), 0.08, 30, (1, -3, -5, -2), dict(leaf_wide_rows=20)),
    ((1_100, 1_000, 1_040), 0.01, 40, (1, -3, -5, -2), dict(leaf_wide_rows=100, leaf_capacity=67)),
    ((600, 600, 600), 0.04, 60, (1, -3, -2, -2), dict(leaf_wide_rows=33, leaf_segment=500)),
    ((9_000,), 0.0, 8_000, (1, -3, -5, -2), dict()),
])
def test_block_walks_equal_warp_walks(lengths, div, H, scheme, opts):
    rng = np.random.default_rng(len(lengths) + H)
    T = iid_text(60_000, DNA, P, rng)
    qs = []
    for q in range(2):
        parts = [iid_text(37, DNA, P, rng)]
        for k, L in enumerate(lengths):
            s = T.size - L if k == 0 else int(rng.integers(0, T.size - L))     # the first one ends with the text
            parts += [mutate(T[s:s + L], DNA, P, div, div / 5, rng), iid_text(50, DNA, P, rng)]
        qs.append(np.concatenate(parts))
    cut = int(T.size - lengths[0] // 2)
    found = 0
    for idx in (ae.ae_index_build(T, ae.AE_DNA), ae.ae_index_build_collection([T[:cut], T[cut:]], ae.AE_DNA)):
        want, wc = ae.ae_search(idx, qs, Scheme(*scheme), H, options=ae.make_options(leaf_wide_rows=0))
        got, gc = ae.ae_search(idx, qs, Scheme(*scheme), H, options=ae.make_options(**opts))
        assert ae.ae_last_stats()["leaf_wide_walks"] > 0
        assert np.array_equal(gc, wc) and np.array_equal(got, want)
        found += want.size
        idx.close()
    assert found > 0


# Injections from a fortieth of the text's positions to most of them: tasks cut at
# 64 positions, at one and a half average gaps, and not at all
@pytest.mark.parametrize("m,queries", [(40, 1), (150, 1), (600, 1), (2_000, 1), (9_000, 1), (1_200, 5)])
def test_task_cuts_by_spacing(m, queries):
    import oracle
    rng = np.random.default_rng(m)
    T = iid_text(30_000, DNA, P, rng)
    qs = []
    for _ in range(queries):
        q = iid_text(m, DNA, P, rng)
        L = min(m - 10, 900)
        s = int(rng.integers(0, T.size - L))
        q[5:5 + L] = T[s:s + L]
        qs.append(q)
    idx = ae.ae_index_build(T, ae.AE_DNA)
    sch = Scheme(1, -3, -5, -2)
    got, counts = ae.ae_search(idx, qs, sch, 11)
    idx.close()
    at = 0
    for q, c in zip(qs, counts):
        i, j, s = oracle.sw_hits(T, q, sch, 11)
        part = got[at:at + c]
        at += int(c)
        assert sorted(zip(part["text_end"].tolist(), part["query_end"].tolist(), part["score"].tolist())) == \
            sorted(zip(np.asarray(i).tolist(), np.asarray(j).tolist(), np.asarray(s).tolist()))
    assert at == got.size > 0


# Rows injected at most positions and merged into the walked row: rows of more than
# 32 entries, buffers grown from the smallest capacity, warps alone and blocks
@pytest.mark.parametrize("m,opts", [
    (150, dict(leaf_wide_rows=0, leaf_capacity=64)),
    (1_500, dict(leaf_wide_rows=0)),
    (1_500, dict(leaf_wide_rows=20, leaf_capacity=64)),
    (4_000, dict(leaf_delay=0)),
    (4_000, dict(leaf_wide_rows=40, leaf_segment=7)),
])
def test_merged_rows(m, opts):
    import oracle
    rng = np.random.default_rng(m)
    T, q = iid_text(3_000, DNA, P, rng), iid_text(m, DNA, P, rng)
    q[20:120] = T[-100:]
    sch = Scheme(2, -3, -2, -1)
    i, j, s = oracle.sw_hits(T, q, sch, 16)
    idx = ae.ae_index_build(T, ae.AE_DNA)
    got, counts = ae.ae_search(idx, [q], sch, 16, options=ae.make_options(**opts))
    st = ae.ae_last_stats()
    idx.close()
    assert st["injections"] > 0 and st["reused"] > 0
    assert np.array_equal(got["text_end"], i) and np.array_equal(got["query_end"], j) and np.array_equal(got["score"], s)
