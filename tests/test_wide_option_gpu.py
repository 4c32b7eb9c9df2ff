"""ae_options.leaf_wide_rows: the library's choice by default, any threshold as
given (128 too)."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


def test_thresholds_are_taken_as_given():
    rng = np.random.default_rng(5)
    T = iid_text(60_000, DNA, [0.25] * 4, rng)
    q = np.concatenate([iid_text(50, DNA, [0.25] * 4, rng), T[20_000:20_170], iid_text(50, DNA, [0.25] * 4, rng)])
    idx = ae.ae_index_build(T, ae.AE_DNA)
    walks, width = {}, 0
    for opts in ({}, dict(leaf_wide_rows=33), dict(leaf_wide_rows=127), dict(leaf_wide_rows=128), dict(leaf_wide_rows=129),
                 dict(leaf_wide_auto=0), dict(leaf_wide_rows=128, leaf_wide_auto=1)):
        hits, _ = ae.ae_search(idx, [q], Scheme(1, -3, -5, -2), 30, options=ae.make_options(**opts))
        st = ae.ae_last_stats()
        walks[tuple(opts.items())] = st["leaf_wide_walks"]
        width = st["leaf_max_width"]
        assert hits.size > 0
    idx.close()
    assert 33 < width <= 127                      # so that the thresholds tell which was taken
    assert walks == {(): 1, (("leaf_wide_rows", 33),): 1, (("leaf_wide_rows", 127),): 0, (("leaf_wide_rows", 128),): 0,
                     (("leaf_wide_rows", 129),): 0, (("leaf_wide_auto", 0),): 0,
                     (("leaf_wide_rows", 128), ("leaf_wide_auto", 1)): 1}
