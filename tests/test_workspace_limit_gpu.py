"""Searches in a capped workspace: what the layouts without gaps and the warp
walks fit into, the default layout and the block walks fit into as well, with the
same results."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402

SCH, H = Scheme(1, -3, -5, -2), 18


def _search(T, qs, **opts):
    idx = ae.ae_index_build(T, ae.AE_DNA)      # a workspace of its own
    try:
        return ae.ae_search(idx, qs, SCH, H, options=ae.make_options(**opts))
    finally:
        idx.close()


def _least(T, qs, lo, hi, **opts):
    """The smallest limit (to 1 %) within which the search succeeds."""
    while hi - lo > hi // 100:
        mid = (lo + hi) // 2
        try:
            _search(T, qs, workspace_limit=mid, **opts)
            hi = mid
        except ae.AEError as e:
            assert e.status == ae.AE_ENOMEM
            lo = mid
    return hi


@pytest.mark.parametrize("n,m", [(200_000, 60), (2_000_000, 1_500)])
def test_default_fits_where_others_fit(n, m):
    rng = np.random.default_rng(m)
    T = iid_text(n, DNA, [0.25] * 4, rng)
    q = iid_text(m, DNA, [0.25] * 4, rng)
    q[5:45] = T[1_000:1_040]
    want, _ = _search(T, [q])
    assert want.size > 0
    # row buffers of 64 entries: 11 MB for the sweep's warps, 12.6 MB for 2^20 hits; walks
    # on blocks take 1.8 MB (1,024 waiting entries of 12 bytes and 3,648 bytes of rows per
    # entry of capacity, 16,384 records of 48 bytes)
    walks = _least(T, [q], 1 << 20, 1 << 29, row_layout=1, leaf_capacity=64, leaf_wide_rows=0)
    least = _least(T, [q], 1 << 20, 1 << 29, leaf_capacity=64)
    assert least <= walks * 1.02 + (2 << 20)
    got, _ = _search(T, [q], workspace_limit=least, leaf_capacity=64)
    assert np.array_equal(got, want)
