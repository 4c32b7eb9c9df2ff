"""The index build and the device suffix array within the device memory their
header states: a device filled up to little more than that much, and texts of few
groups (one letter, a period, a tandem repeat), whose rounds sort short keys."""
import numpy as np
import pytest

from workloads import DNA, Scheme, iid_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


def _fill(leave):
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    free, _ = torch.cuda.mem_get_info()
    return torch.empty(free - leave, dtype=torch.uint8, device="cuda")


@pytest.mark.parametrize("nseq", [1, 9])
def test_build_in_little_memory(nseq):
    n = 40_000_000
    rng = np.random.default_rng(nseq)
    T = iid_text(n, DNA, [0.25] * 4, rng)
    parts = np.split(T, np.sort(rng.integers(1, n, nseq - 1))) if nseq > 1 else None
    # working memory of 33 bytes a letter, 5 of the index (6 with the joined copy of a collection)
    fill = _fill(40 * n + (64 << 20))
    try:
        idx = ae.ae_index_build_collection(parts, ae.AE_DNA) if parts else ae.ae_index_build(T, ae.AE_DNA)
    finally:
        del fill
        torch.cuda.empty_cache()
    q = T[12_345_678:12_345_778].copy()
    hits, _ = ae.ae_search(idx, [q], Scheme(1, -3, -5, -2), 90)
    idx.close()
    assert (12_345_777, 99, 100) in {tuple(int(v) for v in h) for h in hits}


def test_suffix_array_in_little_memory():
    n = 40_000_000
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    codes = torch.randint(0, 4, (n,), generator=gen, device="cuda", dtype=torch.uint8)
    sa = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    fill = _fill(34 * n + (32 << 20))
    try:
        ae.ae_suffix_array_device(codes.data_ptr(), n, 4, sa.data_ptr())
    finally:
        del fill
        torch.cuda.empty_cache()
    assert int(sa[0]) == n and torch.equal(torch.bincount(sa).clamp(max=2), torch.ones(n + 1, dtype=torch.int64, device="cuda"))


@pytest.mark.parametrize("kind", ["one", "two", "period", "repeat", "ends"])
@pytest.mark.parametrize("n", [1, 2, 17, 4_099, 70_001])
def test_suffix_array_of_few_groups(kind, n):
    import oracle
    rng = np.random.default_rng(n)
    if kind == "one":
        c = np.zeros(n, np.uint8)
    elif kind == "two":
        c = (np.arange(n) >= n // 2).astype(np.uint8)
    elif kind == "period":
        c = np.resize(rng.integers(0, 4, 7), n).astype(np.uint8)
    elif kind == "repeat":
        c = np.resize(rng.integers(0, 4, 171), n).astype(np.uint8)
        hit = rng.random(n) < 0.01
        c[hit] = rng.integers(0, 4, int(hit.sum()))
    else:                                    # the text ends in the letter that pads short suffixes
        c = rng.integers(0, 4, n).astype(np.uint8)
        c[-(n // 2 + 1):] = 0
    d = torch.from_numpy(c).cuda()
    sa = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    ae.ae_suffix_array_device(d.data_ptr(), n, 4, sa.data_ptr())
    assert np.array_equal(sa.cpu().numpy(), oracle.suffix_array(c))
