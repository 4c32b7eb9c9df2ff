"""The index arrays filled on the device, byte for byte: occurrence blocks, text
ends, separator records and sequence ends in the saved file against arrays
built here from the oracle's suffix array, at sizes around the 64-row block
and with empty sequences."""
import os
import struct

import numpy as np
import pytest

import oracle
from workloads import DNA, PROTEIN

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


def _expected(seqs, dna, collection):
    """(header words, C, occ, tend, text, sep, ends) of the index of `seqs` (code arrays)."""
    sigma, words = (4, 8) if dna else (20, 32)
    text = np.concatenate(seqs).astype(np.uint8)
    n, nseq = text.size, len(seqs) if collection else 0
    joined, pos = [], []
    for k, q in enumerate(seqs):
        if k:
            joined.append(np.array([0]))
            pos.append(np.array([-1]))
        joined.append(q.astype(np.int64) + 1)
        pos.append(np.arange(q.size) + sum(x.size for x in seqs[:k]))
    joined, pos = np.concatenate(joined), np.concatenate(pos)
    J, N = joined.size, joined.size + 1
    sa = oracle.suffix_array(joined[::-1].astype(np.uint8).copy()).astype(np.int64)
    tend = np.where(sa < J, pos[np.maximum(J - 1 - sa, 0)], -1).astype(np.int32)
    bwt = np.where(sa > 0, joined[np.minimum(J - sa, J - 1)], -1)      # -1: sentinel, 0: separator
    nb = (N + 63) // 64 + 1
    occ, sep, ends = np.zeros((nb, words), np.uint32), np.zeros((nb, 4), np.uint32), np.zeros((n + 31) // 32, np.uint32)
    run, seps = np.zeros(sigma, np.int64), 0
    for b in range(nb):
        occ[b, :sigma], sep[b, 0] = run, seps
        for r in range(min(64, max(0, N - 64 * b))):
            v = bwt[64 * b + r]
            code = max(int(v) - 1, 0)
            if dna:
                occ[b, 4 + r // 16] |= np.uint32(code << (2 * (r % 16)))
            else:
                for t in range(5):
                    occ[b, 22 + 2 * t + r // 32] |= np.uint32(((code >> t) & 1) << (r % 32))
            if v > 0:
                run[code] += 1
            elif v == 0:
                sep[b, 1 + r // 32] |= np.uint32(1 << (r % 32))
                seps += 1
    p = 0
    for q in seqs:
        p += q.size
        if q.size:
            ends[(p - 1) >> 5] |= np.uint32(1 << ((p - 1) & 31))
    C = np.zeros(21, np.uint32)
    C[:sigma + 1] = 1 + seps + np.concatenate([[0], np.cumsum(np.bincount(text, minlength=sigma))])
    hdr = [0 if dna else 1, sigma, n, int(np.flatnonzero(sa == 0)[0]), nb, words, nseq, N if nseq else 0]
    body = struct.pack("<8q", *hdr) + C.tobytes() + occ.tobytes() + tend.tobytes() + text.tobytes()
    return body + (sep.tobytes() + ends.tobytes() if nseq else b"")


@pytest.mark.parametrize("dna", [True, False], ids=["dna", "protein"])
@pytest.mark.parametrize("sizes", [(1,), (62,), (63,), (64,), (65,), (127,), (128,), (4_097,), (0, 3, 0, 60, 0),
                                   (63, 64, 65, 0, 0, 1), (1,) * 70], ids=str)
def test_built_index_file_equals_the_oracles(tmp_path, dna, sizes):
    letters = np.frombuffer(DNA if dna else PROTEIN, np.uint8)
    rng = np.random.default_rng(sum(sizes))
    seqs = [rng.integers(0, letters.size, size=k).astype(np.uint8) for k in sizes]
    alphabet = ae.AE_DNA if dna else ae.AE_PROTEIN
    path = os.path.join(tmp_path, "i.aeidx")
    collection = len(sizes) > 1
    idx = ae.ae_index_build_collection([letters[q] for q in seqs], alphabet) if collection else \
        ae.ae_index_build(letters[seqs[0]], alphabet)
    ae.ae_index_save(idx, path)
    idx.close()
    raw = open(path, "rb").read()
    assert raw[8:-8] == _expected(seqs, dna, collection)
    back = ae.ae_index_load(path)           # a loaded index saves the same file
    ae.ae_index_save(back, path + "2")
    back.close()
    assert open(path + "2", "rb").read() == raw
