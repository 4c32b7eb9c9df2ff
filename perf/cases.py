"""What the library is used for, as cases that can be timed and compared.

The main use is a search: a text is indexed once and stays resident on the GPU,
and queries arrive.  The text of a case is therefore the same for every seed
(it is the database), its index and the stream's workspace are built once per
process and shared by all states, and the seed draws the queries: i.i.d.
letters at the text's composition with a share of each query copied from the
text and mutated, the shapes of the benchmark's workloads.  The other paths a
program takes are indexing a text and searching it once, the suffix array by
itself, and the work predictor (features, forward, gradient, training).

    listed()             the cases by name
    draw(rng)            another case of the same ranges
    prepare(case, seed)  inputs and handles
    run(state)           one pass through the public entry points
    work(case)           bytes and operations a pass cannot do without
    exact(case, seed)    64-bit values of the predictor's outputs
"""
import math

import numpy as np
import torch

from paper_1208_0274_gb300 import ae

DNA, PROTEIN = b"ACGT", b"ARNDCQEGHILKMFPSTWYV"
GC = 0.41                                # composition of the DNA texts

# Background residue frequencies in PROTEIN order (Robinson & Robinson 1991).
RESIDUES = np.array([
    0.07805, 0.05129, 0.04487, 0.05364, 0.01925, 0.04264, 0.06295, 0.07377, 0.02199, 0.05142,
    0.09019, 0.05744, 0.02243, 0.03856, 0.05203, 0.07120, 0.05841, 0.01330, 0.03216, 0.06441])
RESIDUES = RESIDUES / RESIDUES.sum()

# BLOSUM62 (Henikoff & Henikoff 1992), rows and columns in PROTEIN order.
BLOSUM62 = np.array([[int(v) for v in row.split()] for row in """
 4 -1 -2 -2  0 -1 -1  0 -2 -1 -1 -1 -1 -2 -1  1  0 -3 -2  0
-1  5  0 -2 -3  1  0 -2  0 -3 -2  2 -1 -3 -2 -1 -1 -3 -2 -3
-2  0  6  1 -3  0  0  0  1 -3 -3  0 -2 -3 -2  1  0 -4 -2 -3
-2 -2  1  6 -3  0  2 -1 -1 -3 -4 -1 -3 -3 -1  0 -1 -4 -3 -3
 0 -3 -3 -3  9 -3 -4 -3 -3 -1 -1 -3 -1 -2 -3 -1 -1 -2 -2 -1
-1  1  0  0 -3  5  2 -2  0 -3 -2  1  0 -3 -1  0 -1 -2 -1 -2
-1  0  0  2 -4  2  5 -2  0 -3 -3  1 -2 -3 -1  0 -1 -3 -2 -2
 0 -2  0 -1 -3 -2 -2  6 -2 -4 -4 -2 -3 -3 -2  0 -2 -2 -3 -3
-2  0  1 -1 -3  0  0 -2  8 -3 -3 -1 -2 -1 -2 -1 -2 -2  2 -3
-1 -3 -3 -3 -1 -3 -3 -4 -3  4  2 -3  1  0 -3 -2 -1 -3 -1  3
-1 -2 -3 -4 -1 -2 -3 -4 -3  2  4 -2  2  0 -3 -2 -1 -2 -1  1
-1  2  0 -1 -3  1  1 -2 -1 -3 -2  5 -1 -3 -1  0 -1 -3 -2 -2
-1 -1 -2 -3 -1  0 -2 -3 -2  1  2 -1  5  0 -2 -1 -1 -1 -1  1
-2 -3 -3 -3 -2 -3 -3 -3 -1  0  0 -3  0  6 -4 -2 -2  1  3 -1
-1 -2 -2 -1 -3 -1 -1 -2 -2 -3 -3 -1 -2 -4  7 -1 -1 -4 -3 -2
 1 -1  1  0 -1  0  0  0 -1 -2 -2  0 -1 -2 -1  4  1 -3 -2 -2
 0 -1  0 -1 -1 -1 -1 -2 -2 -1 -1 -1 -1 -2 -1  1  5 -2 -2  0
-3 -3 -4 -4 -2 -2 -3 -2 -2 -3 -2 -3 -1  1 -4 -3 -2 11  2 -3
-2 -2 -2 -3 -2 -1 -2 -3  2 -1 -1 -2 -1  3 -3 -2 -2  2  7 -1
 0 -3 -3 -3 -1 -2 -2 -3 -3  3  1 -2  1 -1 -2 -2  0 -3 -1  4
""".strip().splitlines()], dtype=np.int8)

TEXT_100M, PROTEIN_1M = 100_000_000, 1_000_000


def listed():
    """Each kind of call with the sizes it is used at."""
    return [
        # one short query against a small genome region: the shortest whole search, bound by
        # launches and read-backs (the benchmark's small configuration)
        dict(name="small_search", kind="dna", n=100_000, queries=1, lo=1000, hi=1000, H=30, planted=0.5, host=True),
        # one request of a search service: a read-sized query against the resident 100 Mbp text
        dict(name="service_request", kind="dna", n=TEXT_100M, queries=1, lo=613, hi=613, H=19, planted=0.3, host=True),
        # one gene- or contig-sized query, inputs and results kept on the device
        dict(name="contig_search", kind="dna", n=TEXT_100M, queries=1, lo=10_007, hi=10_007, H=19, planted=0.01,
             host=False),
        # a request batch of mixed lengths (log-uniform, 100 bp to 20 kbp), host queries and host hits
        dict(name="mixed_batch", kind="dna", n=TEXT_100M, queries=96, lo=100, hi=20_000, H=20, planted=0.01, host=True),
        # one 1 Mbp query, the longest the benchmark holds, on the device
        dict(name="long_query", kind="dna", n=TEXT_100M, queries=1, lo=1_000_003, hi=1_000_003, H=23, planted=0.01,
             host=False),
        # queries of 10 kbp to 1 Mbp together with the benchmark's batch size and leaf delay
        dict(name="scaled_search", kind="dna", n=TEXT_100M, queries=8, lo=10_000, hi=1_000_000, H=22, planted=0.01,
             host=False, batch_columns=2_000_000, leaf_delay=10),
        # cheap gaps <1,-3,-2,-2>: many more live cells and gap runs per letter
        dict(name="cheap_gaps", kind="dna", n=TEXT_100M, queries=2, lo=60_000, hi=100_000, H=21, planted=0.01, host=False,
             gap_open=-2),
        # long reads that are homologous end to end, strict threshold: the walk along the text
        dict(name="homologous_reads", kind="dna", n=TEXT_100M, queries=6, lo=4_000, hi=12_000, H=48, planted=1.0,
             host=False),
        # protein queries with a substitution matrix: the general row kernel from the trie's root
        dict(name="protein_blosum62", kind="protein", n=PROTEIN_1M, queries=6, lo=100, hi=5_000, H=50, host=False),
        # a collection of sequences indexed and searched once (an ad-hoc database)
        dict(name="index_and_search", kind="build", n=20_000_003, nseq=48, queries=2, lo=1_500, hi=2_500, H=20,
             planted=0.05),
        # the suffix array of a text on the device, a caller building its own index
        dict(name="suffix_array", kind="suffix", n=10_000_019, sigma=4, reversed=True),
        # the work predictor: features of a batch, prediction, gradient and a short training run
        dict(name="predictor", kind="predictor", n=TEXT_100M, queries=64, lo=200, hi=20_000, rows=2_000, batch=64,
             epochs=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "dna", "dna", "batch", "reads", "gaps", "protein", "build", "suffix", "predictor"])
    if kind == "small":
        m = _log(rng, 60, 5_000)
        return dict(kind="dna", n=_log(rng, 20_000, 2_000_000), queries=rng.randint(1, 4), lo=m, hi=m,
                    H=rng.randint(18, 40), planted=0.5, host=rng.random() < 0.5)
    if kind == "dna":
        m = _log(rng, 150, 900_000)
        return dict(kind="dna", n=_log(rng, 5_000_000, TEXT_100M), queries=1, lo=m, hi=m, H=rng.randint(19, 31),
                    planted=0.3 if m < 10_000 else 0.01, host=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind="dna", n=TEXT_100M, queries=_log(rng, 4, 160), lo=_log(rng, 60, 1_000),
                    hi=_log(rng, 2_000, 20_000), H=rng.randint(19, 23), planted=0.01, host=rng.random() < 0.5,
                    leaf_delay=rng.choice([6, 8, 10, 12]))
    if kind == "reads":
        return dict(kind="dna", n=_log(rng, 10_000_000, TEXT_100M), queries=rng.randint(1, 6), lo=_log(rng, 500, 3_000),
                    hi=_log(rng, 3_000, 15_000), H=rng.randint(30, 60), planted=1.0, host=False)
    if kind == "gaps":
        m = _log(rng, 1_000, 60_000)
        return dict(kind="dna", n=_log(rng, 10_000_000, TEXT_100M), queries=rng.randint(1, 3), lo=m, hi=m,
                    H=rng.randint(20, 31), planted=0.1 if m < 10_000 else 0.01, host=False, gap_open=rng.choice([-2, -3, -4]),
                    mismatch=rng.choice([-3, -4]))
    if kind == "protein":
        m = _log(rng, 60, 3_000)
        return dict(kind="protein", n=_log(rng, 50_000, PROTEIN_1M), queries=rng.randint(1, 4), lo=m, hi=m,
                    H=rng.randint(50, 70), host=rng.random() < 0.5)
    if kind == "build":
        return dict(kind="build", n=_log(rng, 300_000, 20_000_000), nseq=rng.choice([1, 1, 7, 300]), queries=1,
                    lo=500, hi=2_000, H=rng.randint(19, 30), planted=0.05)
    if kind == "suffix":
        return dict(kind="suffix", n=_log(rng, 10_000, 30_000_000), sigma=rng.choice([2, 4, 20]),
                    reversed=rng.random() < 0.5)
    return dict(kind="predictor", n=_log(rng, 1_000_000, TEXT_100M), queries=rng.randint(1, 96), lo=200,
                hi=_log(rng, 1_000, 20_000), rows=_log(rng, 100, 4_000), batch=rng.choice([32, 64, 128]), epochs=1)


# ------------------------------------------------------------------ inputs

def _probs(kind):
    if kind == "protein":
        return RESIDUES
    at, gc = (1 - GC) / 2, GC / 2
    return np.array([at, gc, gc, at])


def _letters(kind):
    return np.frombuffer(PROTEIN if kind == "protein" else DNA, dtype=np.uint8)


def _text(kind, n, seed):
    """n i.i.d. letters (host, ASCII), drawn on the GPU in slices."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    cdf = torch.tensor(np.cumsum(_probs(kind))[:-1], dtype=torch.float32, device="cuda")
    table = torch.from_numpy(_letters(kind).copy()).cuda()
    out = np.empty(n, dtype=np.uint8)
    step = 1 << 25
    for s in range(0, n, step):
        u = torch.rand(min(step, n - s), generator=gen, device="cuda")
        out[s:s + u.numel()] = table[torch.bucketize(u, cdf, right=True)].cpu().numpy()
    return out


_resident = {}      # (kind, n) -> (text, index): the databases of this process, the last few kept


def _database(kind, n):
    key = (kind, n)
    if key not in _resident:
        while len(_resident) >= 3:
            _resident.pop(next(iter(_resident)))
        text = _text(kind, n, 20120802)
        _resident[key] = (text, ae.ae_index_build(text, ae.AE_PROTEIN if kind == "protein" else ae.AE_DNA))
    else:
        _resident[key] = _resident.pop(key)
    return _resident[key]


def _mutate(seg, kind, sub, indel, rng):
    """Substitutions at rate `sub`, insertions and deletions of 1-3 letters at rate `indel`."""
    letters, probs = _letters(kind), _probs(kind)
    out = seg.copy()
    hit = rng.random(out.size) < sub
    out[hit] = rng.choice(letters, size=int(hit.sum()), p=probs)
    drop = np.zeros(out.size, dtype=bool)
    for p in np.flatnonzero(rng.random(out.size) < indel / 2):
        drop[p:p + int(rng.integers(1, 4))] = True
    keep = np.flatnonzero(~drop)
    out = out[keep]
    at = np.flatnonzero(rng.random(out.size) < indel / 2)
    at = np.repeat(at, rng.integers(1, 4, size=at.size))
    return np.insert(out, at, rng.choice(letters, size=at.size, p=probs))


def _query(text, m, case, rng):
    """m letters: i.i.d. background with `planted` of them copied from the text and mutated (DNA: segments
    of 300-3,000 letters at 5-15% divergence, 5:1 substitutions to indels; protein: one segment of a tenth
    of the query at 30-60% identity)."""
    kind = "protein" if case["kind"] == "protein" else "dna"
    letters, probs = _letters(kind), _probs(kind)
    cum = np.cumsum(probs)
    cum[-1] = 1.0
    q = letters[np.searchsorted(cum, rng.random(m), side="right")]
    if kind == "protein":
        plan = [min(m, max(60, m // 10))]
    else:
        plan, left = [], int(round(case["planted"] * m))
        while left > 0:
            plan.append(min(left, int(rng.integers(300, 3_001))))
            left -= plan[-1]
    free = m - sum(plan)
    cuts = np.sort(rng.integers(0, free + 1, size=len(plan)))
    pos, prev = 0, 0
    for L, cut in zip(plan, cuts):
        pos += int(cut) - prev
        prev = int(cut)
        s = int(rng.integers(0, text.size - L))
        if kind == "protein":
            piece = _mutate(text[s:s + L], kind, 1.0 - rng.uniform(0.3, 0.6), 0.02, rng)
        else:
            div = rng.uniform(0.05, 0.15)
            piece = _mutate(text[s:s + L], kind, div * 5 / 6, div / 6, rng)
        piece = piece[:L]
        q[pos:pos + piece.size] = piece
        pos += L
    return q


def _lengths(case):
    """The query lengths: log-spaced between lo and hi, the same for every seed."""
    k = case["queries"]
    if k == 1:
        return [case["lo"]]
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [int(round(math.exp(lo + (hi - lo) * i / (k - 1)))) for i in range(k)]


def _queries(text, case, seed):
    rng = np.random.default_rng([seed, 7])
    return [_query(text, m, case, rng) for m in _lengths(case)]


def _scheme(case):
    if case["kind"] == "protein":
        return dict(match=1, mismatch=-3, gap_open=-11, gap_extend=-1, matrix=BLOSUM62)
    return dict(match=1, mismatch=case.get("mismatch", -3), gap_open=case.get("gap_open", -5), gap_extend=-2)


def _options(case):
    kw = {k: case[k] for k in ("batch_columns", "leaf_delay") if k in case}
    return ae.make_options(**kw) if kw else None


def _room(case):
    """Records in the program's result table: a homologous stretch gives some hundreds of results per letter."""
    m = sum(_lengths(case))
    if case["kind"] == "protein":
        return 200_000 + 800 * m
    return 50_000 + 8 * m + int(1_500 * case["planted"] * m)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.kind = case, case["kind"]
    if s.kind in ("dna", "protein"):
        text, s.index = _database(s.kind, case["n"])
        s.queries = _queries(text, case, seed)
        s.scheme, s.options, s.H = _scheme(case), _options(case), [case["H"]] * case["queries"]
        s.host = case["host"]
        if not s.host:
            s.offsets = np.concatenate([[0], np.cumsum([q.size for q in s.queries])]).astype(np.int64)
            s.seq = torch.from_numpy(np.concatenate(s.queries)).cuda()
            s.hits = torch.zeros((_room(case), 4), dtype=torch.int32, device="cuda")
        else:
            s.table = np.zeros(_room(case), dtype=ae.HIT_DTYPE)
    elif s.kind == "build":
        s.text = _text("dna", case["n"], seed)
        rng = np.random.default_rng([seed, 8])
        cuts = np.sort(rng.integers(1, case["n"], size=case["nseq"] - 1))
        s.parts = np.split(s.text, cuts)
        s.queries = _queries(s.text, case, seed)
        s.scheme, s.H = _scheme(case), [case["H"]] * case["queries"]
        s.table = np.zeros(_room(case), dtype=ae.HIT_DTYPE)
    elif s.kind == "suffix":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        s.codes = torch.randint(0, case["sigma"], (case["n"],), generator=gen, device="cuda", dtype=torch.uint8)
        s.sa = torch.empty(case["n"] + 1, dtype=torch.int32, device="cuda")
    else:
        text, s.index = _database("dna", case["n"])
        s.seqs = _queries(text, dict(case, planted=0.01), seed)
        s.offsets = np.concatenate([[0], np.cumsum([q.size for q in s.seqs])]).astype(np.int64)
        s.seq = torch.from_numpy(np.concatenate(s.seqs)).cuda()
        s.mlp = ae.Mlp(seed)
        s.start = s.mlp.get_params()
        x, t, s.norm = _logged(case, seed)
        s.mlp.set_norm(*s.norm)
        s.x, s.t = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
        s.feat = torch.empty((case["queries"], ae.MLP_IN), dtype=torch.float32, device="cuda")
        s.pred = torch.empty((case["queries"], ae.MLP_OUT), dtype=torch.float32, device="cuda")
    return s


def _logged(case, seed):
    """Feature rows and targets of logged searches, and their normalisation."""
    rng = np.random.default_rng([seed, 9])
    r = case["rows"]
    m = np.exp(rng.uniform(math.log(100), math.log(20_000), size=r))
    x = np.empty((r, ae.MLP_IN), dtype=np.float32)
    x[:, :64] = rng.dirichlet(np.full(64, 20.0), size=r)
    x[:, 64] = np.log1p(m)
    x[:, 65] = rng.gamma(1.0, 0.05, size=r)
    t = np.empty((r, ae.MLP_OUT), dtype=np.float32)
    t[:, 0] = np.log(3500 * m) + 0.1 * rng.standard_normal(r)
    t[:, 1] = np.log1p(0.5 * m) + 8 * x[:, 65] + 0.3 * rng.standard_normal(r)
    sd = x.std(0)
    sd[:64] *= 32.0
    return x, t, (x.mean(0), sd, t.mean(0), t.std(0))


# ------------------------------------------------------------------ one pass

def _keep(s, hits, counts):
    """The results of one call in the program's table."""
    if hits.size > s.table.size:      # more results than expected: a larger table
        s.table = np.zeros(hits.size, dtype=ae.HIT_DTYPE)
    s.table[:hits.size] = hits
    return {"text_end": s.table["text_end"], "query_end": s.table["query_end"], "score": s.table["score"],
            "counts": counts}


def run(s):
    if s.kind in ("dna", "protein"):
        if s.host:
            return _keep(s, *ae.ae_search(s.index, s.queries, s.scheme, s.H, s.options))
        status, counts = ae.ae_search_device(s.index, s.seq.data_ptr(), s.offsets, s.scheme, s.H, s.hits.data_ptr(),
                                             s.hits.shape[0], s.options)
        if status == ae.AE_EOVERFLOW:     # more results than expected: make room and search again
            s.hits = torch.zeros((int(counts.sum()), 4), dtype=torch.int32, device="cuda")
            status, counts = ae.ae_search_device(s.index, s.seq.data_ptr(), s.offsets, s.scheme, s.H,
                                                 s.hits.data_ptr(), s.hits.shape[0], s.options)
        return {"hits": s.hits, "counts": counts}
    if s.kind == "build":
        index = ae.ae_index_build_collection(s.parts) if len(s.parts) > 1 else ae.ae_index_build(s.text)
        out = _keep(s, *ae.ae_search(index, s.queries, s.scheme, s.H))
        index.close()
        return out
    if s.kind == "suffix":
        ae.ae_suffix_array_device(s.codes.data_ptr(), s.codes.numel(), s.case["sigma"], s.sa.data_ptr(),
                                  reversed=s.case["reversed"])
        return {"sa": s.sa}
    s.mlp.set_params(s.start)
    ae.ae_mlp_features(s.index, s.seq.data_ptr(), s.offsets, s.feat.data_ptr())
    s.mlp.forward(s.feat.data_ptr(), s.feat.shape[0], s.pred.data_ptr())
    loss, grads = s.mlp.loss_grad(s.x.data_ptr(), s.t.data_ptr(), s.x.shape[0])
    last = s.mlp.train(s.x.data_ptr(), s.t.data_ptr(), s.x.shape[0], s.case["epochs"], s.case["batch"], 1e-3,
                       weight_decay=0.05, seed=3)
    return {"features": s.feat, "predictions": s.pred, "loss": loss, "gradient": grads, "last_loss": last,
            "weights": s.mlp.get_params()}


# ------------------------------------------------------------------ what a pass cannot do without

# Live cells of the Gotoh rows per query letter against 10^8 letters, as the engine counts them for
# <1,-3,-5,-2> (ae_stats.entries over the query letters); they grow with the text like n^0.6 (Section 6).
# Cheaper gaps keep about three times as many, and BLOSUM62 at H = 50 keeps half of all m n cells.
CELLS_PER_LETTER = 3_500


def _search_work(kind, n, m, planted, gap_open):
    if kind == "protein":
        cells, hits = 0.5 * m * n, 0.0
    else:
        cells = CELLS_PER_LETTER * m * (n / 1e8) ** 0.6 * (3.0 if gap_open > -5 else 1.0)
        hits = 10.0 + 100.0 * planted * m
    # per cell: three additions and three maxima; queries in, results out
    return {"bytes": float(m + 16 * hits), "flops": 6.0 * cells}


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "suffix":
        return {"bytes": float(n + 4 * (n + 1)), "flops": 0.0}
    m = sum(_lengths(case))
    if kind == "predictor":
        macs = 66 * 128 + 128 * 128 + 128 * 2
        rows = case["queries"] + 3 * case["rows"] * (1 + case["epochs"])
        # the features count each window of the queries in the index (two 32-byte blocks a letter step)
        return {"bytes": float(m + 4 * 70 * case["rows"] + 4 * 4 * ae.MLP_PARAMS), "flops": 2.0 * macs * rows}
    w = _search_work(kind, n, m, case.get("planted", 0.0), case.get("gap_open", -5))
    if kind == "build":
        w["bytes"] += n + n / 2 + 4.0 * n + n       # text in; blocks, text ends and letters of the index out
    return w


# ------------------------------------------------------------------ 64-bit values

def _window_counts(text, seqs, K):
    """log1p of the occurrences in `text` of every window of K letters, averaged per query."""
    lut = torch.zeros(256, dtype=torch.int64, device="cuda")
    lut[torch.tensor(list(DNA), device="cuda")] = torch.arange(4, device="cuda")

    def grams(a):
        c = lut[torch.from_numpy(a).cuda().long()]
        g = torch.zeros(c.numel() - K + 1, dtype=torch.int64, device="cuda")
        for i in range(K):
            g = g * 4 + c[i:c.numel() - K + 1 + i]
        return g

    table = grams(text).sort().values
    out = []
    for q in seqs:
        if q.size < K:
            out.append(0.0)
            continue
        g = grams(q)
        n = torch.searchsorted(table, g, right=True) - torch.searchsorted(table, g)
        out.append(float(torch.log1p(n.double()).mean()))
    return np.array(out)


def exact(case, seed):
    if case["kind"] != "predictor":
        return None          # searches and suffix arrays are whole numbers
    s = prepare(case, seed)
    text, _ = _database("dna", case["n"])
    f = np.zeros((len(s.seqs), ae.MLP_IN))
    lut = np.zeros(256, dtype=np.int64)
    lut[np.frombuffer(DNA, np.uint8)] = np.arange(4)
    for k, q in enumerate(s.seqs):
        c = lut[q]
        if q.size >= 3:
            f[k, :64] = np.bincount(16 * c[:-2] + 4 * c[1:-1] + c[2:], minlength=64) / (q.size - 2)
        f[k, 64] = math.log1p(q.size)
    K = min(32, next(k for k in range(1, 40) if 4 ** k >= case["n"] + 1) + 4)
    f[:, 65] = _window_counts(text, s.seqs, K)
    x_mu, x_sd, y_mu, y_sd = [torch.tensor(np.asarray(a, np.float32), dtype=torch.float64) for a in s.norm]
    p = torch.tensor(s.start, dtype=torch.float64, requires_grad=True)
    h, i, o = ae.MLP_HIDDEN, ae.MLP_IN, ae.MLP_OUT
    w1, b1, w2, b2, w3, b3 = torch.split(p, [h * i, h, h * h, h, o * h, o])

    def forward(x):
        a = torch.relu((x - x_mu) / x_sd @ w1.view(h, i).T + b1)
        return torch.relu(a @ w2.view(h, h).T + b2) @ w3.view(o, h).T + b3

    x, t = s.x.cpu().double(), s.t.cpu().double()
    loss = ((forward(x) - (t - y_mu) / y_sd) ** 2).sum() / (2 * x.shape[0])
    loss.backward()
    pred = forward(torch.from_numpy(f)) * y_sd + y_mu
    return {"features": torch.from_numpy(f), "predictions": pred.detach(), "loss": loss.item(), "gradient": p.grad,
            "last_loss": None, "weights": None}
