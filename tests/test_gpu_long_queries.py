"""Batches of more than 192 bases per query on average: the packed copy of the
batch, and compares in the text in iterations of their own.  Queries of lengths
around 64-base steps from a text with long repeats (so that several suffixes
tie with a query for hundreds of bases), exact and with one substitution near
the ends of a record's bases, of a step and of the query, some running past the
text's end: equal to the oracle in both orders, on both strands and with
indexes with and without a k-mer table."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu
COMP = np.zeros(256, dtype=np.uint8)
for _a, _b in zip(b"ACGT", b"TGCA"):
    COMP[_a] = _b


@pytest.fixture(scope="module")
def sa():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa as sa_mod

    build_lib.build()
    return sa_mod


@pytest.mark.parametrize("kmer_k", [None, 3, 0])
@pytest.mark.parametrize("rc", [False, True])
def test_long_compares(sa, kmer_k, rc):
    ref = datagen.reference(30_000, 17, gc=0.5)
    block = ref[1000:3500].copy()
    for at in (5000, 9000, 14_000, 27_500):  # the last copy ends the text
        ref[at:at + block.size] = block
    ref[9000 + 700] = ord("A") if ref[9000 + 700] != ord("A") else ord("C")
    T = oracle.normalize(ref)
    osa = oracle.sa_naive(T)
    idx = sa.sa_build(torch.from_numpy(ref.copy()).cuda(), kmer_k=kmer_k)
    rng = np.random.default_rng(23)
    qs = []
    for m in (150, 193, 223, 224, 225, 256, 287, 288, 289, 320, 511, 512, 513, 1024, 1900):
        for at in (1000, 1017, 5000, 9000, 14_031, 27_500, 20_000):
            q = ref[at:at + m].copy()
            qs.append(q)
            for p in (100, 104, 127, 128, 159, 160, 191, 192, 223, m - 33, m - 1):
                if p < q.size:
                    c = q.copy()
                    c[p] = datagen.ASCII[(int(np.nonzero(datagen.ASCII == c[p])[0][0]) + int(rng.integers(1, 4))) % 4]
                    qs.append(c)
        qs.append(np.concatenate([ref[-m + 20:], datagen.ASCII[rng.integers(0, 4, 20)]]))  # runs past the end
    qo = np.zeros(len(qs) + 1, dtype=np.int64)
    np.cumsum([q.size for q in qs], out=qo[1:])
    assert qo[-1] > 192 * len(qs)
    want_b = np.concatenate(qs)
    lo, hi = oracle.search_batch(T, osa, want_b, qo, threads=oracle.cpu_threads())
    fed = np.concatenate([COMP[q][::-1] for q in qs]) if rc else want_b
    for order in (sa.SA_PARAM_INPUT_ORDER, sa.SA_PARAM_KMER_ORDER):
        if kmer_k == 0 and order == sa.SA_PARAM_KMER_ORDER:
            continue
        for probes in (1, 3):
            p = sa.sa_search_params(flags=order | (sa.SA_PARAM_REVERSE_COMPLEMENT if rc else 0), front_probes=probes)
            got = sa.sa_search_batch(idx, torch.from_numpy(fed.copy()).cuda(), torch.from_numpy(qo).cuda(),
                                     params=p).cpu().numpy()
            bad = np.nonzero((got[:, 0] != lo) | (got[:, 1] != hi))[0]
            assert bad.size == 0, (order, probes, bad[:5], got[bad[:5]], lo[bad[:5]], hi[bad[:5]])
