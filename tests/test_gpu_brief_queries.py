"""Queries shorter than k are answered from two k-mer entries' counts and the
text's last k bases.  Every query of up to five bases (and longer ones over a
two-letter alphabet, all-A and all-T ones) against short texts whose ends are
runs of A, T and mixtures, for k above, at and below the query and the text
length: equal to the oracle and to an index without a k-mer table."""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sa():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa as sa_mod

    build_lib.build()
    return sa_mod


def _texts():
    rng = np.random.default_rng(3)
    out = ["A", "T", "AC", "TTTTTTTT", "AAAAAAAAAAAA", "ACGT", "CAAAAAAA", "GTTTAAA", "ACGTACGTAAAAAAAA"]
    for letters in ("AC", "AT", "ACGT", "GA"):
        for n in (1, 2, 3, 5, 7, 8, 9, 14, 15, 16, 31, 32, 33, 40):
            out.append("".join(rng.choice(list(letters), n)))
            out.append("".join(rng.choice(list(letters), n)) + "A" * int(rng.integers(1, 9)))
    return out


@pytest.mark.parametrize("k", [1, 4, 6, 9])
@pytest.mark.parametrize("order", ["kmer", "input"])
def test_every_short_query(sa, k, order):
    qs = ["".join(p) for m in range(1, 6) for p in itertools.product("ACGT", repeat=m)]
    qs += ["".join(p) for m in (6, 7, 8, 9) for p in itertools.product("AT", repeat=m)]
    qs += [c * m for c in "AT" for m in range(6, 16)]
    qb = np.frombuffer("".join(qs).encode(), dtype=np.uint8).copy()
    qo = np.zeros(len(qs) + 1, dtype=np.int64)
    np.cumsum([len(q) for q in qs], out=qo[1:])
    qb_d, qo_d = torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda()
    p = sa.sa_search_params(flags=sa.SA_PARAM_KMER_ORDER if order == "kmer" else sa.SA_PARAM_INPUT_ORDER)
    for text in _texts():
        T = np.frombuffer(text.encode(), dtype=np.uint8)
        osa = oracle.sa_naive(T)
        lo, hi = oracle.search_batch(T, osa, qb, qo)
        idx = sa.sa_build(torch.from_numpy(T.copy()).cuda(), kmer_k=k)
        got = sa.sa_search_batch(idx, qb_d, qo_d, params=p).cpu().numpy()
        bad = np.nonzero((got[:, 0] != lo) | (got[:, 1] != hi))[0]
        assert bad.size == 0, (text, [qs[i] for i in bad[:5]], got[bad[:5]], lo[bad[:5]], hi[bad[:5]])


def test_lengths_around_k_several_references(sa):
    refs = [datagen.reference(n, 900 + n, gc=0.45, tandem_cover=0.1) for n in (30_000, 5_000)]
    idxs = [sa.sa_build(torch.from_numpy(refs[0]).cuda()), sa.sa_build(torch.from_numpy(refs[1]).cuda(), kmer_k=0)]
    qb, qo, _ = datagen.queries(refs[0], 20_000, 901, m=(1, 12), frac_sampled=0.7)
    q_ref = np.random.default_rng(902).integers(0, 2, 20_000).astype(np.uint32)
    got = sa.sa_search_batch(idxs, torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda(),
                             q_ref=torch.from_numpy(q_ref).cuda()).cpu().numpy()
    for i, r in enumerate(refs):
        T = oracle.normalize(r)
        lo, hi = oracle.search_batch(T, oracle.sa_naive(T), qb, qo, threads=oracle.cpu_threads())
        s = q_ref == i
        assert np.array_equal(got[s, 0], lo[s]) and np.array_equal(got[s, 1], hi[s]), i
