"""Both strands of a batch are read from one packing, and its validity from a
bitmap of the words that hold a non-base byte: queries of lengths around a
packed word's 32 bases, a warp's 1024 and the record boundaries, at the very
start and end of the batch, forward and reverse-complemented, with an N at
their first, last and middle base and just outside them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu
COMP = np.zeros(256, dtype=np.uint8)
for _a, _b in zip(b"ACGTN", b"TGCAN"):
    COMP[_a] = _b


@pytest.fixture(scope="module")
def sa():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa as sa_mod

    build_lib.build()
    return sa_mod


@pytest.mark.parametrize("order", ["kmer", "input"])
@pytest.mark.parametrize("with_n", [False, True])
@pytest.mark.parametrize("shift", [0, 5])  # the batch's bases on and off a 16-byte boundary
def test_lengths_around_words(sa, order, with_n, shift):
    ref = datagen.reference(30_000, 7, gc=0.5, sd_cover=0.2)
    T = oracle.normalize(ref)
    osa = oracle.sa_naive(T)
    idx = sa.sa_build(torch.from_numpy(ref.copy()).cuda())
    rng = np.random.default_rng(11)
    lens = [1, 2, 9, 31, 32, 33, 63, 64, 65, 96, 97, 127, 128, 129, 159, 160, 161, 191, 192, 193, 224, 1000, 1023,
            1024, 1025, 2100]
    qs = []
    for m in [5] + lens + lens[::-1] + [40, 3]:
        s = int(rng.integers(0, ref.size - m + 1))
        qs.append(ref[s:s + m].copy())
    rc = np.arange(len(qs)) % 2 == 1
    rc[0] = rc[1] = True  # the batch starts with queries of the other strand
    fed = [COMP[q][::-1].copy() if r else q.copy() for q, r in zip(qs, rc)]
    bad = np.zeros(len(qs), dtype=bool)
    if with_n:
        for i in range(2, len(qs), 3):  # the neighbours of a marked query stay valid
            fed[i][{0: 0, 1: fed[i].size - 1, 2: fed[i].size // 2}[i % 4 % 3]] = ord("N")
            bad[i] = True
    qb = np.concatenate([np.full(shift, ord("A"), np.uint8)] + fed)
    qo = np.zeros(len(qs) + 1, dtype=np.int64)
    np.cumsum([q.size for q in qs], out=qo[1:])
    qo += shift
    flags = sa.SA_PARAM_STRAND_PER_QUERY | (sa.SA_PARAM_KMER_ORDER if order == "kmer" else sa.SA_PARAM_INPUT_ORDER)
    q_ref = np.where(rc, sa.STRAND_BIT, 0).astype(np.uint32)
    got = sa.sa_search_batch(idx, torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda(),
                             q_ref=torch.from_numpy(q_ref).cuda(), params=sa.sa_search_params(flags=flags)).cpu().numpy()
    plain = sa.sa_search_batch_plain(idx, torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda()).cpu().numpy()
    for i, q in enumerate(qs):
        if bad[i]:
            assert got[i].tolist() == [-1, -1, -1, sa.SA_RESULT_INVALID], i
            assert plain[i].tolist() == [-1, -1, -1, sa.SA_RESULT_INVALID], i
        else:
            lo, hi = oracle.search(T, osa, q)
            assert hi > lo and got[i].tolist() == [lo, hi, hi - lo, 0], (i, q.size)
            assert plain[i, :2].tolist() == list(oracle.search(T, osa, fed[i])), (i, q.size)
