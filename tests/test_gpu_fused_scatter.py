"""In k-mer order a batch of up to 192 bases per query on average is packed by
the scatter's own tiles.  Batches around that average and around a tile's room
(98,304 bases per 512 queries), with one query longer than a tile, queries of
lengths around the 192 bases a record carries, Ns, empty queries, both strands,
offsets that go back, and bases on and off an aligned address: equal to the
input order's results and to the oracle."""
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


@pytest.fixture(scope="module")
def ref(sa):
    r = datagen.reference(120_000, 77, gc=0.45, sd_cover=0.2, tandem_cover=0.05)
    T = oracle.normalize(r)
    return r, T, oracle.sa_naive(T), sa.sa_build(torch.from_numpy(r.copy()).cuda())


@pytest.mark.parametrize("lens", [[150], [192], [191, 193], [1, 2, 9, 31, 33, 64, 127, 129, 191, 192, 193, 260],
                                  [20] * 700 + [100_000] + [20] * 700, [193]],
                         ids=["150", "192", "around192", "mixed", "longer-than-a-tile", "193-packed"])
@pytest.mark.parametrize("shift", [0, 7])
def test_tiles(sa, ref, lens, shift):
    r, T, osa, idx = ref
    rng = np.random.default_rng(len(lens) + shift)
    n_q = 1537 if len(lens) < 100 else len(lens)
    fed, want = [], []
    rc = rng.random(n_q) < 0.5
    for q in range(n_q):
        m = lens[q % len(lens)]
        s = int(rng.integers(0, r.size - m + 1))
        p = r[s:s + m].copy()
        if rng.random() < 0.3:
            p[int(rng.integers(0, m))] = datagen.ASCII[int(rng.integers(0, 4))]
        f = COMP[p][::-1].copy() if rc[q] else p.copy()
        if rng.random() < 0.03:
            f[int(rng.choice([0, m - 1, m // 2]))] = ord("N")
            p = None
        elif rng.random() < 0.02:
            f = p = f[:0]
        fed.append(f)
        want.append(p)
    qb = np.concatenate([np.full(shift, 65, np.uint8)] + fed)
    qo = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum([f.size for f in fed], out=qo[1:])
    qo += shift
    ids = np.where(rc, sa.STRAND_BIT, 0).astype(np.uint32)
    got = []
    for order in (sa.SA_PARAM_KMER_ORDER, sa.SA_PARAM_INPUT_ORDER):
        p = sa.sa_search_params(flags=order | sa.SA_PARAM_STRAND_PER_QUERY)
        got.append(sa.sa_search_batch(idx, torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda(),
                                      q_ref=torch.from_numpy(ids).cuda(), params=p).cpu().numpy())
    assert np.array_equal(got[0], got[1])
    for q in range(n_q):
        if want[q] is None:
            assert got[0][q].tolist() == [-1, -1, -1, sa.SA_RESULT_INVALID], q
        elif q % 3 == 0:
            lo, hi = (0, T.size) if want[q].size == 0 else oracle.search(T, osa, want[q])
            assert got[0][q].tolist() == [lo, hi, hi - lo, 0], (q, want[q].size)


def test_offsets_that_go_back(sa, ref):
    r, _, _, idx = ref
    qb = torch.from_numpy(r[:60_000].copy()).cuda()
    rng = np.random.default_rng(5)
    qo = np.concatenate([[0], np.cumsum(rng.integers(1, 200, 600)), [5, 45, 30_000, 30_100, 20, 60_000]])
    qo = np.minimum(qo, 60_000).astype(np.int64)
    got = []
    for order in (sa.SA_PARAM_KMER_ORDER, sa.SA_PARAM_INPUT_ORDER):
        p = sa.sa_search_params(flags=order | sa.SA_PARAM_Q_RANGE, q_first=0, q_total=60_000)
        got.append(sa.sa_search_batch(idx, qb, torch.from_numpy(qo).cuda(), params=p).cpu())
    assert torch.equal(got[0], got[1])
    assert got[0][-6:, 3].tolist() == [1, 0, 0, 0, 1, 0]
