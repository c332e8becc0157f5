"""Small batches run in one kernel (packing included), large ones through the
packing, the first and the persistent pass; setting a knob of the latter
selects them for a small batch too.  Both must give the oracle's results on
batches of one query up to several per warp and tile, with every length around
the packed words and the records, wide brackets (tandem and long repeats),
indexes without a k-mer table, both strands, empty and invalid queries, bad
offsets and reference ids, bases on and off an aligned address, and locate."""
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
def refs(sa):
    out = []
    for n, k in ((150_000, None), (90_000, 3), (40_000, 0)):  # k = 3: brackets of 1400 suffixes
        r = datagen.reference(n, 600 + n, gc=0.45, sd_cover=0.2, tandem_cover=0.15)
        r[-2000:] = r[500:2500]
        T = oracle.normalize(r)
        out.append((r, T, oracle.sa_naive(T), sa.sa_build(torch.from_numpy(r.copy()).cuda(), kmer_k=k)))
    return out


@pytest.mark.parametrize("n_q", [1, 2, 31, 33, 700, 4096, 4097, 40_000])
@pytest.mark.parametrize("shift", [0, 3])
def test_against_oracle_and_the_other_path(sa, refs, n_q, shift):
    rng = np.random.default_rng(n_q + shift)
    lens = np.array([1, 2, 5, 9, 31, 32, 33, 64, 96, 97, 103, 104, 105, 128, 129, 160, 192, 193, 260, 700])
    q_ref = rng.integers(0, 3, n_q).astype(np.uint32)
    rc = rng.random(n_q) < 0.5
    fed, want = [], []
    for q in range(n_q):
        r = refs[q_ref[q]][0]
        m = int(rng.choice(lens))
        s = int(rng.integers(0, r.size - m + 1)) if rng.random() < 0.9 else r.size - m
        p = r[s:s + m].copy()
        if rng.random() < 0.3:
            p[int(rng.integers(0, m))] = datagen.ASCII[int(rng.integers(0, 4))]
        want.append(p)
        f = COMP[p][::-1].copy() if rc[q] else p.copy()
        if rng.random() < 0.02:
            f[int(rng.integers(0, m))] = ord("N")
            want[-1] = None
        if rng.random() < 0.02:
            f, want[-1] = f[:0], f[:0]
        fed.append(f)
    qb = np.concatenate([np.full(shift, 65, np.uint8)] + fed + [np.zeros(0, np.uint8)])
    qo = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum([f.size for f in fed], out=qo[1:])
    qo += shift
    ids = q_ref | np.where(rc, sa.STRAND_BIT, 0).astype(np.uint32)
    if n_q > 10:
        ids[7], want[7] = 3, None  # no such reference
    qb_d = torch.from_numpy(qb if qb.size else np.zeros(1, np.uint8)).cuda()
    qo_d, ids_d = torch.from_numpy(qo).cuda(), torch.from_numpy(ids).cuda()
    idxs = [x[3] for x in refs]
    got = []
    for kw in ({}, {"front_probes": 3}):
        st = torch.full((1,), 77, dtype=torch.int32, device="cuda")
        p = sa.sa_search_params(flags=sa.SA_PARAM_STRAND_PER_QUERY, device_status=st.data_ptr(), **kw)
        res, offs, pos = sa.sa_search_locate(idxs, qb_d, qo_d, 5, q_ref=ids_d, params=p)
        total = int(offs[-1].item())
        got.append((res.cpu().numpy(), offs.cpu().numpy(), pos[:total].cpu().numpy(), int(st.item())))
    for a, b in zip(got[0], got[1]):
        assert np.array_equal(a, b)
    res, offs, pos, _ = got[0]
    for q in range(0, n_q, max(1, n_q // 3000)):
        if want[q] is None:
            assert res[q].tolist() == [-1, -1, -1, sa.SA_RESULT_INVALID], q
            continue
        _, T, osa, idx = refs[q_ref[q]]
        lo, hi = (0, T.size) if want[q].size == 0 else oracle.search(T, osa, want[q])
        assert res[q, :3].tolist() == [lo, hi, hi - lo], (q, want[q].size)
        assert pos[offs[q]:offs[q + 1]].tolist() == osa[lo:lo + min(hi - lo, 5)].tolist(), q


def test_offsets_outside_the_batch(sa, refs):
    idx = refs[0][3]
    qb = torch.from_numpy(refs[0][0][:300].copy()).cuda()
    qo = torch.tensor([0, 40, 30, 100, 500, 120, 200], dtype=torch.int64, device="cuda")
    got = []
    for kw in ({}, {"front_probes": 3}):
        p = sa.sa_search_params(flags=sa.SA_PARAM_Q_RANGE, q_first=0, q_total=200, **kw)
        got.append(sa.sa_search_batch(idx, qb, qo, params=p).cpu())
    assert torch.equal(got[0], got[1])
    assert got[0][:, 3].tolist() == [0, 1, 0, 1, 1, 0]
