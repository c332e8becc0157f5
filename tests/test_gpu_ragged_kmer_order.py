"""K-mer order with some queries far longer than the others.  Tiles of the
scatter whose bases fit its shared memory write the packed words that compares
past the records read; tiles that do not fit are packed and scattered by kernels
of their own.  Results equal input order's (which packs the whole batch) at the
lengths where a record ends, for both strands, with Ns, without a k-mer table
and with offsets that go back; and one long query costs no more than a few times
what it costs there."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu
COMP = np.zeros(256, dtype=np.uint8)
COMP[list(b"ACGTN")] = list(b"TGCAN")


@pytest.fixture(scope="module")
def env():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa

    build_lib.build()
    refs = []
    for n, k in ((700_000, None), (300_000, 0)):  # 0: the key tables' descent
        r = datagen.reference(n, n, gc=0.45, sd_cover=0.2, tandem_cover=0.1)
        r[-150_000:] = r[1000:151_000]  # long queries match twice
        refs.append((r, sa.sa_build(torch.from_numpy(r.copy()).cuda(), kmer_k=k)))
    return sa, refs


MIXES = {
    "records-end": [64, 65, 104, 105, 128, 129, 159, 160, 161, 191, 192, 193, 224, 225, 300],
    "one-tile": [60] * 3000 + [120_000] + [60] * 1000,
    "around-a-tile": [100] * 511 + [98_304 - 51_100] + [60] * 700 + [100] * 511 + [98_304 - 51_100 + 64] + [20] * 900,
    "many": ([40] * 700 + [100_000]) * 4 + [1] * 4000,
    "longest": [30] * 2000 + [149_000] * 2 + [30] * 600,
}


@pytest.mark.parametrize("mix", list(MIXES))
@pytest.mark.parametrize("shift", [0, 9])
@pytest.mark.parametrize("which", ["table", "no-table", "both"])
def test_ragged(env, mix, shift, which):
    sa, refs = env
    rng = np.random.default_rng(len(mix) + shift)
    lens = MIXES[mix] if len(MIXES[mix]) > 100 else MIXES[mix] * 90
    n_q = len(lens)
    ref = {"table": np.zeros(n_q, int), "no-table": np.ones(n_q, int), "both": rng.integers(0, 2, n_q)}[which]
    rc = rng.random(n_q) < 0.5
    fed, bad = [], np.zeros(n_q, dtype=bool)
    for q, m in enumerate(lens):
        r = refs[ref[q]][0]
        at = int(rng.integers(0, r.size - m + 1))
        p = r[at:at + m].copy()
        if rng.random() < 0.4:
            p[int(rng.integers(0, m))] = datagen.ASCII[int(rng.integers(0, 4))]
        if rng.random() < 0.1 or (m > 1000 and q % 2):
            p[int(rng.choice([0, m // 2, m - 1]))] = ord("N")
            bad[q] = True
        fed.append(COMP[p][::-1] if rc[q] else p)
    qo = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum([f.size for f in fed], out=qo[1:])
    bases = torch.from_numpy(np.concatenate([np.full(shift, 67, np.uint8)] + fed)).cuda()
    offs = torch.from_numpy(qo + shift).cuda()
    idxs = [r[1] for r in refs] if which == "both" else [refs[ref[0]][1]]
    ids = torch.from_numpy(np.where(rc, sa.STRAND_BIT, 0).astype(np.uint32) | (ref if which == "both" else 0 * ref).astype(np.uint32)).cuda()
    got = []
    for order in (sa.SA_PARAM_KMER_ORDER, sa.SA_PARAM_INPUT_ORDER):
        p = sa.sa_search_params(flags=order | sa.SA_PARAM_STRAND_PER_QUERY)
        out, loc, pos = sa.sa_search_locate(idxs, bases, offs, 3, q_ref=ids, params=p)
        got.append((out.cpu(), loc.cpu(), pos[:int(loc[-1])].cpu()))
    assert all(torch.equal(a, b) for a, b in zip(*got))
    assert np.array_equal(got[0][0][:, 3].numpy() == sa.SA_RESULT_INVALID, bad)
    assert (got[0][0][:, 2][torch.from_numpy(~bad)] > 0).float().mean() > 0.5


def test_offsets_that_go_back(env):
    """Tiles whose words overlap, more in all than the batch has."""
    sa, refs = env
    qb = refs[0][0][:400_000].copy()
    qb[[3, 350_000]] = ord("N")
    rng = np.random.default_rng(3)
    qo = np.sort(rng.integers(0, 400_000, 4000))
    for at in range(100, 4000, 300):  # a query that starts over, and a long one
        qo[at], qo[at + 1] = 0, 399_000 - at
        qo[at + 2] = 10 + at
    bases, offs = torch.from_numpy(qb).cuda(), torch.from_numpy(qo.astype(np.int64)).cuda()
    got = []
    for order in (sa.SA_PARAM_KMER_ORDER, sa.SA_PARAM_INPUT_ORDER):
        p = sa.sa_search_params(flags=order | sa.SA_PARAM_Q_RANGE, q_first=0, q_total=400_000)
        got.append(sa.sa_search_batch(refs[0][1], bases, offs, params=p).cpu())
    assert torch.equal(got[0], got[1])
    assert 12 <= int((got[0][:, 3] == 1).sum()) < 200


@pytest.mark.parametrize("longest", [1_000_000, 30_000_000])
def test_one_long_query_costs_little(env, longest):
    sa, refs = env
    n_q = 1 << 21
    lens = torch.full((n_q,), 100, device="cuda", dtype=torch.int64)
    lens[77_777] = longest
    offs = torch.zeros(n_q + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=offs[1:])
    g = torch.Generator(device="cuda").manual_seed(4)
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    bases = letters[torch.randint(0, 4, (int(offs[-1]),), device="cuda", generator=g)]
    out = torch.empty((n_q, sa.RESULT_FIELDS), dtype=torch.int64, device="cuda")
    best = []
    for order in (sa.SA_PARAM_KMER_ORDER, sa.SA_PARAM_INPUT_ORDER):
        p = sa.sa_search_params(flags=order)
        ts = []
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            sa.sa_search_batch(refs[0][1], bases, offs, out=out, params=p)
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t)
        best.append(min(ts))
    assert best[0] < 4 * best[1], [b * 1e6 for b in best]
