"""The one-kernel search of small batches with queries of any length.  Who checks
that a query's bytes are bases depends on its length -- its lane, its warp, its
CTA, a kernel over the whole grid -- and a batch of very long queries takes the
other path: results, marks and locate offsets equal the other path's at the
lengths where that changes, and one long query costs no more than a few times
what it costs there.  Batches whose brackets hold many suffixes are small up to
fewer queries: that path is known by the scratch it takes, none here."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
N = 12_000_000
LENGTHS = [1, 127, 128, 129, 511, 512, 513, 700, 8191, 8192, 8193, 9000, (1 << 17) - 1, 1 << 17, (1 << 17) + 1, 140_000]


@pytest.fixture(scope="module")
def env():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa

    build_lib.build()
    g = torch.Generator(device="cuda").manual_seed(12)
    codes = torch.randint(0, 4, (N,), device="cuda", dtype=torch.uint8, generator=g)
    codes[5_000_000:9_000_000] = codes[:4_000_000]  # long queries match twice, or tie for long
    codes[9_500_000:9_600_000] = 2
    text = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")[codes.to(torch.int32)]
    return sa, text.cpu().numpy(), [sa.sa_build(text), sa.sa_build(text, kmer_k=4)]


def batch(text, lens, seed):
    """Copies of the text, some with one base changed and some with an N, at the
    ends and at the 16-byte steps around the lengths above."""
    rng = np.random.default_rng(seed)
    qo = np.zeros(len(lens) + 1, dtype=np.int64)
    np.cumsum(lens, out=qo[1:])
    qb = np.empty(int(qo[-1]), dtype=np.uint8)
    for q, m in enumerate(lens):
        s = int(rng.integers(0, min(4_000_000, N - m) if q % 2 else N - m + 1))
        p = text[s:s + m].copy()
        at = int(rng.choice([0, m - 1, m // 2, min(m - 1, 127), min(m - 1, 130), max(0, m - 17)]))
        if q % 5 == 1:
            p[at] = ord("A") if p[at] != ord("A") else ord("C")
        elif q % 5 == 3:
            p[at] = ord("N")
        qb[qo[q]:qo[q + 1]] = p
    return qb, qo


def other(sa, flags=0):
    """Parameters that select the path of large batches."""
    return sa.sa_search_params(front_probes=1, flags=flags)


# one batch below the size from which the whole grid checks the longest, one above
@pytest.mark.parametrize("repeat", [2, 22])
@pytest.mark.parametrize("shift", [0, 5])
@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("revcomp", [False, True])
def test_lengths(env, repeat, shift, which, revcomp):
    sa, text, idxs = env
    lens = LENGTHS * repeat + [33] * 41
    qb, qo = batch(text, lens, repeat + shift)
    assert (qo[-1] > 1 << 23) == (repeat > 2)
    if revcomp:
        comp = np.full(256, ord("N"), dtype=np.uint8)
        comp[list(b"ACGT")] = list(b"TGCA")
        for q in range(len(lens)):
            qb[qo[q]:qo[q + 1]] = comp[qb[qo[q]:qo[q + 1]]][::-1]
    bases = torch.from_numpy(np.concatenate([np.full(shift, 65, np.uint8), qb])).cuda()
    offs = torch.from_numpy(qo + shift).cuda()
    flags = sa.SA_PARAM_REVERSE_COMPLEMENT if revcomp else 0
    got = []
    for p in (sa.sa_search_params(flags=flags), other(sa, flags)):
        status = torch.full((1,), 77, dtype=torch.int32, device="cuda")
        p.device_status = status.data_ptr()
        out, loc, pos = sa.sa_search_locate(idxs[which], bases, offs, 5, params=p)
        k = int(loc[-1])
        got.append((out.cpu(), loc.cpu(), pos[:k].cpu(), int(status)))
    assert torch.equal(got[0][0], got[1][0])
    assert torch.equal(got[0][1], got[1][1]) and torch.equal(got[0][2], got[1][2])
    assert got[0][3] == got[1][3] == sa.SA_ERR_BASE
    invalid = got[0][0][:, 3] == sa.SA_RESULT_INVALID
    assert torch.equal(invalid, torch.from_numpy(np.arange(len(lens)) % 5 == 3))


def test_long_queries_that_overlap(env):
    """Offsets that go back: more long queries than their bases would allow."""
    sa, text, idxs = env
    n = 9_000_000
    qb = text[:n].copy()
    qb[7_000_000] = ord("N")
    qo = np.array([0, 6_500_000] + [0, n] * 3 + [0, 100, 200_000, 6_999_990, 7_000_010, n], dtype=np.int64)
    # and short ones, so that the batch's mean length is a small batch's
    qo = np.concatenate([qo[:-1], np.arange(7_000_020, 7_000_020 + 40 * 900, 40), [n]])
    bases, offs = torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda()
    got = [sa.sa_search_batch(idxs[0], bases, offs, params=p).cpu() for p in (sa.sa_search_params(), other(sa))]
    assert torch.equal(got[0], got[1])
    assert got[0][:9, 3].tolist() == [0, 1, 1, 1, 1, 1, 1, 1, 0]


def shortest(f):
    f()
    ts = []
    for _ in range(7):
        torch.cuda.synchronize()
        t = time.perf_counter()
        f()
        torch.cuda.synchronize()
        ts.append(time.perf_counter() - t)
    return min(ts)


# random queries: a compare ends at once, so what is timed is the call and the check of every byte
@pytest.mark.parametrize("lens", [[100_000] * 20, [1_000_000], [60_000_000], [100] * 20_000 + [1_000_000],
                                  [100] * 500_000 + [10_000_000], [20] * 65_000 + [60_000_000]],
                         ids=["20x1e5", "1x1e6", "1x6e7", "20000x100+1e6", "500000x100+1e7", "65000x20+6e7"])
def test_one_long_query_costs_little(env, lens):
    sa, _, idxs = env
    g = torch.Generator(device="cuda").manual_seed(13)
    offs = torch.zeros(len(lens) + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.tensor(lens, device="cuda"), 0, out=offs[1:])
    letters = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")
    bases = letters[torch.randint(0, 4, (int(offs[-1]),), device="cuda", generator=g)]
    out = torch.empty((len(lens), sa.RESULT_FIELDS), dtype=torch.int64, device="cuda")
    mine = shortest(lambda: sa.sa_search_batch(idxs[0], bases, offs, out=out))
    p = other(sa)
    theirs = shortest(lambda: sa.sa_search_batch(idxs[0], bases, offs, out=out, params=p))
    assert mine < 3 * theirs, (mine * 1e6, theirs * 1e6)


# n = 12,000,000: 187,500 suffixes per k-mer at k = 3, 183 and 45 around the line
# at 128, 11 and 2.9 around the one at 8
@pytest.mark.parametrize("k, most", [(0, 1 << 15), (3, 1 << 15), (8, 1 << 15), (9, 1 << 17), (10, 1 << 17), (11, 1 << 19),
                                     (None, 1 << 19)])
def test_wide_brackets_are_small_batches_of_fewer_queries(env, k, most):
    sa, text, _ = env
    idx = sa.sa_build(torch.from_numpy(text).cuda(), kmer_k=k)
    rng = np.random.default_rng(14)
    at = rng.integers(0, N - 40, most + 1)
    qb = text[at[:, None] + np.arange(40)]
    swap = rng.random(most + 1) < 0.3
    qb[swap, rng.integers(0, 40, int(swap.sum()))] = ord("G")
    bases = torch.from_numpy(qb.reshape(-1)).cuda()
    for n_q in (most, most + 1):
        offs = torch.arange(0, 40 * n_q + 1, 40, device="cuda", dtype=torch.int64)
        torch.cuda.synchronize()
        sa.sa_scratch_info(reset_high=True)
        got = sa.sa_search_batch(idx, bases, offs)
        torch.cuda.synchronize()
        assert (sa.sa_scratch_info()["used_high"] == 0) == (n_q <= most)
        assert torch.equal(got, sa.sa_search_batch(idx, bases, offs, params=other(sa)))
