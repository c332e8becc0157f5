"""The common prefixes that suffix records and k-mer entries carry let a probe
settle the ranks beside it unread; they are cut at 255.  Texts with exact
repeats of lengths around the record (104 bases), its four windows (128), the
entry (192) and the cut, searched by queries of lengths around them, and sizes
around the 30 ranks a warp makes: every result must equal the oracle's, in
both orders and for every probe budget of the first pass."""
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


def _check(sa, ref, qs, kmer_k=None):
    T = oracle.normalize(ref)
    osa = oracle.sa_naive(T)
    qb = np.frombuffer(b"".join(qs), dtype=np.uint8).copy()
    qo = np.zeros(len(qs) + 1, dtype=np.int64)
    np.cumsum([len(q) for q in qs], out=qo[1:])
    lo, hi = oracle.search_batch(T, osa, qb, qo, threads=oracle.cpu_threads())
    idx = sa.sa_build(torch.from_numpy(ref.copy()).cuda(), kmer_k=kmer_k)
    for flags in (sa.SA_PARAM_INPUT_ORDER, sa.SA_PARAM_KMER_ORDER):
        if kmer_k == 0 and flags == sa.SA_PARAM_KMER_ORDER:
            continue
        for probes in (1, 3, 64):
            got = sa.sa_search_batch(idx, torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda(),
                                     params=sa.sa_search_params(flags=flags, front_probes=probes)).cpu().numpy()
            bad = np.nonzero((got[:, 0] != lo) | (got[:, 1] != hi))[0]
            assert bad.size == 0, (flags, probes, bad[:5], got[bad[:5]], lo[bad[:5]], hi[bad[:5]])


@pytest.mark.parametrize("rep", [103, 104, 105, 127, 128, 129, 191, 192, 193, 254, 255, 256, 300])
@pytest.mark.parametrize("kmer_k", [None, 2, 0])
def test_repeats_around_the_prefix_cut(sa, rep, kmer_k):
    ref = datagen.reference(4000, 500 + rep, gc=0.5)
    block = ref[100:100 + rep].copy()
    for at in (700, 1500, 2600, 4000 - rep):  # copies with different neighbours, one at the text's end
        ref[at:at + rep] = block
    rng = np.random.default_rng(rep)
    qs = []
    for m in (20, rep - 1, rep, rep + 1, rep + 2, 250, 254, 255, 256, 257, 400):
        for at in (100, 700, 1500, 2600, 4000 - rep):
            for shift in (-1, 0, 1):
                s = at + shift
                q = ref[s:s + m]
                if 0 <= s and q.size:
                    qs.append(q.tobytes())
                    c = q.copy()
                    p = int(rng.integers(0, c.size))
                    c[p] = datagen.ASCII[(int(np.nonzero(datagen.ASCII == c[p])[0][0]) + 1 + int(rng.integers(0, 3))) % 4]
                    qs.append(c.tobytes())
                    qs.append(q.tobytes() + b"ACGT"[at % 4:at % 4 + 1])
    _check(sa, ref, qs, kmer_k)


@pytest.mark.parametrize("n", [1, 2, 29, 30, 31, 32, 59, 60, 61, 89, 90, 91])
def test_sizes_around_a_warps_ranks(sa, n):
    rng = np.random.default_rng(n)
    for text in ("A" * n, ("AC" * n)[:n], "".join(rng.choice(list("ACGT"), n)), "".join(rng.choice(list("AT"), n))):
        ref = np.frombuffer(text.encode(), dtype=np.uint8).copy()
        qs = [text[s:s + m].encode() for m in (1, 2, 3, 7, n) for s in range(0, n, 3)]
        qs += [q + b"A" for q in qs[:20]] + [b"T" + q for q in qs[:20]]
        _check(sa, ref, [q for q in qs if q])


@pytest.mark.parametrize("n", [63, 64, 65, 95, 96, 97, 127, 128, 129, 159, 160, 161, 191, 192, 193, 223, 224, 225, 256, 257])
def test_windows_at_the_texts_end(sa, n):
    # the windows of records (4 words on from a suffix) and entries (3 more) come
    # by pairs of words: the last pairs of the text, at either parity
    ref = datagen.reference(n, n, gc=0.5)
    qs = [ref[s:s + m].tobytes() for s in range(n) for m in (40, 100, 104, 105, 128, 192, n) if s + m <= n]
    qs += [q + b"A" for q in qs[::5]] + [q[:-1] + b"T" for q in qs[::7]]
    _check(sa, ref, qs, 2)
    _check(sa, ref, qs)
