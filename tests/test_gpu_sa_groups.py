"""The suffix array's small groups are ordered by compares in the text, its
large ones by sorts of their next bases, long repeats by prefix doubling.
Texts whose groups of suffixes with equal first 16 bases are around 32
members, whose common prefixes are around 16 bases, a window and the compares'
limit, that end inside a repeat or in a run of A's, and sizes around a block's
items: the array must be the oracle's.  One larger text takes the sorts by
groups too, and must equal the DC3 construction's array."""
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


def _check(sa, text, width=32):
    T = np.ascontiguousarray(text)
    got = sa.sa_suffix_array_gpu(torch.from_numpy(T.copy()).cuda(), width=width).cpu().numpy().astype(np.int64)
    assert np.array_equal(got, oracle.sa_naive(oracle.normalize(T)))


@pytest.mark.parametrize("copies", [2, 3, 31, 32, 33, 34, 64, 65])
@pytest.mark.parametrize("length", [15, 16, 17, 31, 48, 49, 80, 300, 1100])
def test_group_sizes_and_prefixes(sa, copies, length):
    rng = np.random.default_rng(copies * 1000 + length)
    unit = datagen.ASCII[rng.integers(0, 4, length)]
    parts = []
    for c in range(copies):
        parts += [unit, datagen.ASCII[rng.integers(0, 4, int(rng.integers(1, 20)))]]
    _check(sa, np.concatenate(parts[:-1]))            # ends with a whole copy
    _check(sa, np.concatenate(parts + [unit[:length // 2]]))  # ends inside one
    _check(sa, np.concatenate(parts + [np.full(40, 65, np.uint8)]), width=64)  # ends in a run of A's


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 447, 448, 449, 480, 895, 896, 897])
def test_sizes_and_runs(sa, n):
    rng = np.random.default_rng(n)
    for text in (np.full(n, 65), np.full(n, 84), np.resize([65, 67], n), datagen.ASCII[rng.integers(0, 4, n)],
                 np.concatenate([datagen.ASCII[rng.integers(0, 2, n)], np.full(n, 65)])):
        _check(sa, text.astype(np.uint8))


@pytest.mark.parametrize("width", [32, 64])
def test_group_sorts_of_a_large_text(sa, width):
    ref = datagen.reference(26_000_001, 41, gc=0.41, family_cover=0.45, tandem_cover=0.05, sd_cover=0.1)
    ref[-5000:] = ref[1000:6000]  # a repeat at the end
    t = torch.from_numpy(ref).cuda()
    assert torch.equal(sa.sa_suffix_array_gpu(t, width=width), sa.sa_suffix_array_gpu(t, width=width, dc3=True))
