"""A build gives back what the scratch pool kept of earlier calls before it
allocates the index's arrays, so that memory a search left in the pool never
makes a build fail."""
import pytest

torch = pytest.importorskip("torch")

from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sa():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa as sa_mod

    build_lib.build()
    return sa_mod


@pytest.mark.parametrize("host_text", [False, True])
def test_build_beside_a_full_pool(sa, host_text):
    ref = datagen.reference(2_000_000, 3)
    idx = sa.sa_build(torch.from_numpy(ref.copy()).cuda())
    # a search whose worklist room (64 bytes per query) stays in the pool
    n_q = 1 << 25
    qb = torch.from_numpy(ref[:64].copy()).cuda()
    qo = torch.zeros(n_q + 1, dtype=torch.int64, device="cuda")
    qo[1:] = 20
    p = sa.sa_search_params(front_probes=1)
    out = sa.sa_search_batch(idx, qb, qo, params=p)
    torch.cuda.synchronize()
    kept = sa.sa_scratch_info()["reserved"]
    assert kept >= 64 * n_q
    del out, qb, qo
    torch.cuda.empty_cache()
    # leave too little for the new index (1.1 GB) beside what is kept (2.1 GB)
    free = torch.cuda.mem_get_info()[0]
    ballast = torch.empty(free - (600 << 20), dtype=torch.uint8, device="cuda")
    try:
        text = ref[:1_500_000].copy()
        new = sa.sa_build(text if host_text else torch.from_numpy(text).cuda(), kmer_k=12)  # 1 GB of entries
        assert new.n == 1_500_000
    finally:
        del ballast
        torch.cuda.empty_cache()
