"""The search kernels of sa_search_locate add up each locate tile's kept counts.
With no cap to speak of and queries that match everywhere, 32 queries' counts
pass 2^32: the offsets must be the 64-bit prefix sums all the same, on every
path that adds them."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
N = 140_000_003  # 32 N > 2^32


@pytest.fixture(scope="module")
def env():
    from paper_1303_3692_gb300 import build_lib
    from paper_1303_3692_gb300 import sa

    build_lib.build()
    g = torch.Generator(device="cuda").manual_seed(11)
    codes = torch.randint(0, 4, (N,), device="cuda", dtype=torch.uint8, generator=g)
    text = torch.tensor([65, 67, 71, 84], dtype=torch.uint8, device="cuda")[codes.to(torch.int32)]
    idx = sa.sa_build(text, kmer_k=8)
    del text, codes
    torch.cuda.empty_cache()
    return sa, idx


@pytest.mark.parametrize("path", ["one-kernel", "input-order", "kmer-order"])
@pytest.mark.parametrize("n_q", [5003, 200_003])  # a few queries a warp in the one kernel, and 32
@pytest.mark.parametrize("cap", [0xFFFFFFFF, 0xFFFFFFFF // 32 + 1, 0xFFFFFFFF // 32, 7])
def test_offsets_are_64_bit_sums(env, path, cap, n_q):
    sa, idx = env
    m = np.where(np.arange(n_q) % 97 == 0, 1, 0)  # empty queries match at every rank
    qo = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum(m, out=qo[1:])
    bases = torch.full((int(qo[-1]),), 65, dtype=torch.uint8, device="cuda")
    offs = torch.from_numpy(qo).cuda()
    out = torch.empty((n_q, sa.RESULT_FIELDS), dtype=torch.int64, device="cuda")
    loc = torch.empty(n_q + 1, dtype=torch.int64, device="cuda")
    p = sa.sa_search_params(front_probes=1 if path == "input-order" else 0,
                            flags=sa.SA_PARAM_KMER_ORDER if path == "kmer-order" else 0)
    refs = (ctypes.c_void_p * 1)(idx.handle.value)
    st = sa.lib().sa_search_locate(refs, 1, bases.data_ptr(), offs.data_ptr(), None, n_q, out.data_ptr(), cap,
                                   loc.data_ptr(), None, 0, torch.cuda.current_stream().cuda_stream, ctypes.byref(p))
    assert st == sa.SA_OK
    counts = out[:, 2].cpu().numpy()
    assert (counts[m == 0] == N).all()
    want = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum(np.minimum(counts, cap), out=want[1:])
    assert np.array_equal(loc.cpu().numpy(), want)
