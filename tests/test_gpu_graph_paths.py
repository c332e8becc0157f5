"""CUDA-graph capture of search + locate on every path a batch can take: the one
kernel with the check of its longest queries, input order with a packed batch,
k-mer order from the ASCII bases (with a tile that does not fit) and from a
packed batch.  Replays over other bases -- with and without Ns -- give what plain
calls give."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1303_3692_gb300 import datagen

pytestmark = pytest.mark.gpu

PATHS = {
    "one-kernel": ([1100] * 4000 + [50_000], {}),
    "input-order": ([100] * 4000 + [700] * 50, {"front_probes": 1}),
    "kmer-order": ([100] * 2000 + [99_000] + [150] * 2000, {"order": True}),
    "kmer-order-packed": ([250] * 4000, {"order": True}),
}


@pytest.mark.parametrize("path", list(PATHS))
@pytest.mark.parametrize("strands", [False, True])
def test_capture(path, strands):
    from paper_1303_3692_gb300 import build_lib, sa

    build_lib.build()
    ref = datagen.reference(200_000, 31, sd_cover=0.2, tandem_cover=0.1)
    idx = sa.sa_build(torch.from_numpy(ref.copy()).cuda())
    lens, knobs = PATHS[path]
    n_q, rng = len(lens), np.random.default_rng(5)
    qo = np.zeros(n_q + 1, dtype=np.int64)
    np.cumsum(lens, out=qo[1:])

    def batch(with_n):
        qb = np.concatenate([ref[s:s + m] for m in lens for s in [int(rng.integers(0, ref.size - m + 1))]])
        qb[rng.integers(0, qb.size, n_q // 2)] = ord("G")
        if with_n:
            qb[rng.integers(0, qb.size, n_q // 20)] = ord("N")
            qb[qo[lens.index(max(lens))] + max(lens) // 2] = ord("N")
        return torch.from_numpy(qb).cuda()

    contents = [batch(False), batch(True), batch(False)]
    bases, offs = contents[0].clone(), torch.from_numpy(qo).cuda()
    ids = torch.from_numpy(np.where(rng.random(n_q) < 0.5, sa.STRAND_BIT, 0).astype(np.uint32)).cuda() if strands else None
    out = torch.empty((n_q, sa.RESULT_FIELDS), dtype=torch.int64, device="cuda")
    loc_off = torch.empty(n_q + 1, dtype=torch.int64, device="cuda")
    loc_pos = torch.empty(n_q * 8, dtype=torch.int32, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    p = sa.sa_search_params(front_probes=knobs.get("front_probes", 0), q_total=int(qo[-1]),
                            flags=sa.SA_PARAM_Q_RANGE | (sa.SA_PARAM_KMER_ORDER if "order" in knobs else 0)
                            | (sa.SA_PARAM_STRAND_PER_QUERY if strands else 0), device_status=status.data_ptr())

    def call():
        sa.sa_search_locate(idx, bases, offs, 8, q_ref=ids, out=out, out_offsets=loc_off, out_pos=loc_pos,
                            capacity=loc_pos.numel(), params=p)

    s = torch.cuda.Stream()
    with torch.cuda.stream(s):  # warm up (kernel attributes, pool) outside capture
        call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call()
    for c in (contents[1], contents[0], contents[2]):
        bases.copy_(c)
        for x in (out, loc_off, loc_pos, status):
            x.fill_(99)
        g.replay()
        torch.cuda.synchronize()
        k = int(loc_off[-1])
        got = [out.clone(), loc_off.clone(), loc_pos[:k].clone(), status.clone()]
        call()
        torch.cuda.synchronize()
        for a, b in zip(got, (out, loc_off, loc_pos[:k], status)):
            assert torch.equal(a, b)
        assert int(status) == (sa.SA_ERR_BASE if c is contents[1] else sa.SA_OK)
        assert int((out[:, 3] == sa.SA_RESULT_INVALID).sum()) >= (n_q // 40 if c is contents[1] else 0)
