"""The autotuner times the call that sets nothing beside those that choose a
launch shape: a batch of few queries runs as one kernel only without knobs."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_1303_3692_gb300 import autotune


def test_first_candidate_sets_nothing():
    p = autotune.params_from(autotune.DEFAULT_CANDIDATES[0])
    assert [p.threads_per_block, p.blocks_per_sm, p.key_depth, p.chunk, p.front_probes] == [0] * 5


def test_few_and_many_queries_are_cached_apart():
    refs = [types.SimpleNamespace(n=10, width=4, kmer_k=2)]
    few, most, many = (autotune.cache_key("gpu", refs, 100.0, n) for n in (20, 1 << 19, (1 << 19) + 1))
    assert few == most != many


@pytest.mark.gpu
def test_small_batch_is_left_to_the_default(tmp_path):
    from paper_1303_3692_gb300 import build_lib, datagen, sa

    build_lib.build()
    r = datagen.reference(300_000, 21)
    idx = sa.sa_build(torch.from_numpy(r.copy()).cuda())
    qb, qo, _ = datagen.queries(r, 20_000, 22, m=(20, 200), frac_sampled=0.7, subs=(0, 1))
    bases, offs = torch.from_numpy(qb).cuda(), torch.from_numpy(qo).cuda()
    p, rep = autotune.autotune(idx, bases, offs, reps=7, cache_path=str(tmp_path / "tune.json"))
    assert rep["best"] == [0, 0, 0, 0, 0] and len(rep["all"]) == len(autotune.DEFAULT_CANDIDATES)
    torch.cuda.synchronize()
    sa.sa_scratch_info(reset_high=True)
    sa.sa_search_batch(idx, bases, offs, params=p)
    torch.cuda.synchronize()
    assert sa.sa_scratch_info()["used_high"] == 0  # the one kernel takes none
