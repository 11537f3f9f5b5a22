"""The batched sweep times what it can change: the raster strip (bm) of each
size class, once each; bn and bk, which reach no kernel, are the class's own."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import tuning

pytestmark = pytest.mark.gpu


@pytest.fixture
def table(alp):
    old = [alp.alp_batched_get_class_config(c) for c in range(9)]
    yield old
    for c, cfg in enumerate(old):
        alp.alp_batched_set_class_config(c, *cfg)


@pytest.mark.parametrize("tiles,bks", [((32, 64, 128), (16, 32)), ((64, 32), (16,))])
def test_each_strip_is_timed_once(alp, table, monkeypatch, tiles, bks):
    import torch
    sizes = [(20, 24, 40), (64, 64, 9), (33, 200, 17), (130, 20, 5), (300, 129, 64), (100, 31, 33)]
    M, N, K = (np.array(x, dtype=np.int64) for x in zip(*sizes))
    buf = [[torch.ones(int(a) * int(b), dtype=torch.float64, device="cuda")
            for a, b in zip(x, y)] for x, y in ((M, K), (K, N), (M, N))]
    ptrs = [np.array([t.data_ptr() for t in b], dtype=np.int64) for b in buf]
    timed = []
    call = alp.alp_gemm_batched_varsize
    monkeypatch.setattr(alp, "alp_gemm_batched_varsize",
                        lambda n, *a, **k: (timed.append(n), call(n, *a, **k))[1])
    res = tuning.tune_batched_classes(M, N, K, *ptrs, runs=2, tiles=tiles, bks=bks)
    classes = {alp.alp_batched_class_of(int(m), int(n)) for m, n in zip(M, N)}
    assert set(res) == classes and len(classes) > 2
    for c, (win, ms, times) in res.items():
        assert [k[0] for k in times] == list(tiles)
        bn, bk = table[c][1], table[c][2]
        expected = (bn if bn in tiles else tiles[0], bk if bk in bks else bks[0])
        assert {k[1:] for k in times} == {expected}
        assert alp.alp_batched_get_class_config(c) == win and ms == times[win] > 0
    # a warm-up and two runs of each strip, then of at most three whole tables
    assert timed.count(len(sizes)) <= 9
    assert len(timed) - timed.count(len(sizes)) == 3 * len(tiles) * len(classes)
    assert alp.alp_get_device_error() == alp.ALP_OK
