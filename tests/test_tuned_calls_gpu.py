"""Native calls without a config after tuning: the sweep and a loaded cost model
leave them on the register-direct kernels where no config is faster; a config
set by hand is run.  Which kernel ran shows in the bits: at these shapes the
direct kernels share the k range among warps or blocks, so that their sums
have another order than those of any config (checked first)."""
import os

import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs, tuning

pytestmark = pytest.mark.gpu

# the smallest config tile is 64 x 64: at these shapes the best config needs
# twice (512^3) to ten times (64^3) the direct kernels' time
SHAPES = [(64, 64, 64), (200, 150, 1000), (512, 512, 512), (131, 67, 333)]


class Calls:
    """The calls of one shape: plain, and with both operands stored transposed."""

    def __init__(self, alp, M, N, K):
        import torch
        self.alp, self.sizes = alp, (M, N, K)
        A, B, _ = inputs.gemm_operands(8300 + M + N + K, M, N, K, with_c=False)
        t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
        self.A, self.B, self.At, self.Bt = t(A), t(B), t(A.T), t(B.T)
        self.C = torch.empty(M, N, dtype=torch.float64, device="cuda")
        self.ws = alp.alp_gemm_f64_ex_workspace(1, 1, M, N, K)
        self.work = torch.empty(self.ws, dtype=torch.uint8, device="cuda")

    def plain(self, cfg=None):
        M, N, K = self.sizes
        self.C.fill_(float("nan"))
        self.alp.alp_gemm_f64(M, N, K, 1.0, self.A, K, self.B, N, 0.0, self.C, N, cfg)
        return self.C.cpu().numpy()

    def transposed(self):
        M, N, K = self.sizes
        self.C.fill_(float("nan"))
        self.alp.alp_gemm_f64_ex(1, 1, M, N, K, 1.0, self.At, M, self.Bt, K, 0.0, self.C, N, None,
                                 self.work, self.ws)
        return self.C.cpu().numpy()


@pytest.fixture
def clean(alp, monkeypatch):
    monkeypatch.setenv("ALP_TUNE_RUNS", "2")
    alp.alp_tune_clear_cache()
    alp.alp_tune_unload_model()
    yield
    alp.alp_tune_unload_model()
    alp.alp_tune_clear_cache()


@pytest.mark.parametrize("shape", SHAPES)
def test_the_sweep_leaves_calls_on_the_faster_kernels(alp, clean, shape):
    call = Calls(alp, *shape)
    direct = call.plain()
    assert np.array_equal(call.transposed(), direct)
    _, cfg, tflops = alp.alp_tune(*shape, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_EXHAUSTIVE)
    with_config = call.plain(cfg)
    assert not np.array_equal(with_config, direct)   # else nothing below shows anything
    assert np.array_equal(call.plain(), direct)
    assert np.array_equal(call.transposed(), direct)
    # the sweep's winner is still what a lookup answers
    _, found, _ = alp.alp_tune(*shape, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_LOOKUP)
    assert found.astuple() == cfg.astuple() and tflops > 0
    # and a config put into the cache by hand is what runs
    alp.alp_tune_set_cached(*shape, alp.ALP_PATH_NATIVE, cfg)
    assert np.array_equal(call.plain(), with_config)
    assert np.array_equal(call.transposed(), with_config)
    alp.alp_tune_clear_cache()
    assert np.array_equal(call.plain(), direct)


@pytest.mark.parametrize("shape", SHAPES)
def test_a_loaded_model_leaves_calls_on_the_faster_kernels(alp, clean, shape):
    call = Calls(alp, *shape)
    direct = call.plain()
    C = alp.alp_config_count(alp.ALP_PATH_NATIVE) + alp.alp_config_count(alp.ALP_PATH_EMUL)
    alp.alp_tune_load_model(tuning.init_params(C, 1706), C, np.zeros(7, np.float32),
                            np.ones(7, np.float32))
    _, cfg, _ = alp.alp_tune(*shape, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_PREDICT)
    assert not np.array_equal(call.plain(cfg), direct)
    assert np.array_equal(call.plain(), direct)
    assert np.array_equal(call.transposed(), direct)


def test_the_sweep_records_the_direct_kernels(alp, clean, monkeypatch, tmp_path):
    """The database's "direct" entry against the whole call: within the 15 % that
    the configs' proxy is held to, for a split cut and for whole tiles whose k
    and waves are capped."""
    import torch
    db = str(tmp_path / "db.jsonl")
    monkeypatch.setenv("ALP_TUNE_DB", db)
    for M, N, K in ((700, 700, 2000), (2048, 2048, 1024)):
        alp.alp_tune(M, N, K, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_EXHAUSTIVE)
        rec = tuning.load_db(db)[-1]
        assert (rec["M"], rec["N"], rec["K"]) == (M, N, K)
        alp.alp_tune_clear_cache()
        call = Calls(alp, M, N, K)
        ts = []
        for _ in range(4):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            alp.alp_gemm_f64(M, N, K, 1.0, call.A, K, call.B, N, 0.0, call.C, N)
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        assert abs(rec["direct"] / min(ts) - 1) < 0.15, (rec["direct"], ts)
    os.environ.pop("ALP_TUNE_DB", None)


@pytest.mark.parametrize("shape", [(232, 15888, 80), (173, 9398, 79), (3000, 4000, 77),
                                   (1000, 1000, 33), (5000, 3000, 126)])
def test_tuned_calls_of_short_k_are_no_slower(alp, clean, shape):
    """The sweep's proxies at short K: the call that it leaves behind is within 3 %
    (the runs' own spread, and what a proxy may be off between near equals) of the
    call without it.  The two are timed in turn, best of four."""
    import torch
    M, N, K = shape
    call = Calls(alp, M, N, K)
    ts = {True: [], False: []}
    for _ in range(4):
        for tuned in (True, False):
            if tuned:
                alp.alp_tune(M, N, K, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_EXHAUSTIVE)
            else:
                alp.alp_tune_clear_cache()
            alp.alp_gemm_f64(M, N, K, 1.0, call.A, K, call.B, N, 0.0, call.C, N)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            alp.alp_gemm_f64(M, N, K, 1.0, call.A, K, call.B, N, 0.0, call.C, N)
            e1.record()
            e1.synchronize()
            ts[tuned].append(e0.elapsed_time(e1))
    assert min(ts[True]) <= 1.03 * min(ts[False]) + 0.002, ts


@pytest.mark.parametrize("shape", [(3000, 4000, 142), (7961, 3610, 142), (633, 1840, 12151),
                                   (1531, 2351, 12150), (3367, 5475, 1913), (629, 937, 11136)])
def test_the_direct_estimate_of_capped_launches(alp, clean, monkeypatch, tmp_path, shape):
    """Few k per tile, and long k ranges shared by clusters: the database's figure
    within 4 % of the call (2 % that runs differ by, 2 for whole waves)."""
    import torch
    db = str(tmp_path / "db.jsonl")
    monkeypatch.setenv("ALP_TUNE_DB", db)
    M, N, K = shape
    alp.alp_tune(M, N, K, alp.ALP_PATH_NATIVE, alp.ALP_TUNE_EXHAUSTIVE)
    rec = tuning.load_db(db)[-1]
    alp.alp_tune_clear_cache()
    call = Calls(alp, M, N, K)
    ts = []
    for _ in range(4):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        alp.alp_gemm_f64(M, N, K, 1.0, call.A, K, call.B, N, 0.0, call.C, N)
        e1.record()
        e1.synchronize()
        ts.append(e0.elapsed_time(e1))
    assert abs(rec["direct"] / min(ts) - 1) < 0.04, (rec["direct"], ts)
