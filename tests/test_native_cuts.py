"""Every cut of the register-direct native kernels (alp_native_cut) at ragged
sizes, odd leading dimensions and transposed operands.  The shapes are chosen
for 152 SMs, which is asserted without a GPU."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs

# shape -> its cut on 152 SMs
CUTS = {(700, 701, 699): 2,      # clusters of two blocks
        (249, 255, 515): 2,
        (1021, 771, 1333): 1,    # the warps of a block alone, 41 waves
        (509, 517, 515): 1,
        (201, 149, 997): 4,
        (31, 19, 1021): 8,
        (1000, 700, 70): 0,      # whole tiles
        (333, 401, 271): 0}


def test_cuts_at_152_sms(alp):
    assert {s: alp.alp_native_cut(*s, 152) for s in CUTS} == CUTS
    assert alp.alp_native_cut(512, 512, 512, 152) == 2
    assert alp.alp_native_cut(2048, 2048, 2048, 152) == 0
    for bad in ((0, 1, 1, 152), (1, -1, 1, 152), (1, 1, 0, 152), (1, 1, 1, 0)):
        assert alp.alp_native_cut(*bad) == -1


@pytest.mark.gpu
@pytest.mark.parametrize("shape", sorted(CUTS))
@pytest.mark.parametrize("ta,tb,pad,shift", [(0, 0, 1, 1), (1, 0, 3, 0), (0, 1, 0, 1), (1, 1, 1, 0)])
def test_cut_is_exact_on_integers(alp, shape, ta, tb, pad, shift):
    """Integer operands and power-of-two scalars: every partial sum is exact in
    any order, so the result must equal the exact product bit for bit; the
    NaN padding of every buffer must stay and must not be read."""
    import torch
    M, N, K = shape

    def device(x):
        r, c = x.shape
        buf = torch.full((shift + r * (c + pad),), float("nan"), dtype=torch.float64,
                         device="cuda")
        view = buf[shift:].view(r, c + pad)
        view[:, :c] = torch.from_numpy(np.ascontiguousarray(x))
        return view

    A, B, C = inputs.gemm_operands(8400 + M + N + K, M, N, K, kind="int")
    dA, dB, dC = device(A.T if ta else A), device(B.T if tb else B), device(C)
    ws = alp.alp_gemm_f64_ex_workspace(ta, tb, M, N, K)
    work = torch.empty(max(ws, 1), dtype=torch.uint8, device="cuda")
    alp.alp_tune_clear_cache()
    alp.alp_gemm_f64_ex(ta, tb, M, N, K, 2.0, dA, dA.shape[1], dB, dB.shape[1], 0.5, dC,
                        dC.shape[1], None, work if ws else None, ws)
    full = dC.cpu().numpy()
    assert alp.alp_get_device_error() == alp.ALP_OK
    assert np.isnan(full[:, N:]).all()
    assert np.array_equal(full[:, :N], 2.0 * (A @ B) + 0.5 * C)
