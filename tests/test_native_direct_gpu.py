"""The native FP64 GEMM without a tile config (alp_gemm_f64 and
alp_gemm_f64_ex with cfg = NULL): whole 32 x 16 tiles, and 16 x 8 fragments
whose k range is shared by four warps of 1, 2, 4 or 8 blocks, at the sizes
where fragments, k-steps and parts are ragged or empty.  Integer operands and
power-of-two scalars: every partial sum is exact in any order, so the result
must equal the exact product bit for bit."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (16, 8, 4), (15, 7, 3), (17, 9, 5), (5, 300, 2), (64, 64, 64), (128, 128, 131),
          (33, 17, 1023),      # few fragments, a long k: a cluster of eight
          (200, 150, 1000),    # clusters of four
          (1000, 700, 70),     # splits among the warps alone
          (1500, 1501, 37)]    # whole tiles


def padded(x, pad, shift):
    """x on the device with `pad` NaN columns and a base `shift` doubles past a
    16-byte boundary; the buffer that holds it and its leading dimension."""
    import torch
    r, c = x.shape
    buf = torch.full((shift + r * (c + pad),), float("nan"), dtype=torch.float64, device="cuda")
    view = buf[shift:].view(r, c + pad)
    view[:, :c] = torch.from_numpy(np.ascontiguousarray(x))
    return buf, view, c + pad


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("ta,tb,pad,shift", [(0, 0, 0, 0), (0, 1, 1, 1), (1, 0, 2, 0), (1, 1, 3, 1)])
def test_direct_shapes_strides_and_transposes(alp, shape, ta, tb, pad, shift):
    import torch
    M, N, K = shape
    A, B, C = inputs.gemm_operands(8100 + M + N + K, M, N, K, kind="int")
    _, vA, lda = padded(A.T if ta else A, pad, shift)
    _, vB, ldb = padded(B.T if tb else B, pad, shift)
    _, vC, ldc = padded(C, pad, shift)
    ws = alp.alp_gemm_f64_ex_workspace(ta, tb, M, N, K)
    work = torch.empty(max(ws, 1), dtype=torch.uint8, device="cuda")
    alp.alp_tune_clear_cache()
    alp.alp_gemm_f64_ex(ta, tb, M, N, K, 2.0, vA, lda, vB, ldb, 0.5, vC, ldc, None,
                        work if ws else None, ws)
    torch.cuda.synchronize()
    assert alp.alp_get_device_error() == alp.ALP_OK
    full = vC.cpu().numpy()
    got = full[:, :N]
    assert np.isnan(full[:, N:]).all()
    assert np.array_equal(got, 2.0 * (A @ B) + 0.5 * C)
    # beta = 0 reads no C (NaN there)
    vC.fill_(float("nan"))
    alp.alp_gemm_f64_ex(ta, tb, M, N, K, -1.0, vA, lda, vB, ldb, 0.0, vC, ldc, None,
                        work if ws else None, ws)
    torch.cuda.synchronize()
    assert np.array_equal(vC.cpu().numpy()[:, :N], -(A @ B))


@pytest.mark.parametrize("shape", SHAPES)
def test_direct_transposes_give_the_same_bits(alp, shape):
    """Uniform operands: the order of the sums is fixed by the shape, so every
    storage of the same matrices gives the same bits."""
    import torch
    M, N, K = shape
    A, B, _ = inputs.gemm_operands(8200 + M + N + K, M, N, K, with_c=False)
    alp.alp_tune_clear_cache()
    got = []
    for ta in (0, 1):
        for tb in (0, 1):
            dA = torch.from_numpy(np.ascontiguousarray(A.T if ta else A)).cuda()
            dB = torch.from_numpy(np.ascontiguousarray(B.T if tb else B)).cuda()
            dC = torch.empty(M, N, dtype=torch.float64, device="cuda")
            ws = alp.alp_gemm_f64_ex_workspace(ta, tb, M, N, K)
            work = torch.empty(max(ws, 1), dtype=torch.uint8, device="cuda")
            alp.alp_gemm_f64_ex(ta, tb, M, N, K, 1.0, dA, dA.shape[1], dB, dB.shape[1], 0.0, dC, N,
                                None, work if ws else None, ws)
            torch.cuda.synchronize()
            got.append(dC.cpu().numpy())
    assert all(np.array_equal(got[0], g) for g in got[1:])
