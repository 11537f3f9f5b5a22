"""Modular products of few tiles, cut into columns of 128 or 64 so that every
unit has a cluster: at the edges of those tiles and of the counts that choose
them, element for element as the stages give them (256-column tiles, products
and reconstruction in two calls)."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,n", [
    (1, 1, 1, 4), (256, 64, 64, 15), (256, 65, 1025, 15), (255, 128, 1024, 16),
    (257, 129, 300, 15), (250, 257, 65, 4), (512, 320, 130, 15),
    (200, 1216, 90, 4), (200, 1217, 90, 4), (700, 256, 2049, 8)])
@pytest.mark.parametrize("alpha,beta", [(1.0, 0.0), (-0.75, 0.5)])
def test_narrow_tiles_match_the_stages(alp, M, N, K, n, alpha, beta):
    import torch
    A, B, C = inputs.gemm_operands(7300 + M + N + K, M, N, K, kind="scaled", phi=3)
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
    crt = alp.ALP_SLICE_BF16_CRT
    ws = alp.alp_gemm_f64_emul_workspace(M, N, K, n, crt)
    work = torch.full((ws,), 255, dtype=torch.uint8, device="cuda")
    got = torch.from_numpy(C.copy()).cuda()
    alp.alp_gemm_f64_emul(M, N, K, alpha, dA, K, dB, N, beta, got, N, n, crt, work, ws)
    kpad, ldg = (K + 63) // 64 * 64, (N + 255) // 256 * 256
    de = torch.empty(M, dtype=torch.int32, device="cuda")
    df = torch.empty(N, dtype=torch.int32, device="cuda")
    alp.alp_emul_exponents(M, K, dA, K, 0, de)
    alp.alp_emul_exponents(N, K, dB, N, 1, df)
    da = torch.empty((n, M, kpad), dtype=torch.bfloat16, device="cuda")
    db = torch.empty((n, N, kpad), dtype=torch.bfloat16, device="cuda")
    alp.alp_emul_split(M, K, dA, K, 0, de, n, crt, da, kpad)
    alp.alp_emul_split(N, K, dB, N, 1, df, n, crt, db, kpad)
    G = torch.full((n, M, ldg), 255, dtype=torch.uint8, device="cuda")
    alp.alp_emul_slice_products(M, N, K, n, crt, da, db, kpad, G, ldg)
    want = torch.from_numpy(C.copy()).cuda()
    alp.alp_emul_recombine_crt(M, N, K, n, G, ldg, de, df, alpha, beta, want, N)
    torch.cuda.synchronize()
    assert alp.alp_get_device_error() == alp.ALP_OK
    assert np.array_equal(got.cpu().numpy(), want.cpu().numpy())
