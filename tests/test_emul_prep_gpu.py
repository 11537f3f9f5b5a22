"""The emulated GEMM calls, whose operands are prepared by one launch (lines
walked by warps or blocks, strided operands in strips shared by a cluster),
against the stages run one by one through the C-ABI (scan, split, products,
recombination): the same C bit for bit, at the sizes where lines, strips,
clusters and the cut of the fused launch change."""
import numpy as np
import pytest

from paper_1706_10086_gb300 import inputs

from .test_emul_crt_gpu import MODULI, check_residues, crt_k

pytestmark = pytest.mark.gpu


def stored(x, trans, pad, shift, dtype):
    """x (or x^T) on the device, `pad` NaN columns after each row and the base
    `shift` elements past a 16-byte boundary."""
    import torch
    a = torch.from_numpy(np.ascontiguousarray(x.T if trans else x)).cuda().to(dtype)
    r, c = a.shape
    buf = torch.full((shift + r * (c + pad),), float("nan"), dtype=dtype, device="cuda")
    view = buf[shift:].view(r, c + pad)
    view[:, :c] = a
    return view, c + pad


def by_stages(alp, f32, ta, tb, M, N, K, alpha, A, lda, B, ldb, beta, C, n, kind):
    import torch
    crt = kind == alp.ALP_SLICE_BF16_CRT
    kpad, ldg = (K + 63) // 64 * 64, (N + 255) // 256 * 256
    exps = alp.alp_emul_exponents_f32 if f32 else alp.alp_emul_exponents
    split = alp.alp_emul_split_f32 if f32 else alp.alp_emul_split
    e = torch.empty(M, dtype=torch.int32, device="cuda")
    f = torch.empty(N, dtype=torch.int32, device="cuda")
    da = torch.empty((n, M, kpad), dtype=torch.bfloat16, device="cuda")
    db = torch.empty((n, N, kpad), dtype=torch.bfloat16, device="cuda")
    exps(M, K, A, lda, ta, e)
    exps(N, K, B, ldb, 1 - tb, f)
    split(M, K, A, lda, ta, e, n, kind, da, kpad)
    split(N, K, B, ldb, 1 - tb, f, n, kind, db, kpad)
    G = torch.empty((n, M, ldg), dtype=torch.uint8 if crt else torch.int32, device="cuda")
    alp.alp_emul_slice_products(M, N, K, n, kind, da, db, kpad, G, ldg)
    if crt:
        alp.alp_emul_recombine_crt(M, N, K, n, G, ldg, e, f, alpha, beta, C, N)
    else:
        rec = alp.alp_emul_recombine_f32 if f32 else alp.alp_emul_recombine
        rec(M, N, n, kind, G, ldg, e, f, alpha, beta, C, N)


def check(alp, M, N, K, kind, n, f32=False, ta=0, tb=0, pad=0, shift=0, zero_lines=True):
    import torch
    dtype = torch.float32 if f32 else torch.float64
    A, B, C = inputs.gemm_operands(9000 + M + N + K + n, M, N, K, kind="scaled", phi=6)
    if zero_lines:
        A[M // 2] = 0.0
        B[:, N // 2] = 0.0
    dA, lda = stored(A, ta, pad, shift, dtype)
    dB, ldb = stored(B, tb, pad, shift, dtype)
    got = torch.from_numpy(C).cuda().to(dtype)
    want = got.clone()
    call = alp.alp_gemm_f32_emul_ex if f32 else alp.alp_gemm_f64_emul_ex
    size = alp.alp_gemm_f32_emul_workspace if f32 else alp.alp_gemm_f64_emul_workspace
    ws = size(M, N, K, n, kind)
    work = torch.full((ws,), 0x5A, dtype=torch.uint8, device="cuda")
    call(ta, tb, M, N, K, 1.5, dA, lda, dB, ldb, 0.5, got, N, n, kind, work, ws)
    by_stages(alp, f32, ta, tb, M, N, K, 1.5, dA, lda, dB, ldb, 0.5, want, n, kind)
    torch.cuda.synchronize()
    assert alp.alp_get_device_error() == alp.ALP_OK
    assert torch.equal(got, want)


@pytest.mark.parametrize("K", [1, 3, 63, 129, 1023, 1025, 2047, 2049, 8191, 8193])
@pytest.mark.parametrize("ta,tb,pad,shift", [(0, 0, 0, 0), (1, 1, 1, 1)])
def test_crt_lines_and_clusters(alp, K, ta, tb, pad, shift):
    """k ranges of one block, several, the longest cluster and past it; odd
    leading dimensions and bases off 16 bytes (no vector loads)."""
    check(alp, 37, 21, K, alp.ALP_SLICE_BF16_CRT, 15, ta=ta, tb=tb, pad=pad, shift=shift)


@pytest.mark.parametrize("kind,n", [("b7", 8), ("b7", 3), ("b8", 7), ("b8t", 5)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 1)])
def test_digits_prepared_as_by_stages(alp, kind, n, ta, tb):
    k = {"b7": alp.ALP_SLICE_BF16, "b8": alp.ALP_SLICE_BF16_B8, "b8t": alp.ALP_SLICE_BF16_B8_TRIM}
    check(alp, 131, 66, 1500, k[kind], n, ta=ta, tb=tb, pad=1)


@pytest.mark.parametrize("kind,n", [("b7", 4), ("b8", 2), ("b8", 3)])
@pytest.mark.parametrize("ta,tb,pad,shift", [(0, 0, 0, 0), (1, 1, 3, 1), (0, 1, 0, 2)])
def test_f32_prepared_as_by_stages(alp, kind, n, ta, tb, pad, shift):
    k = {"b7": alp.ALP_SLICE_BF16, "b8": alp.ALP_SLICE_BF16_B8}
    check(alp, 70, 133, 2100, k[kind], n, f32=True, ta=ta, tb=tb, pad=pad, shift=shift)


@pytest.mark.parametrize("M,N,K,n", [
    (2300, 64, 4000, 4),        # a strided operand past the strips' size, one within it
    (1280, 1280, 300, 15),      # fewer tiles than clusters: units shared by all of them
    (5120, 5120, 2600, 15),     # a whole wave joins the tail
    (5000, 2600, 3300, 14),     # reconstruction in the launch, hidden by the tail
    (4096, 5200, 700, 16)])     # short products: every tile reconstructed after the launch
def test_crt_launch_cuts(alp, M, N, K, n):
    check(alp, M, N, K, alp.ALP_SLICE_BF16_CRT, n, ta=1, zero_lines=False)


@pytest.mark.parametrize("n", [15, 16])
def test_crt_residues_of_wide_integers(alp, n):
    """k up to 60 (short K, many moduli): entries at both ends of the scaled
    range, next to 2^52 and 2^53, ties and tiny values; every residue is one of
    the exact integer RN(a 2^(k-e)) and at most 128."""
    from fractions import Fraction

    import torch
    for K in (4, 5000):
        k = crt_k(K, n)
        rng = np.random.default_rng(40 + n + K)
        X = rng.uniform(-1, 1, (6, K))
        X[0, :4] = [1.0 - 2.0 ** -53, -(1.0 - 2.0 ** -53), 0.5, -0.5]
        X[1, :4] = np.ldexp([1.0, 1.0 - 2.0 ** -53, -1.0, 1.0 + 2.0 ** -52], 52 - k)
        X[1, 3] = 0.75
        X[2, :4] = np.ldexp([3.0, -5.0, 2.0 ** 50 + 1, 2.0 ** 52 + 1], -k - 1)   # ties
        X[3, :4] = [2.0 ** -70, -2.0 ** -900, 0.0, 0.9]
        X[4] *= 2.0 ** 900
        X[5] *= 2.0 ** -900
        kpad = (K + 63) // 64 * 64
        dX = torch.from_numpy(X).cuda()
        e = torch.empty(6, dtype=torch.int32, device="cuda")
        out = torch.zeros((n, 6, kpad), dtype=torch.bfloat16, device="cuda")
        alp.alp_emul_exponents(6, K, dX, K, 0, e)
        alp.alp_emul_split(6, K, dX, K, 0, e, n, alp.ALP_SLICE_BF16_CRT, out, kpad)
        torch.cuda.synchronize()
        r = out.float().cpu().numpy().astype(np.int64)
        ex = e.cpu().numpy()
        for i in range(6):
            cols = np.arange(min(K, 400))
            ints = [round(Fraction(float(a)) * Fraction(2) ** (k - int(ex[i]))) for a in X[i, cols]]
            for l in range(n):
                check_residues(r[l, i, cols], np.array(ints, dtype=object), MODULI[l])
