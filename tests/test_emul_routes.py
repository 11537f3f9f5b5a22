"""Which launches an emulated GEMM call makes: its strided operands prepared in
strips together with the others, or by a scan and a split of their own; the sums
recombined by a kernel that starts while the products drain, or after them; the
tiles that the products share; the tiles and blocks of the splits.  A C program
stands in for the runtime and records the launches, so no GPU is needed; the GPU
tests compare the routes with the stages bit for bit."""
import subprocess

import pytest

from paper_1706_10086_gb300 import alp as lib

from .test_emul_prep_gpu import check

PROGRAM = r"""
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
static int word, launches, last_attrs;
static unsigned grids[16];   /* x, by launch */
static const void* last_kernel;
static dim3 last_grid, last_block;
cudaError_t cudaGetDevice(int* d) { *d = 0; return 0; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { *v = 152; return 0; }
cudaError_t cudaMalloc(void** p, size_t n) { *p = &word; return 0; }
cudaError_t cudaMemset(void* p, int v, size_t n) { return 0; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { return 0; }
cudaError_t cudaMemcpyAsync(void* d, const void* x, size_t n, enum cudaMemcpyKind k,
                            cudaStream_t s) {
    if (k == cudaMemcpyDeviceToHost) memset(d, 0, n);   /* no statistics: fewest moduli */
    return 0;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return 0; }
cudaError_t cudaDeviceSynchronize(void) { return 0; }
cudaError_t cudaGetLastError(void) { return 0; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) { return 0; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    *n = 76;
    return 0;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
    grids[launches++ % 16] = g.x;
    last_attrs = 0;
    last_kernel = f;
    last_grid = g;
    last_block = b;
    return 0;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
    *k = (cudaKernel_t)f;
    return 0;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t f, dim3 g, dim3 b, void** a, size_t m, cudaStream_t s) {
    return cudaLaunchKernel((const void*)f, g, b, a, m, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** a) {
    grids[launches++ % 16] = c->gridDim.x;
    last_attrs = (int)c->numAttrs;
    return 0;
}
static int encode() { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** fn, unsigned v,
                                             unsigned long long flags,
                                             enum cudaDriverEntryPointQueryResult* r) {
    *fn = (void*)encode;
    *r = cudaDriverEntryPointSuccess;
    return 0;
}

typedef int (*gemm64)(int, int, int64_t, int64_t, int64_t, double, const void*, int64_t,
                      const void*, int64_t, double, void*, int64_t, int, int, void*, size_t, void*);
typedef int (*gemm32)(int, int, int64_t, int64_t, int64_t, float, const void*, int64_t,
                      const void*, int64_t, float, void*, int64_t, int, int, void*, size_t, void*);

typedef int (*split)(int64_t, int64_t, const void*, int64_t, int, const void*, int, int, void*,
                     int64_t, void*);

int main(int argc, char** argv) {
    void* so = dlopen(argv[1], RTLD_NOW);
    if (!so) return fprintf(stderr, "%s\n", dlerror()), 2;
    gemm64 f64 = (gemm64)dlsym(so, "alp_gemm_f64_emul_ex");
    gemm32 f32 = (gemm32)dlsym(so, "alp_gemm_f32_emul_ex");
    char* p = (char*)0x10000000;   /* never read: nothing is launched */
    int64_t M, N, K;
    int is32, kind, n;
    if (argc > 2) {   /* the split of R lines of K: which kernel, its grid and block */
        split s64 = (split)dlsym(so, "alp_emul_split"), s32 = (split)dlsym(so, "alp_emul_split_f32");
        int trans, shift;
        while (scanf("%d %d %d %ld %ld %d %d", &is32, &kind, &n, &M, &K, &trans, &shift) == 7) {
            const int rc = (is32 ? s32 : s64)(M, K, p, trans ? M : K, trans, p, n, kind, p + shift,
                                              (K + 63) / 64 * 64, 0);
            printf("%d %ld %u %u %u\n", rc, (long)last_kernel, last_grid.x, last_grid.y,
                   last_block.x);
        }
        return 0;
    }
    while (scanf("%d %d %d %ld %ld %ld", &is32, &kind, &n, &M, &N, &K) == 6) {
        launches = 0;
        const int rc =
            is32 ? f32(0, 0, M, N, K, 1, p, K, p, N, 0, p, N, n, kind, p, (size_t)1 << 60, 0)
                 : f64(0, 0, M, N, K, 1, p, K, p, N, 0, p, N, n, kind, p, (size_t)1 << 60, 0);
        printf("%d %d %d %u\n", rc, launches, last_attrs, grids[(launches - 2) % 16]);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def recorded(alp, tmp_path_factory):
    d = tmp_path_factory.mktemp("routes")
    src, exe = d / "routes.c", d / "routes"
    src.write_text(PROGRAM)
    subprocess.run(["gcc", "-O1", "-w", "-rdynamic", "-I/usr/local/cuda/include", "-o", str(exe),
                    str(src), "-ldl"], check=True)

    def run(calls, *args):
        text = "\n".join(" ".join(str(int(v)) for v in c) for c in calls)
        r = subprocess.run([str(exe), alp.LIB_PATH, *args], input=text, capture_output=True,
                           text=True, timeout=120)
        assert r.returncode == 0, r.stderr
        rows = [[int(v) for v in l.split()] for l in r.stdout.splitlines()]
        assert len(rows) == len(calls) and all(row[0] == 0 for row in rows)
        return [row[1:] for row in rows]
    return run


@pytest.fixture(scope="module")
def routes(recorded):
    """calls -> (launches, whether the last one may start early) of each."""
    return lambda calls: [(n, attrs > 0) for n, attrs, _ in recorded(calls)]


B7, B8, CRT = lib.ALP_SLICE_BF16, lib.ALP_SLICE_BF16_B8, lib.ALP_SLICE_BF16_CRT
# (float, kind, slices, M, N, K): whether B is prepared in strips
STRIPS = {
    (0, B7, 8, 64, 64, 64): True, (0, CRT, 15, 64, 16384, 64): True,
    (0, B7, 8, 64, 24576, 128): True, (0, B7, 8, 64, 24577, 128): False,
    (0, CRT, 15, 64, 24576, 64): True, (0, CRT, 15, 64, 24580, 1): False,
    (0, B7, 8, 64, 131072, 64): False, (0, CRT, 15, 64, 131072, 16): False,
    (0, B7, 8, 64, 32768, 129): True, (0, B7, 8, 64, 32769, 129): False,
    (0, B7, 8, 64, 32768, 256): True, (0, CRT, 15, 64, 1024, 8192): True,
    (0, CRT, 15, 64, 1024, 8193): False, (0, CRT, 15, 64, 4097, 2048): False,
    (1, B8, 3, 64, 49152, 128): True, (1, B8, 3, 64, 49153, 128): False,
    (1, B8, 3, 64, 262144, 64): False, (1, B8, 3, 64, 131072, 129): True,
    (1, B8, 3, 64, 131072, 256): True, (1, B8, 3, 64, 131073, 256): False}


def test_strips_or_separate(routes):
    """In strips: one preparation launch, then products and sums.  Separate:
    the scan's two or three launches and the split before the other operand's."""
    got = routes(STRIPS)
    assert {c: n == 3 for c, (n, _) in zip(STRIPS, got)} == STRIPS
    assert all(n in (3, 6) for n, _ in got), got


# the automatic count (float, kind, 0, M, N, K): whether B's statistics come in strips
AUTO = {
    (0, CRT, 0, 64, 256, 256): True, (0, CRT, 0, 64, 700, 8190): True,
    (0, CRT, 0, 64, 768, 8192): True, (0, CRT, 0, 64, 769, 8192): False,
    (0, CRT, 0, 64, 1024, 8192): False, (0, CRT, 0, 64, 2048, 4096): True,
    (0, CRT, 0, 64, 1535, 4097): True, (0, CRT, 0, 64, 1536, 4097): False,
    (0, CRT, 0, 64, 24576, 64): True, (0, CRT, 0, 64, 24577, 64): False}


def test_statistics_in_strips_or_separate(routes):
    """In strips: statistics, preparation, products, reconstruction."""
    got = routes(AUTO)
    assert {c: n == 4 for c, (n, _) in zip(AUTO, got)} == AUTO
    assert all(n == 4 or n >= 8 for n, _ in got), got


# whether the kernel that makes C of the sums starts while the products drain
EARLY = {
    (0, B7, 8, 256, 256, 256): True, (0, B7, 8, 1280, 2048, 64): True,
    (0, B7, 8, 1281, 2048, 64): False, (0, B7, 8, 1281, 2048, 2048): False,
    (0, B7, 4, 2048, 2048, 64): True, (0, B7, 8, 8192, 8192, 64): False,
    (1, B8, 3, 724, 724, 64): True, (1, B8, 3, 2048, 2048, 64): True,
    (1, B8, 3, 4096, 4096, 64): False, (1, B8, 2, 3072, 3072, 64): True,
    (1, B8, 3, 8192, 8192, 256): False, (0, CRT, 15, 4096, 4096, 64): True}


def test_recombination_early_or_after(routes):
    got = routes(EARLY)
    assert {c: early for c, (_, early) in zip(EARLY, got)} == EARLY


# whether the tiles of the last wave are shared by all 76 CTA pairs of the products
# (digit schemes; tiles of 256 x 256): not where the pair that gets most of them
# would get a whole tile's products
SHARED = {
    (1, B8, 3, 2048, 2048, 512): False, (1, B8, 3, 60 * 256, 256, 512): True,
    (1, B8, 3, 61 * 256, 256, 512): False, (1, B8, 2, 50 * 256, 256, 64): True,
    (1, B8, 2, 51 * 256, 256, 64): False, (0, B7, 4, 65 * 256, 256, 64): True,
    (0, B7, 4, 66 * 256, 256, 64): False, (0, B7, 8, 2048, 2048, 64): True,
    (0, B7, 8, 68 * 256, 256, 64): True, (0, B7, 8, 69 * 256, 256, 64): False,
    (0, lib.ALP_SLICE_BF16_B8_TRIM, 4, 66 * 256, 256, 64): False,
    (0, lib.ALP_SLICE_BF16_B8_TRIM, 7, 64 * 256, 256, 64): True, (1, B8, 3, 256, 256, 64): True}


def largest_share(tiles, s, trim, pairs):
    """The units (groups of `tiles` tiles) in descending order of their products,
    dealt out to the pairs in turns of alternating direction."""
    groups = [s - r for r in range(s)] if not trim else list(range(s - 1, 0, -1)) + [2]
    units = [g for g in sorted(groups, reverse=True) for _ in range(tiles)]
    shares = [0] * min(pairs, len(units))
    for i in range(0, len(units), len(shares)):
        turn = units[i:i + len(shares)]
        order = range(len(shares)) if i // len(shares) % 2 == 0 else reversed(range(len(shares)))
        for c, u in zip(order, turn + [0] * (len(shares) - len(turn))):
            shares[c] += u
    return max(shares), sum(groups)


def test_shared_tiles_pay(recorded):
    got = recorded(SHARED)
    for call, (_, _, grid) in zip(SHARED, got):
        _, kind, s, M, N, _ = call
        tiles = M // 256 * (N // 256)
        most, whole = largest_share(tiles, s, kind == lib.ALP_SLICE_BF16_B8_TRIM, 76)
        assert SHARED[call] == (10 * tiles <= 9 * 76 and most < whole), call
        assert grid == 2 * (min(76, tiles * s) if SHARED[call] else tiles), call


# (float, kind, slices, lines, K): whether the columns are split by 128-k tiles
BY_128 = {
    (0, B7, 8, 65536, 64): False, (0, B7, 8, 65536, 65): True, (0, B7, 8, 65536, 128): True,
    (0, B7, 8, 65536, 129): False, (0, B7, 4, 65536, 192): False, (0, B7, 4, 32768, 448): False,
    (0, B8, 7, 4096, 960): False, (0, B8, 7, 4096, 1088): True, (0, B7, 8, 8192, 8192): True,
    (0, B7, 8, 512, 512): False, (0, B7, 8, 19424, 128): False, (0, B7, 8, 19425, 128): True,
    (1, B8, 3, 262144, 64): False, (1, B8, 3, 65536, 128): True, (0, CRT, 15, 65536, 64): False,
    (0, CRT, 15, 4096, 4096): True}


def test_column_split_tiles(recorded):
    """Told apart by the kernel: output off 8 bytes always takes the 64-k tiles."""
    both = recorded([c + (1, shift) for shift in (0, 4) for c in BY_128], "split")
    got, by_64 = both[:len(BY_128)], both[len(BY_128):]
    assert {c: g[0] != h[0] for c, g, h in zip(BY_128, got, by_64)} == BY_128
    for (_, _, _, R, K), g, h in zip(BY_128, got, by_64):
        kpad = (K + 63) // 64 * 64
        assert h[1:] == [(R + 31) // 32, kpad // 64, 256]
        assert g == h or g[1:] == [(R + 31) // 32, (kpad + 127) // 128, 256]


def test_row_split_blocks(recorded):
    """Digit rows: no more threads than a row of four k each needs, and as many
    on an SM as with the widest blocks."""
    calls = [(f, k, n, R, K) for f, k, n in ((0, B7, 4), (0, B8, 7), (1, B8, 3))
             for R in (5, 1000, 262144) for K in (1, 64, 128, 129, 256, 300, 512, 513, 1024, 4097)]
    for (_, _, _, R, K), (_, gx, gy, threads) in zip(
            calls, recorded([c + (0, 0) for c in calls], "split")):
        kpad = (K + 63) // 64 * 64
        assert threads == (32 if kpad <= 128 else 64 if kpad <= 256 else 128 if kpad <= 512 else 256)
        assert gx == (kpad + 1023) // 1024 and gx * threads * 4 >= min(kpad, 1024)
        assert gy == min(R, 152 * (2048 // threads) // gx)


def test_residue_row_blocks(recorded):
    """16 blocks per SM, 64 where each would walk four rows or more."""
    shapes = [(8192, 8192), (4096, 4096), (2048, 2048), (16384, 8192), (9728, 512), (9727, 512),
              (262144, 64), (5, 64), (1, 60000)]
    for (R, K), (_, gx, gy, threads) in zip(
            shapes, recorded([(0, CRT, 15, R, K, 0, 0) for R, K in shapes], "split")):
        by = 152 * 16 // gx
        assert threads == 128 and gx == ((K + 63) // 64 * 64 + 511) // 512
        assert gy == min(max(by * (4 if R >= 4 * by else 1), 1), R)


@pytest.mark.gpu
@pytest.mark.parametrize("call", [(0, B7, 8, 3, 24576, 70), (0, B7, 8, 3, 24577, 70),
                                  (0, CRT, 15, 5, 24579, 33), (0, B7, 3, 2, 32769, 130),
                                  (1, B8, 3, 3, 49152, 70), (1, B8, 3, 3, 49157, 70)])
@pytest.mark.parametrize("ta,pad,shift", [(0, 0, 0), (1, 1, 1)])
def test_routes_agree_with_the_stages(alp, call, ta, pad, shift):
    """Both sides of each line; with ta the long operand is A, stored K x M."""
    f32, kind, n, M, N, K = call
    if ta:
        M, N = N, M
    check(alp, M, N, K, kind, n, f32=bool(f32), ta=ta, pad=pad, shift=shift)


@pytest.mark.gpu
@pytest.mark.parametrize("M,N,K", [(70, 768, 8192), (70, 769, 8192), (800, 90, 8000),
                                   (10, 24577, 40)])
@pytest.mark.parametrize("ta,tb", [(0, 0), (1, 0), (1, 1)])
def test_automatic_count_is_the_given_count(alp, M, N, K, ta, tb):
    """The count and C of nslices = 0, on either route, against the same call
    with that count given."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(M + N + K)
    rand = lambda r, c: torch.rand((r, c), dtype=torch.float64, device="cuda", generator=g) - 0.5
    A = rand(K, M) if ta else rand(M, K)
    B = rand(N, K) if tb else rand(K, N)
    ws = alp.alp_gemm_f64_emul_workspace(M, N, K, 0, CRT)
    work = torch.empty(ws, dtype=torch.uint8, device="cuda")
    n, _ = alp.alp_emul_crt_choose(ta, tb, M, N, K, A, A.shape[1], B, B.shape[1], work, ws)
    out = []
    for count in (0, n):
        C = torch.full((M, N), float("nan"), dtype=torch.float64, device="cuda")
        alp.alp_gemm_f64_emul_ex(ta, tb, M, N, K, 1.0, A, A.shape[1], B, B.shape[1], 0.0, C, N,
                                 count, CRT, work, ws)
        out.append(C)
    torch.cuda.synchronize()
    assert alp.alp_get_device_error() == alp.ALP_OK
    assert torch.equal(out[0], out[1]) and n >= 4


@pytest.mark.gpu
@pytest.mark.parametrize("call", [(0, B7, 8, 1280, 2048, 40), (0, B7, 8, 1281, 2047, 40),
                                  (1, B8, 3, 3300, 2048, 100), (0, B7, 3, 3000, 2600, 33)])
def test_sums_agree_with_the_stages(alp, call):
    f32, kind, n, M, N, K = call
    check(alp, M, N, K, kind, n, f32=bool(f32))


@pytest.mark.gpu
@pytest.mark.parametrize("f32,kind,n", [(0, B7, 4), (0, B7, 8), (0, CRT, 15), (1, B8, 3)])
@pytest.mark.parametrize("R,K", [(19425, 65), (19424, 128), (20001, 129), (700, 1088), (700, 301),
                                 (3, 64), (33, 1), (2500, 513)])
@pytest.mark.parametrize("trans", [0, 1])
def test_split_agrees_with_the_general_kernels(alp, f32, kind, n, R, K, trans):
    """Output 8-byte aligned, and off it, where the kernels of two k per thread
    and 64-k tiles run."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(R + K)
    X = torch.rand((K, R) if trans else (R, K), dtype=torch.float32 if f32 else torch.float64,
                   device="cuda", generator=g) - 0.5
    kpad = (K + 63) // 64 * 64
    e = torch.empty(R, dtype=torch.int32, device="cuda")
    exps = alp.alp_emul_exponents_f32 if f32 else alp.alp_emul_exponents
    split = alp.alp_emul_split_f32 if f32 else alp.alp_emul_split
    exps(R, K, X, X.shape[1], trans, e)
    bufs = [torch.full((n * R * kpad + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
            for _ in range(2)]
    for buf, shift in zip(bufs, (0, 2)):
        split(R, K, X, X.shape[1], trans, e, n, kind, buf[shift:], kpad)
    torch.cuda.synchronize()
    assert alp.alp_get_device_error() == alp.ALP_OK
    size = n * R * kpad
    assert torch.equal(bufs[0][:size], bufs[1][2:2 + size])
    assert (bufs[0][size:] == 7.0).all() and (bufs[1][size + 2:] == 7.0).all()
    assert (bufs[1][:2] == 7.0).all()
