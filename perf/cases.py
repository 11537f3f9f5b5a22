"""The GEMM library's work as a user's program has it do: its public calls at
the sizes of this repository's own workloads, from calls of a few microseconds
to the 8192-cubed product, timed one pass at a time.

A case names a family and its sizes:

* ``native``   alp_gemm_f64 (or alp_gemm_f64_ex when an operand is transposed),
  the config left to the library;
* ``emul``     alp_gemm_f64_emul (alp_gemm_f64_emul_ex): the modular scheme with
  a given or automatic count of moduli, or a digit scheme;
* ``f32``      alp_gemm_f32_emul (alp_gemm_f32_emul_ex);
* ``batched``  alp_gemm_batched_varsize, called directly or replayed as a graph;
* ``mlp``      one training step of the tile-config cost model: forward,
  backward and Adam.

Inputs are synthetic, made on the GPU from the seed: entries uniform in
[-1, 1), times 2^e with e a uniform integer in [-phi, phi] where phi > 0.
"""
import math

import numpy as np
import torch

from paper_1706_10086_gb300 import alp, inputs, tuning

KINDS = {"crt": alp.ALP_SLICE_BF16_CRT, "b7": alp.ALP_SLICE_BF16, "b8": alp.ALP_SLICE_BF16_B8,
         "b8trim": alp.ALP_SLICE_BF16_B8_TRIM}


def _gemm(name, path, M, N, K, alpha=1.0, beta=0.0, ta=0, tb=0, phi=0, kind="", slices=0):
    return {"name": name, "path": path, "M": M, "N": N, "K": K, "alpha": alpha, "beta": beta,
            "trans_a": ta, "trans_b": tb, "phi": phi, "kind": kind, "slices": slices}


def listed():
    return [
        # a small block of a larger algorithm (a panel update, a reduced basis): the
        # smallest shapes of the predictor's range, where the call itself counts
        _gemm("native 64", "native", 64, 64, 64),
        # the plain DGEMM of 512, alpha = 1, beta = 0
        _gemm("native 512", "native", 512, 512, 512),
        # a member of the native size scan: alpha = 1.5, beta = 0.5, C updated in place
        _gemm("native 2048", "native", 2048, 2048, 2048, 1.5, 0.5),
        # odd sizes and leading dimensions with a transposed operand: a normal-equations
        # product on data whose rows are not 16-byte multiples
        _gemm("native ragged", "native", 1021, 771, 1333, 1.5, 0.5, ta=1),
        # the emulated product on small matrices, where its stages are launches
        _gemm("emul 256", "emul", 256, 256, 256, kind="crt", slices=15),
        # the automatic count of moduli on entries of spread exponents: the call a user
        # makes who does not know the data
        _gemm("emul auto 1024", "emul", 1024, 1024, 1024, phi=8, kind="crt", slices=0),
        # a rectangular product with ragged sides, B stored transposed, alpha and beta
        _gemm("emul ragged", "emul", 3000, 1500, 2100, 0.75, -0.5, tb=1, phi=32, kind="crt",
              slices=16),
        # the headline: 8192 cubed with 15 moduli
        _gemm("emul 8192", "emul", 8192, 8192, 8192, kind="crt", slices=15),
        # a digit scheme at the count that is accurate for spread exponents
        _gemm("digits 2048", "emul", 2048, 2048, 2048, phi=8, kind="b7", slices=8),
        # the emulated FP32 product with three 8-bit slices
        _gemm("f32 4096", "f32", 4096, 4096, 4096, kind="b8", slices=3),
        # thousands of uneven problems in one graph launch
        {"name": "batched 4096", "path": "batched", "count": 4096, "lo": 16, "hi": 1024,
         "sizes": inputs.workload_seed("batched_4096"), "alpha": 1.5, "beta": 0.5, "graph": True},
        # one epoch of the cost model: 2000 shapes on both paths, all configs
        {"name": "mlp epoch", "path": "mlp", "batch": 4000, "outputs": 78},
    ]


def draw(rng):
    """Another case of the same families: sizes log-uniform, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def shape(lo, hi, most):
        while True:
            M, N, K = size(lo, hi), size(lo, hi), size(lo, hi)
            if 2.0 * M * N * K <= most:
                return M, N, K

    path = rng.choice(["native", "native", "emul", "emul", "f32", "batched", "mlp"])
    if path == "batched":
        return {"path": path, "count": size(60, 4096), "lo": 16, "hi": size(200, 1024),
                "sizes": rng.randrange(1 << 30), "alpha": 1.5, "beta": rng.choice([0.0, 0.5]),
                "graph": rng.random() < 0.5}
    if path == "mlp":
        return {"path": path, "batch": size(100, 4000), "outputs": 78}
    scalars = rng.choice([(1.0, 0.0), (1.5, 0.5), (-1.0, 1.0)])
    ta, tb = rng.choice([(0, 0), (0, 0), (1, 0), (0, 1), (1, 1)])
    if path == "native":
        M, N, K = shape(64, 4096, 5e10)
        c = _gemm("", path, M, N, K, *scalars, ta, tb)
    elif path == "f32":
        M, N, K = shape(128, 8192, 5e11)
        c = _gemm("", path, M, N, K, *scalars, ta, tb, phi=rng.choice([0, 4]), kind="b8",
                  slices=rng.choice([2, 3, 3, 4]))
    else:
        M, N, K = shape(128, 8192, 5e11)
        kind, slices, phi = rng.choice([("crt", 0, 0), ("crt", 14, 0), ("crt", 15, 0),
                                        ("crt", 15, 8), ("crt", 16, 32), ("crt", 0, 32),
                                        ("b8trim", 7, 0), ("b7", 8, 8)])
        c = _gemm("", path, M, N, K, *scalars, ta, tb, phi=phi, kind=kind, slices=slices)
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1706 + seed)
    return g


def _entries(g, shape, phi=0, dtype=torch.float64):
    x = torch.rand(shape, dtype=dtype, device="cuda", generator=g).mul_(2).sub_(1)
    if phi:
        e = torch.randint(-phi, phi + 1, shape, device="cuda", generator=g)
        x = torch.ldexp(x, e.to(dtype))
    return x


def _gemm_inputs(case, seed):
    g = _generator(seed)
    dtype = torch.float32 if case["path"] == "f32" else torch.float64
    M, N, K = case["M"], case["N"], case["K"]
    A = _entries(g, (K, M) if case["trans_a"] else (M, K), case["phi"], dtype)
    B = _entries(g, (N, K) if case["trans_b"] else (K, N), case["phi"], dtype)
    C = _entries(g, (M, N), 0, dtype)
    return A, B, C


def _batched_sizes(case):
    return inputs.shapes(case["sizes"], case["count"], case["lo"], case["hi"])


def _batched_inputs(case, seed):
    """All A, all B and all C of the batch, each in one buffer, row-major and
    tight, with the offset of each problem's matrix (in elements)."""
    s = _batched_sizes(case)
    g = _generator(seed)
    pools, offsets = [], []
    for x, y in ((0, 2), (2, 1), (0, 1)):
        n = s[:, x] * s[:, y]
        pools.append(_entries(g, (int(n.sum()),)))
        offsets.append(np.concatenate([[0], np.cumsum(n)[:-1]]).astype(np.int64))
    return s, pools, offsets


def _mlp_inputs(case, seed):
    """A training set of the predictor's shape (sizes log-uniform in [64, 16384],
    targets ln(t / t_best) >= 0, a few configs that could not run) and parameters
    as the trainer starts them."""
    B, C = case["batch"], case["outputs"]
    g = _generator(seed)
    lg = torch.rand((B, 3), device="cuda", generator=g).mul_(8).add_(6)
    sizes = torch.exp2(lg).round().to(torch.int64)
    flag = torch.randint(0, 2, (B,), device="cuda", generator=g, dtype=torch.int32)
    T = torch.rand((B, C), device="cuda", generator=g).mul_(3)
    mask = (torch.rand((B, C), device="cuda", generator=g) < 0.5).float()
    params = torch.from_numpy(tuning.init_params(C, 1706 + seed)).cuda()
    return sizes, flag, T, mask, params


class _Graph:
    """A captured batched call, given back with the state that holds it."""

    def __init__(self, args, work, ws):
        self.handle = alp.alp_batched_graph_create(*args, work, ws)

    def __del__(self):
        alp.alp_batched_graph_destroy(self.handle)


def prepare(case, seed):
    st = {"case": case}
    path = case["path"]
    if path == "batched":
        s, (A, B, C), offs = _batched_inputs(case, seed)
        hM, hN, hK = (np.ascontiguousarray(s[:, i]) for i in range(3))
        n = len(s)

        def dev(a, dtype=torch.int64):
            return torch.tensor(a, dtype=dtype, device="cuda")

        ptr = [dev(p.data_ptr() + 8 * o) for p, o in zip((A, B, C), offs)]
        dM, dN, dK = dev(hM), dev(hN), dev(hK)
        args = (n, dM, dN, dK, dev(np.full(n, case["alpha"]), torch.float64), ptr[0], dK, ptr[1],
                dN, dev(np.full(n, case["beta"]), torch.float64), ptr[2], dN, hM, hN, hK)
        ws = alp.alp_gemm_batched_workspace(n, hM, hN, hK)
        work = torch.empty(ws, dtype=torch.uint8, device="cuda")
        st.update(A=A, B=B, C=C, args=args, work=work, ws=ws,
                  graph=_Graph(args, work, ws) if case["graph"] else None)
        return st
    if path == "mlp":
        sizes, flag, T, mask, params = _mlp_inputs(case, seed)
        B, C = case["batch"], case["outputs"]
        f32 = {"dtype": torch.float32, "device": "cuda"}
        M, N, K = (sizes[:, i].contiguous() for i in range(3))
        raw, X = torch.empty(B, 7, **f32), torch.empty(B, 7, **f32)
        mean, std = torch.empty(7, **f32), torch.empty(7, **f32)
        alp.alp_mlp_features(B, M, N, K, flag, None, None, raw)
        alp.alp_mlp_feature_stats(B, raw, mean, std)
        alp.alp_mlp_features(B, M, N, K, flag, mean, std, X)
        st.update(X=X, T=T, mask=mask, params=params, grads=torch.zeros_like(params),
                  m=torch.zeros_like(params), v=torch.zeros_like(params),
                  Y=torch.empty(B, C, **f32), cache=torch.empty(B, 128, **f32),
                  work=torch.empty(B * (C + 128), **f32), loss=torch.zeros(2, **f32), step=0)
        return st
    A, B, C = _gemm_inputs(case, seed)
    M, N, K, ta, tb = (case[k] for k in ("M", "N", "K", "trans_a", "trans_b"))
    if path == "native":
        ws = alp.alp_gemm_f64_ex_workspace(ta, tb, M, N, K)
    elif path == "emul":
        ws = alp.alp_gemm_f64_emul_workspace(M, N, K, case["slices"], KINDS[case["kind"]])
    else:
        ws = alp.alp_gemm_f32_emul_workspace(M, N, K, case["slices"], KINDS[case["kind"]])
    st.update(A=A, B=B, C=C, ws=ws, lda=A.shape[1], ldb=B.shape[1], ldc=N,
              work=torch.empty(ws, dtype=torch.uint8, device="cuda") if ws else None)
    return st


def run(st):
    c = st["case"]
    path = c["path"]
    if path == "batched":
        if st["graph"] is not None:
            alp.alp_batched_graph_launch(st["graph"].handle)
        else:
            alp.alp_gemm_batched_varsize(*st["args"], st["work"], st["ws"])
        return st["C"]
    if path == "mlp":
        B, C = c["batch"], c["outputs"]
        alp.alp_mlp_forward(st["params"], C, st["X"], B, st["Y"], st["cache"])
        alp.alp_mlp_backward(st["params"], C, st["X"], B, st["cache"], st["Y"], st["T"],
                             st["mask"], st["grads"], st["work"], st["loss"])
        st["step"] += 1
        alp.alp_mlp_adam(st["params"], st["grads"], st["m"], st["v"], st["params"].numel(),
                         st["step"], 3e-3)
        return [st[k] for k in ("Y", "cache", "loss", "grads", "params", "m", "v")]
    M, N, K, ta, tb, al, be = (c[k] for k in ("M", "N", "K", "trans_a", "trans_b", "alpha", "beta"))
    A, B, C, lda, ldb, ldc = (st[k] for k in ("A", "B", "C", "lda", "ldb", "ldc"))
    plain = not ta and not tb
    if path == "native":
        if plain:
            alp.alp_gemm_f64(M, N, K, al, A, lda, B, ldb, be, C, ldc)
        else:
            alp.alp_gemm_f64_ex(ta, tb, M, N, K, al, A, lda, B, ldb, be, C, ldc, None, st["work"],
                                st["ws"])
        return C
    call = {("emul", True): alp.alp_gemm_f64_emul, ("emul", False): alp.alp_gemm_f64_emul_ex,
            ("f32", True): alp.alp_gemm_f32_emul, ("f32", False): alp.alp_gemm_f32_emul_ex}
    lead = () if plain else (ta, tb)
    call[path, plain](*lead, M, N, K, al, A, lda, B, ldb, be, C, ldc, c["slices"],
                      KINDS[c["kind"]], st["work"], st["ws"])
    return C


def _products(case):
    """Tensor-core products of one emulated call (an automatic count as 15)."""
    s = case["slices"]
    if case["kind"] == "crt":
        return s or 15
    return s * (s - 1) // 2 + 2 if case["kind"] == "b8trim" else s * (s + 1) // 2


def work(case):
    path = case["path"]
    if path == "batched":
        M, N, K = (_batched_sizes(case)[:, i].astype(np.float64) for i in range(3))
        c = 2 if case["beta"] else 1
        return {"bytes": float(8 * (M * K + K * N + c * M * N).sum()),
                "flops": float(2 * (M * N * K).sum())}
    if path == "mlp":
        B, C = case["batch"], case["outputs"]
        p = alp.alp_mlp_param_count(C)
        # inputs, targets and mask read, outputs and pre-activations written; parameters
        # and both moments read and written, gradients written
        return {"bytes": 4 * (B * (7 + 2 * C + C + 128) + 7 * p), "flops": 6.0 * B * p}
    M, N, K = case["M"], case["N"], case["K"]
    e = 4 if path == "f32" else 8
    n = 1 if path == "native" else _products(case)
    return {"bytes": e * (M * K + K * N + M * N * (2 if case["beta"] else 1)),
            "flops": 2.0 * M * N * K * n}


# ---- what run() returns, in 64 bits ---------------------------------------------

def _product(A, B):
    """A B with an error far below one rounding of its terms: the leading bits
    of each row of A and column of B multiply exactly, the rest adds little."""
    K = A.shape[1]
    s = (52 - math.ceil(math.log2(max(K, 2)))) // 2

    def head(X, dim):
        top = X.abs().amax(dim, keepdim=True).clamp_min(1e-300)
        unit = torch.exp2(torch.ceil(torch.log2(top)) - s)
        return torch.round(X / unit) * unit

    Ah, Bh = head(A, 1), head(B, 0)
    return (Ah @ (B - Bh) + (A - Ah) @ B) + Ah @ Bh


def exact(case, seed):
    path = case["path"]
    if path == "batched":
        s, (A, B, C), (oa, ob, oc) = _batched_inputs(case, seed)
        out = torch.empty_like(C)
        for (M, N, K), a, b, c in zip(s.tolist(), oa.tolist(), ob.tolist(), oc.tolist()):
            P = _product(A[a:a + M * K].view(M, K), B[b:b + K * N].view(K, N))
            out[c:c + M * N] = (case["alpha"] * P + case["beta"] * C[c:c + M * N].view(M, N)).view(-1)
        return out
    if path == "mlp":
        return _mlp_exact(case, seed)
    A, B, C = (x.double() for x in _gemm_inputs(case, seed))
    P = _product(A.t().contiguous() if case["trans_a"] else A,
                 B.t().contiguous() if case["trans_b"] else B)
    return case["alpha"] * P + case["beta"] * C


def _mlp_exact(case, seed):
    B, C = case["batch"], case["outputs"]
    sizes, flag, T, mask, params = _mlp_inputs(case, seed)
    l2 = torch.log2(sizes.double())
    X = torch.stack([l2[:, 0], l2[:, 1], l2[:, 2], l2[:, 0] - l2[:, 1], l2[:, 1] - l2[:, 2],
                     l2[:, 0] - l2[:, 2], flag.double()], 1)
    X = (X - X.mean(0)) / X.std(0, unbiased=False)
    p = params.double().requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(p, [64 * 7, 64, 64 * 64, 64, C * 64, C])
    z1 = X @ W1.view(64, 7).t() + b1
    z2 = torch.relu(z1) @ W2.view(64, 64).t() + b2
    Y = torch.relu(z2) @ W3.view(C, 64).t() + b3
    count = mask.double().sum()
    loss = (mask.double() * (Y - T.double()) ** 2).sum() / count
    loss.backward()
    g = p.grad
    m, v = 0.1 * g, 0.001 * g * g
    # after one step the bias corrections cancel: m / (1 - beta1) = g, v / (1 - beta2) = g^2
    new = p.detach() - 3e-3 * g / (g.abs() + 1e-8)
    cache = torch.cat([z1, z2], 1)
    return [Y.detach(), cache.detach(), torch.stack([loss.detach(), count]), g, new, m, v]
