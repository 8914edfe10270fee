"""What is timed: the calls a user of this library makes, over the range of
sizes, storage types and options it is used with.

A case is one of five kinds:
  decompose  tt.decompose of a dense tensor (Alg. 3, or Alg. 4 with method
             "rsi"), FP32 or BF16 storage; "dims" of two sizes is one mode
             step on its own (an unfolding and its core)
  batch      many independent problems of uneven order, sizes and ranks as
             one graph launch (tt.BatchGraph)
  passes     the streaming passes over one unfolding (tt.tt_pass): sketch,
             Gram-apply, projection
  permute    tt.permute_convert, a strided tensor made dense in another mode
             order and converted to the storage type
  eig        tt.sym_eig_top, the Rayleigh-Ritz eigensolver

Tensors are of low TT rank plus 5% Gaussian noise.  Every unfolding's
leading squared singular values are evenly spaced from 1 down to 0.2, so
that each column of a core is determined by the input (a core whose singular
values nearly coincide is determined only up to a rotation) and two
implementations can be compared entry by entry.  For the same reason the
decompositions of BF16 tensors keep their remainders in FP32 (an option of
the library): with BF16 remainders the last core is itself rounded to BF16,
and one rounding that falls the other way is 2^-9 of an entry.  The passes
over BF16 remainders are timed as single unfoldings.
"""
import math

import torch

import paper_2308_01480_gb300 as tt

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def _dims(text):
    return [int(x) for x in text.split("x")]


def listed():
    return [
        # the smallest call: every kernel is short, launches and the small algebra count
        dict(name="tt16x4_f32", kind="decompose", dims="16x16x16x16", dtype="f32", rank=4, p=5, q=2, method="rbki"),
        # an ordinary FP32 decomposition
        dict(name="tt32x5_f32", kind="decompose", dims="32x32x32x32x32", dtype="f32", rank=8, p=5, q=3,
             method="rbki"),
        # the largest FP32 decomposition: the 45^5 tensor of the accuracy study (odd sizes, unaligned rows)
        dict(name="tt45x5_f32", kind="decompose", dims="45x45x45x45x45", dtype="f32", rank=4, p=2, q=2,
             method="rbki"),
        # the precision form on the 40^5 tensor of the benchmark, FP32 remainders
        dict(name="tt40x5_bf16", kind="decompose", dims="40x40x40x40x40", dtype="bf16", rank=10, p=10, q=4,
             method="rbki"),
        # the benchmark's second mode on its own: an 800-row BF16 unfolding, five Krylov blocks
        dict(name="mode800_bf16", kind="decompose", dims="800x64000", dtype="bf16", rank=10, p=10, q=4,
             method="rbki"),
        # the second mode of the 256 x 256 x 64 x 32 tensor at rank 30: a tall unfolding, FP32
        dict(name="mode7680_f32", kind="decompose", dims="7680x2048", dtype="f32", rank=10, p=10, q=3,
             method="rbki"),
        # subspace iteration (Alg. 4) on the 500^3 tensor of the accuracy study
        dict(name="rsi500x3_bf16", kind="decompose", dims="500x500x500", dtype="bf16", rank=8, p=4, q=2,
             method="rsi"),
        # BF16 storage whose rows are not 16-byte aligned (odd trailing sizes)
        dict(name="ragged_bf16", kind="decompose", dims="61x53x47x45", dtype="bf16", rank=8, p=5, q=2,
             method="rbki"),
        # a batch of uneven problems in one graph launch, as the batched workload draws them
        dict(name="batch48_bf16", kind="batch", count=48, dtype="bf16", p=5, q=2, cap=1 << 22),
        # the streaming passes over the 256 x 524288 first unfolding of the 256 x 256 x 64 x 32 tensor
        dict(name="passes256_bf16", kind="passes", m=256, n=524288, b=40, dtype="bf16"),
        # canonicalising a 256 x 256 x 64 x 32 tensor: modes permuted, FP32 to BF16
        dict(name="permute_f32_bf16", kind="permute", dims="256x256x64x32", perm="3x1x0x2", dtype="f32", to="bf16"),
        # Rayleigh-Ritz of a 150-column basis
        dict(name="eig150", kind="eig", k=150, r=20),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["decompose", "decompose", "decompose", "mode", "mode", "batch", "passes", "permute", "eig"])
    if kind == "decompose":
        d = rng.choice([3, 4, 5])
        while True:
            dims = [_log_int(rng, 12, 500) for _ in range(d)]
            if 2 ** 14 <= math.prod(dims) <= 2 ** 26:
                break
        return dict(kind="decompose", dims="x".join(map(str, dims)), dtype=rng.choice(["f32", "bf16"]),
                    rank=rng.randint(2, 8), p=rng.randint(2, 10), q=rng.randint(2, 4),
                    method=rng.choice(["rbki", "rbki", "rsi"]))
    if kind == "mode":
        # taller BF16 unfoldings stream their powers through a BF16 block,
        # whose rounding any change of summation order moves: FP32 there
        m = _log_int(rng, 40, 8000)
        n = _log_int(rng, 200, min(2 ** 20, 2 ** 26 // m))
        if rng.random() < 0.5:
            n = (n + 7) // 8 * 8
        return dict(kind="decompose", dims="%dx%d" % (m, n), dtype=rng.choice(["f32", "bf16"]) if m <= 1024 else "f32",
                    rank=rng.randint(2, 10), p=rng.randint(2, 10), q=rng.randint(2, 4), method="rbki")
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 40), dtype=rng.choice(["f32", "bf16"]), p=5, q=2, cap=1 << 21)
    if kind == "passes":
        m = _log_int(rng, 16, 2048)
        n = _log_int(rng, 512, min(2 ** 21, 2 ** 26 // m))
        if rng.random() < 0.6:
            n = (n + 7) // 8 * 8
        return dict(kind="passes", m=m, n=n, b=rng.randint(4, 48), dtype=rng.choice(["f32", "bf16"]))
    if kind == "permute":
        d = rng.choice([3, 4, 5])
        while True:
            dims = [_log_int(rng, 3, 300) for _ in range(d)]
            if 2 ** 14 <= math.prod(dims) <= 2 ** 27:
                break
        perm = list(range(d))
        rng.shuffle(perm)
        return dict(kind="permute", dims="x".join(map(str, dims)), perm="x".join(map(str, perm)),
                    dtype=rng.choice(["f32", "bf16"]), to=rng.choice(["f32", "bf16"]))
    k = _log_int(rng, 8, 160)
    return dict(kind="eig", k=k, r=rng.randint(1, min(30, max(1, k // 3))))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _factor(n, r, g):
    return torch.linalg.qr(torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64))[0].float().contiguous()


def _spectrum(r):
    return (1.0 - 0.8 * torch.arange(r, device="cuda") / max(1, r - 1)).sqrt()


def _tensor(dims, r, g, dtype, noise=0.05):
    """sum_j s_j a_j (x) b_j (x) ... with orthonormal factors, entries of unit
    size, plus Gaussian noise of that relative size."""
    r = min(r, min(dims))
    s = _spectrum(r)
    rest = _factor(dims[-1], r, g).T
    for n in reversed(dims[1:-1]):
        rest = (_factor(n, r, g).T.unsqueeze(2) * rest.unsqueeze(1)).reshape(r, -1)
    X = (_factor(dims[0], r, g) * s) @ rest
    X *= math.sqrt(math.prod(dims)) / float(s.norm())
    X += noise * torch.randn(X.shape, generator=g, device="cuda")
    return X.reshape(dims).to(DTYPES[dtype])


def _batch_problems(case, seed):
    """Sizes and ranks of the batch: part of the workload, the same for every
    seed of the inputs."""
    rng = torch.Generator()
    rng.manual_seed(1000 + case["count"])

    def ints(lo, hi, n):
        return [int(x) for x in torch.randint(lo, hi + 1, (n,), generator=rng)]
    out = []
    for i in range(case["count"]):
        d = ints(3, 6, 1)[0]
        while True:
            dims = ints(8, 64, d)
            if math.prod(dims) <= case["cap"]:
                break
        out.append((dims, min(ints(2, 8, 1)[0], min(dims)), 1000 * (seed % 100003) + i))
    return out


def prepare(case, seed):
    kind, g = case["kind"], _gen(seed)
    if kind == "decompose":
        dims = _dims(case["dims"])
        A = _tensor(dims, case["rank"], g, case["dtype"])
        ranks = [case["rank"]] * (len(dims) - 1)
        opts = tt.options(storage=tt.TT_BF16 if case["dtype"] == "bf16" else tt.TT_F32, remainder=tt.TT_F32,
                          method=tt.TT_METHOD_RSI if case["method"] == "rsi" else tt.TT_METHOD_RBKI)
        ws = torch.empty(tt.workspace_size(dims, ranks, case["p"], case["q"], opts), dtype=torch.uint8, device="cuda")
        return dict(kind=kind, A=A, ranks=ranks, p=case["p"], q=case["q"], opts=opts, ws=ws, seed=seed)
    if kind == "batch":
        plan = _batch_problems(case, seed)
        sizes = []
        for dims, r, _ in plan:
            sizes.append(tt.core_sizes(dims, [r] * (len(dims) - 1)))
        flat = torch.zeros(sum(sum(c) for _, c in sizes), device="cuda")
        probs, at = [], 0
        for (dims, r, s), (rr, counts) in zip(plan, sizes):
            cores = []
            for k, c in enumerate(counts):
                cores.append(flat[at:at + c].view(rr[k], dims[k], rr[k + 1]))
                at += c
            probs.append(tt.Problem(_tensor(dims, r, g, case["dtype"]), [r] * (len(dims) - 1), case["p"], case["q"],
                                    s, cores=cores))
        opts = tt.options(storage=tt.TT_BF16 if case["dtype"] == "bf16" else tt.TT_F32, remainder=tt.TT_F32,
                          batch_streams=32)
        return dict(kind=kind, graph=tt.BatchGraph(probs, opts), flat=flat)
    if kind == "passes":
        m, n, b = case["m"], case["n"], case["b"]
        C = _tensor([m, n], min(20, m), g, case["dtype"])
        code = tt.TT_BF16 if case["dtype"] == "bf16" else tt.TT_F32
        ops = (tt.TT_PASS_SKETCH, tt.TT_PASS_GRAMAPPLY, tt.TT_PASS_PROJECT)
        ws = torch.empty(max(tt.pass_workspace_size(op, m, n, b, code) for op in ops), dtype=torch.uint8,
                         device="cuda")
        return dict(kind=kind, C=C, ws=ws, omega=torch.randn(n, b, generator=g, device="cuda"),
                    x=_factor(m, b, g) if m >= b else torch.randn(m, b, generator=g, device="cuda"))
    if kind == "permute":
        A = torch.randn(_dims(case["dims"]), generator=g, device="cuda").to(DTYPES[case["dtype"]])
        return dict(kind=kind, A=A, perm=_dims(case["perm"]), to=DTYPES[case["to"]])
    k, r = case["k"], case["r"]
    V = _factor(k, k, g)
    lam = torch.cat([_spectrum(r) ** 2, 0.01 * torch.rand(k - r, generator=g, device="cuda")])
    H = (V * lam) @ V.T
    return dict(kind=kind, H=((H + H.T) / 2).contiguous(), r=r)


# --------------------------------------------------------------------- run
def run(state):
    kind = state["kind"]
    if kind == "decompose":
        return tt.decompose(state["A"], state["ranks"], state["p"], state["q"], omega_seed=state["seed"],
                            opts=state["opts"], workspace=state["ws"])[0]
    if kind == "batch":
        state["graph"].launch()
        return state["flat"]
    if kind == "passes":
        C, ws = state["C"], state["ws"]
        return [tt.tt_pass(tt.TT_PASS_SKETCH, C, x=state["omega"], workspace=ws),
                tt.tt_pass(tt.TT_PASS_GRAMAPPLY, C, x=state["x"], workspace=ws),
                tt.tt_pass(tt.TT_PASS_PROJECT, C, x=state["x"], y_dtype=C.dtype, workspace=ws)]
    if kind == "permute":
        return tt.permute_convert(state["A"], state["perm"], state["to"])
    return list(tt.sym_eig_top(state["H"], state["r"]))


# -------------------------------------------------------------------- work
def _decompose_work(dims, rank, p, q, elem):
    """Per mode: the sketch and the projection read the unfolding once each,
    the powers cost the cheaper of two products a power and one Gram."""
    rr, _ = tt.core_sizes(dims, [rank] * (len(dims) - 1))
    flops, out = 0.0, 0
    for k in range(len(dims) - 1):
        m, n, r = rr[k] * dims[k], math.prod(dims[k + 1:]), rr[k + 1]
        b = min(r + p, m, n)
        flops += 2.0 * m * n * (b + r) + min(4.0 * m * n * b * (q + 1), 1.0 * m * m * n)
        out += m * r
    out += rr[-2] * dims[-1]
    return math.prod(dims) * elem + 4 * out, flops


def work(case):
    kind = case["kind"]
    elem = {"f32": 4, "bf16": 2}
    if kind == "decompose":
        by, fl = _decompose_work(_dims(case["dims"]), case["rank"], case["p"], case["q"], elem[case["dtype"]])
        return {"bytes": by, "flops": fl}
    if kind == "batch":
        both = [_decompose_work(dims, r, case["p"], case["q"], elem[case["dtype"]])
                for dims, r, _ in _batch_problems(case, 0)]
        return {"bytes": sum(x[0] for x in both), "flops": sum(x[1] for x in both)}
    if kind == "passes":
        m, n, b, e = case["m"], case["n"], case["b"], elem[case["dtype"]]
        return {"bytes": 3 * m * n * e + n * b * (4 + e) + 4 * 4 * m * b, "flops": 8.0 * m * n * b}
    if kind == "permute":
        total = math.prod(_dims(case["dims"]))
        return {"bytes": total * (elem[case["dtype"]] + elem[case["to"]]), "flops": 0}
    k, r = case["k"], case["r"]
    return {"bytes": 4 * (k * k + k * r + r), "flops": 4.0 / 3.0 * k ** 3 + 4.0 * k * k * r}


# ------------------------------------------------------------------- exact
def exact(case, seed):
    """In 64 bits.  A core or an eigenvector is defined up to the sign of each
    column, so those outputs have no exact value."""
    kind = case["kind"]
    if kind in ("decompose", "batch"):
        return None
    s = prepare(case, seed)
    if kind == "permute":
        return s["A"].permute(s["perm"]).contiguous().to(s["to"])
    if kind == "eig":
        return [None, torch.linalg.eigvalsh(s["H"].double()).flip(0)[:s["r"]]]
    C, x = s["C"].double(), s["x"].double()
    T = x.T @ C
    return [C @ s["omega"].double(), C @ T.T, T]
