"""The work the FP4 linear layer is put to in use, as cases that can be timed and compared.

A case is a dict of plain values.  `listed()` holds the fixed ones, `draw(rng)` makes more of the same
ranges, `prepare` makes what a program has in hand before the call, `run` is one pass through the
public entry points of the package.  Kinds of a case:

  step      forward and backward of one linear (training)
  layer     forward and backward of the seven linears of a decoder layer; q/k/v and gate/up read the
            same activation, as in the model (training)
  fwd       forward alone on a weight that is already quantised (evaluation, or the later
            micro-batches of an optimizer step)
  quantize  one tensor quantised by itself (an activation with or without the clamp, a weight)
  gemm      the GEMM on codes that are already there
  host      forward and backward with pinned host buffers

Sizes are those of the LLaMA 1.3B / 7B / 13B linears and multiples of 128 around them; tensors follow
the package's synthetic workloads: normal weights (0.02) and output gradients (1e-3), activations
that are normal, Student-t or Laplace with outliers in a few channels or in single elements.
"""
import math

import torch

import paper_2501_17116_b200 as fp4

DEV = "cuda:0"
E2M1, E4M3, E5M2 = 0, 1, 2          # operand formats of the package

# activation families: (distribution, share of outliers, their factor, where they sit)
ACTIVATIONS = {
    "normal": ("normal", 0.01, 50.0, "channels"),
    "student": ("student", 0.005, 30.0, "channels"),
    "student50": ("student", 0.01, 50.0, "channels"),
    "laplace": ("laplace", 0.002, 100.0, "elements"),
}


def listed():
    return [
        # the smallest layer of the test configurations: latency and launches count
        dict(name="step-fc1024", kind="step", M=256, K=1024, N=1024, alpha=0.99, act="normal"),
        # one optimizer micro-step of a 1.3B decoder layer, the paper's main setting
        dict(name="layer-1.3b", kind="layer", M=4096, K=2048, N=5504, alpha=0.999, act="student"),
        # 7B MLP, long contraction in the forward, heavy residual
        dict(name="step-7b-down", kind="step", M=8192, K=11008, N=4096, alpha=0.99, act="normal"),
        # 13B attention projection, outliers in single elements and a light clamp
        dict(name="step-13b-attn", kind="step", M=8192, K=5120, N=5120, alpha=0.9999, act="laplace"),
        # the largest linear: 13B gate/up projection of 16384 tokens, heavy residual
        dict(name="step-13b-gate", kind="step", M=16384, K=5120, N=13824, alpha=0.99, act="student50"),
        # evaluation of few tokens on a 7B up projection
        dict(name="fwd-128-7b-up", kind="fwd", M=128, K=4096, N=11008, alpha=0.999, act="normal"),
        # evaluation of a batch whose token count fills no power of two, strongest clamp of the paper
        dict(name="fwd-1920-1.3b-down", kind="fwd", M=1920, K=5504, N=2048, alpha=0.97, act="student"),
        # mixed precision: FP4 weight, FP8 activation and output gradient, no clamp
        dict(name="step-w4a8", kind="step", M=4096, K=2048, N=2048, alpha=1.0, act="student", fmt_a=E4M3, fmt_dy=E5M2),
        # the GEMM by itself at a square size
        dict(name="gemm-8192", kind="gemm", M=8192, K=8192, N=8192, out_f32=False),
        # an activation quantised by itself with the clamp (shared by several consumers)
        dict(name="quantize-act", kind="quantize", M=8192, K=4096, alpha=0.999, act="normal", axis=0),
        # a weight quantised once per optimizer step, odd number of column tiles
        dict(name="quantize-weight", kind="quantize", M=5120, K=13824, alpha=1.0, act="weight", axis=1),
        # a step whose tensors live in pinned host memory
        dict(name="host-1.3b-q", kind="host", M=4096, K=2048, N=2048, alpha=0.999, act="student"),
    ]


def _size(rng, lo, hi):
    """A multiple of 128, spread evenly over the logarithm of [lo, hi]."""
    return 128 * max(1, round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 128))


def _cost(M, K, N, alpha, act):
    """Rough cost of a step: the GEMMs, plus the residual (dearer where no channel collects it)."""
    return M * K * N * (1.0 + (400.0 if act == "laplace" else 100.0) * (1.0 - alpha))


def draw(rng):
    kind = rng.choices(["step", "fwd", "quantize", "gemm", "host"], [9, 5, 3, 2, 1])[0]
    while True:
        M, K, N = _size(rng, 128, 16384), _size(rng, 512, 13824), _size(rng, 512, 13824)
        alpha = rng.choice([0.97, 0.99, 0.995, 0.999, 0.9999, 1.0])
        act = rng.choice(["normal", "student", "student50", "laplace"])
        if _cost(M, K, N, alpha, act) > _cost(16384, 5120, 13824, 0.99, "student50") / 2:
            continue
        if kind == "host" and M * K + K * N + M * N > 1e8:
            continue
        break
    if kind == "gemm":
        return dict(kind=kind, M=M, K=K, N=N, out_f32=rng.random() < 0.5)
    if kind == "quantize":
        if rng.random() < 0.4:
            return dict(kind=kind, M=K, K=N, alpha=1.0, act="weight", axis=1)
        return dict(kind=kind, M=M, K=K, alpha=alpha, act=act, axis=0)
    case = dict(kind=kind, M=M, K=K, N=N, alpha=alpha, act=act)
    if kind == "step":
        if rng.random() < 0.2:                       # the mixed-precision settings
            fmt = rng.choice(["a", "w", "dy"])
            if fmt == "a":
                case.update(alpha=1.0, fmt_a=rng.choice([E4M3, E5M2]))
            elif fmt == "w":
                case.update(fmt_w=E4M3)
            case.update(fmt_dy=rng.choice([E4M3, E5M2]) if fmt == "dy" else E2M1)
        elif rng.random() < 0.15:
            case.update(out_f32=True)
        if rng.random() < 0.15:
            case.update(dge=False)                   # straight-through estimator
    return case


# ------------------------------------------------------------------------------------------------
def _activation(g, M, K, act):
    dist, frac, scale, where = ACTIVATIONS[act]
    a = torch.randn((M, K), device=DEV, generator=g)
    if dist == "student":                            # three degrees of freedom
        d = torch.zeros((M, K), device=DEV)
        t = torch.empty((M, K), device=DEV)
        for _ in range(3):
            t.normal_(generator=g)
            d.addcmul_(t, t)
        a.mul_(d.div_(3.0).rsqrt_())
        del t, d
    elif dist == "laplace":
        e = torch.empty((M, K), device=DEV).exponential_(generator=g)
        a = torch.copysign(e, a)
    if where == "elements":
        a = torch.where(torch.rand((M, K), device=DEV, generator=g) < frac, a * scale, a)
    else:
        ch = torch.randperm(K, device=DEV, generator=g)[:max(1, round(frac * K))]
        a[:, ch] *= scale
    return a.to(torch.bfloat16)


def _normal(g, rows, cols, std):
    return torch.randn((rows, cols), device=DEV, generator=g).mul_(std).to(torch.bfloat16)


def _linears(case):
    """[(K, N, index of the activation, whether that activation is already quantised)]"""
    K, N = case["K"], case.get("N", 0)
    if case["kind"] != "layer":
        return [(K, N, 0, False)]
    return [(K, K, 0, False), (K, K, 0, True), (K, K, 0, True), (K, K, 1, False),      # q k v o
            (K, N, 2, False), (K, N, 2, True), (N, K, 3, False)]                       # gate up down


def _gemm_kind(case):
    fp8 = case.get("fmt_a", E2M1) or case.get("fmt_w", E2M1) or case.get("fmt_dy", E2M1)
    return fp4.FP4_GEMM_F8F6F4 if fp8 else fp4.FP4_GEMM_MXF4


def prepare(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    M, kind = case["M"], case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "gemm":
        s["ctx"] = fp4.Context.for_shape(M, case["K"], case["N"])
        a, b = _normal(g, M, case["K"], 1.0), _normal(g, case["N"], case["K"], 0.02)
        s["a"] = fp4.fp4_quantize(s["ctx"], a, 0, codes_t=False)
        s["b"] = fp4.fp4_quantize(s["ctx"], b, 0, codes_t=False)
        s["out"] = torch.empty((M, case["N"]), dtype=torch.float32 if case["out_f32"] else torch.bfloat16, device=DEV)
        return s
    if kind == "quantize":
        K = case["K"]
        s["ctx"] = fp4.Context.for_shape(M, K, K)
        s["x"] = _normal(g, M, K, 0.02) if case["act"] == "weight" else _activation(g, M, K, case["act"])
        s["q"] = fp4.QTensor(M, K, case["axis"], DEV, fp4.tail_capacity(M, K, case["alpha"]))
        return s
    lin = _linears(case)
    if kind == "host":
        K, N = case["K"], case["N"]
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)          # noqa: E731
        s["in"] = [pin(_activation(g, M, K, case["act"])), pin(_normal(g, K, N, 0.02)), pin(_normal(g, M, N, 1e-3))]
        s["out"] = [torch.empty(shape, dtype=torch.bfloat16, pin_memory=True) for shape in ((M, N), (M, K), (K, N))]
        lib = fp4.load_library()
        s["ctx"] = fp4.Context(0, int(lib.fp4_step_host_workspace_bytes(M, K, N, float(case["alpha"]))))
        return s
    # one workspace serves all linears of the case
    lib = fp4.load_library()
    s["ctx"] = fp4.Context(0, max(int(lib.fp4_workspace_bytes(M, K, N)) for K, N, _, _ in lin))
    dt = torch.float32 if case.get("out_f32") else torch.bfloat16
    acts = {}
    s["linears"] = []
    for K, N, which, shared in lin:
        if not shared:
            cap = fp4.tail_capacity(M, K, case["alpha"])
            acts[which] = (_activation(g, M, K, case["act"]),
                           fp4.QTensor(M, K, 0, DEV, cap, fmt=case.get("fmt_a", E2M1)))
        a, sa = acts[which]
        p = {"A": a, "sa": sa, "reuse_a": shared, "W": _normal(g, K, N, 0.02),
             "sw": fp4.QTensor(K, N, 1, DEV, fmt=case.get("fmt_w", E2M1)),
             "y": torch.empty((M, N), dtype=dt, device=DEV)}
        if kind == "fwd":                            # the weight was quantised when it last changed
            fp4.fp4_quantize(s["ctx"], p["W"], 1, out=p["sw"])
        else:
            p["dY"] = _normal(g, M, N, 1e-3)
            p["dA"] = torch.empty((M, K), dtype=dt, device=DEV)
            p["dW"] = torch.empty((K, N), dtype=dt, device=DEV)
        s["linears"].append(p)
    return s


def _operand(q):
    """What a quantised operand holds for its later uses."""
    out = {"codes": q.codes, "codes_t": q.codes_t, "amax": q.amax}
    if q.sparse_cap:
        out.update(thresholds=q.thresholds, nnz=q.nnz, csr_rowptr=q.csr_rowptr, csr_col=q.csr_col, csr_val=q.csr_val,
                   csc_colptr=q.csc_colptr, csc_row=q.csc_row, csc_val=q.csc_val)
    return out


def run(s):
    case, kind, ctx = s["case"], s["kind"], s["ctx"]
    if kind == "gemm":
        return fp4.fp4_gemm(ctx, s["a"].codes, s["b"].codes, s["a"].amax, s["b"].amax, out_f32=case["out_f32"], out=s["out"])
    if kind == "quantize":
        return _operand(fp4.fp4_quantize(ctx, s["x"], case["axis"], alpha=case["alpha"], out=s["q"]))
    if kind == "host":
        fp4.fp4_linear_step_host(ctx, *s["in"], case["alpha"], *s["out"], read_status=False)
        return s["out"]
    gk, f32 = _gemm_kind(case), bool(case.get("out_f32"))
    for p in s["linears"]:
        fp4.fp4_linear_fwd(ctx, p["A"], p["W"], case["alpha"], saved_a=p["sa"], saved_w=p["sw"], reuse_w=kind == "fwd",
                           reuse_a=p["reuse_a"], gemm_kind=gk, out_f32=f32, out=p["y"])
    if kind == "fwd":
        return {"y": p["y"], "saved_a": _operand(p["sa"])}
    for p in reversed(s["linears"]):
        fp4.fp4_linear_bwd(ctx, p["dY"], p["W"], p["sa"], p["sw"], dge_on=case.get("dge", True), gemm_kind=gk, out_f32=f32,
                           dA=p["dA"], dW=p["dW"], dy_fmt=case.get("fmt_dy", E2M1))
    if kind == "step":
        return {"y": p["y"], "dA": p["dA"], "dW": p["dW"], "saved_a": _operand(p["sa"]), "saved_w": _operand(p["sw"])}
    return [(p["y"], p["dA"], p["dW"]) for p in s["linears"]]


def work(case):
    """Inputs read once, outputs written once; the products of the GEMMs and of the residual."""
    M, kind = case["M"], case["kind"]
    nnz = lambda rows, cols: 2 * round((1.0 - case["alpha"]) * rows * cols)                    # noqa: E731
    if kind == "gemm":
        K, N = case["K"], case["N"]
        return {"bytes": (M * K + K * N) / 2 + 4 * (M + N) + (4 if case["out_f32"] else 2) * M * N, "flops": 2.0 * M * K * N}
    if kind == "quantize":                           # both code layouts, the residual by rows and by columns
        K = case["K"]
        return {"bytes": 3.0 * M * K + 16 * nnz(M, K), "flops": 3.0 * M * K}
    out = 4 if case.get("out_f32") else 2
    byte, flop = 0.0, 0.0
    for K, N, _, shared in _linears(case):
        e = nnz(M, K)
        code = lambda f: 0.5 if case.get(f, E2M1) == E2M1 else 1.0                             # noqa: E731
        saved_a = 0.0 if shared else 2 * code("fmt_a") * M * K + 16 * e
        read_a = 0.0 if shared else 2.0 * M * K
        flop += 2.0 * M * K * N + 2.0 * e * N
        byte += read_a + out * M * N
        if kind == "host":
            saved_a = 0.0                            # the saved operands never leave the library here
        byte += saved_a
        if kind == "fwd":
            byte += K * N / 2 + (2.0 * K * N if e else 0.0)
            continue
        flop += 4.0 * M * K * N + 2.0 * e * N
        byte += 2.0 * K * N + (0.0 if kind == "host" else 2 * code("fmt_w") * K * N)           # W and its codes
        byte += 2.0 * M * N + out * (M * K + K * N)                                            # dY, dA, dW
    return {"bytes": byte, "flops": flop}


def tolerance(case):
    """Codes, amax, thresholds and the residual are specified bit for bit.  Outputs in BF16: sums of another
    order move a value across a rounding boundary now and then, by one unit in the last place
    (2^-7 of the value at most).  Outputs in fp32: sums of another order, some over FP8 products."""
    if case["kind"] == "quantize":
        return "exact"
    if case.get("out_f32"):
        return {"rel": 1e-5, "max": 1e-3}
    return {"rel": 2e-3, "max": 1e-2}
