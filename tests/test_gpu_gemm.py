"""GPU parity of fp4_gemm against the oracle: exact accumulators and the two de-scales."""
import numpy as np
import pytest
import torch

from conftest import pair_launches
from oracle import fp4_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    c = lib.Context(0, 64 << 20)
    yield c
    c.close()


def _codes(rng, rows, cols):
    c = rng.integers(0, 16, (rows, cols), dtype=np.uint8)
    c[c == 8] = 0                      # the library never writes a negative-zero code
    return c


def _run(lib, ctx, ca, cb, kind, **kw):
    a = torch.from_numpy(O.pack_nibbles(ca)).cuda()
    b = torch.from_numpy(O.pack_nibbles(cb)).cuda()
    ctx.status.zero_()
    out = lib.fp4_gemm(ctx, a, b, gemm_kind=kind, **kw)
    torch.cuda.synchronize()
    assert ctx.read_status() == 0
    return out


KINDS = [0, 1]          # FP4_GEMM_MXF4, FP4_GEMM_F8F6F4
SHAPES = [(128, 128, 128), (128, 256, 256), (256, 384, 640), (384, 640, 1152), (512, 1024, 4096)]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", SHAPES)
def test_accumulators_are_exact(lib, ctx, kind, shape):
    """Every product is a multiple of 1/4 and the sums stay below 2^24 quarter units, so the
    fp32 accumulators must equal the oracle's integers exactly, in any summation order."""
    I, J, C = shape
    rng = np.random.default_rng(I + J + C + kind)
    ca, cb = _codes(rng, I, C), _codes(rng, J, C)
    got = _run(lib, ctx, ca, cb, kind).cpu().numpy().astype(np.float64)
    np.testing.assert_array_equal(got, O.gemm_codes(ca, cb))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(128, 1024, 512), (128, 11008, 256), (1024, 1024, 128), (512, 5120, 128), (2304, 1408, 256),
                                   (1152, 3200, 384), (640, 13824, 128), (2048, 2048, 256)])
@pytest.mark.parametrize("f32", [True, False])
def test_tile_widths(lib, ctx, kind, shape, f32):
    """Shapes for which the launch picks tiles of 32 to 256 columns, most with a ragged last tile: fp32 exact,
    BF16 the rounding of the exact sum."""
    I, J, C = shape
    rng = np.random.default_rng(I + J + C)
    ca, cb = _codes(rng, I, C), _codes(rng, J, C)
    got = _run(lib, ctx, ca, cb, kind, out_f32=f32).cpu()
    val = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64)
    want = val[torch.from_numpy(ca.astype(np.int64))] @ val[torch.from_numpy(cb.astype(np.int64))].T      # exact in double
    assert torch.equal(got, want.float() if f32 else want.to(torch.bfloat16))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(4224, 4096, 4224), (3200, 2944, 6144)])
@pytest.mark.parametrize("f32", [True, False])
def test_pairs_of_ctas(lib, ctx, kind, shape, f32):
    """Sizes that are computed by pairs of CTAs, with an odd number of 128-row blocks (the last pair's second half is
    missing) and a ragged last tile: exact; and a wait that runs out in a pair ends both CTAs."""
    I, J, C = shape
    rng = np.random.default_rng(I + J + C)
    ca, cb = _codes(rng, I, C), _codes(rng, J, C)
    got = _run(lib, ctx, ca, cb, kind, out_f32=f32)
    val = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")
    dec = lambda c: val[torch.from_numpy(c).cuda().long()]                                     # noqa: E731
    want = (dec(ca) @ dec(cb).T).to(got.dtype)                                                 # exact in double
    assert torch.equal(got, want)
    c = lib.Context(0, 1 << 20)
    a, b = torch.from_numpy(O.pack_nibbles(ca)).cuda(), torch.from_numpy(O.pack_nibbles(cb)).cuda()
    assert pair_launches(lambda: lib.fp4_gemm(c, a, b, gemm_kind=kind, out_f32=f32, out=got)) == 1
    c.debug_set(lib.binding.FP4_DEBUG_WAIT_LIMIT_US, 1000)
    c.debug_set(lib.binding.FP4_DEBUG_SKIP_FILL, 7)
    lib.fp4_gemm(c, a, b, gemm_kind=kind, out_f32=f32)
    torch.cuda.synchronize()
    assert c.read_status() & lib.FP4_DEV_TIMEOUT
    c.debug_set(lib.binding.FP4_DEBUG_SKIP_FILL, -1)
    c.debug_set(lib.binding.FP4_DEBUG_WAIT_LIMIT_US, 0)
    c.status.zero_()
    again = lib.fp4_gemm(c, a, b, gemm_kind=kind, out_f32=f32)
    torch.cuda.synchronize()
    assert c.read_status() == 0 and torch.equal(again, want)
    c.close()


def test_both_gradients_by_pairs_of_ctas(lib):
    """The two backward GEMMs of a layer of 63 x 25 row blocks share a launch of pairs; slices of the layer, too small for
    pairs, give the same bits (every sum is exact; the scales are pinned by a large value in each slice)."""
    M, K, N = 8064, 3200, 4096
    g = torch.Generator(device="cuda").manual_seed(3)
    A = torch.randn((M, K), device="cuda", generator=g).bfloat16()
    W = (torch.randn((K, N), device="cuda", generator=g) * 0.02).bfloat16()
    dY = (torch.randn((M, N), device="cuda", generator=g) * 1e-3).bfloat16()
    A[:, 0] = A[:, K - 256] = 8.0
    W[0] = W[K - 256] = 0.25
    c = lib.Context.for_shape(M, K, N)
    _, sa, sw = lib.fp4_linear_fwd(c, A, W, 1.0)
    dA, dW = lib.fp4_linear_bwd(c, dY, W, sa, sw)
    assert pair_launches(lambda: lib.fp4_linear_bwd(c, dY, W, sa, sw, dA=torch.empty_like(dA), dW=torch.empty_like(dW))) == 1
    for k0 in (0, K - 256):
        As, Ws = A[:, k0:k0 + 256].contiguous(), W[k0:k0 + 256].contiguous()
        _, sas, sws = lib.fp4_linear_fwd(c, As, Ws, 1.0)
        _, dWs = lib.fp4_linear_bwd(c, dY, Ws, sas, sws)
        assert torch.equal(dW[k0:k0 + 256], dWs)
    for m0 in (0, M - 256):
        _, sas, _ = lib.fp4_linear_fwd(c, A[m0:m0 + 256].contiguous(), W, 1.0)
        dAs, _ = lib.fp4_linear_bwd(c, dY[m0:m0 + 256].contiguous(), W, sas, sw)
        assert torch.equal(dA[m0:m0 + 256], dAs)
    assert c.read_status() == 0
    c.close()


@pytest.mark.parametrize("a_fmt,b_fmt", [("e4m3", "e2m1"), ("e2m1", "e4m3"), ("e4m3", "e5m2"), ("e5m2", "e4m3")])
@pytest.mark.parametrize("shape", [(4224, 4096, 4224), (3200, 2944, 6144)])
def test_pairs_of_ctas_with_fp8_operands(lib, ctx, a_fmt, b_fmt, shape):
    """FP8 bytes in a pair: both CTAs' copies count in bytes read, which differ by the operands' formats; an odd number of row
    blocks and a ragged last tile.  The products are exact, an instruction adds 32 of them into the fp32 accumulator and
    cuts the sum off: each is off by at most 2^-23 of the summed magnitudes."""
    I, J, C = shape
    g = torch.Generator(device="cuda").manual_seed(I + len(a_fmt + b_fmt))
    types = {"e4m3": torch.float8_e4m3fn, "e5m2": torch.float8_e5m2}
    val = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")

    def operand(rows, fmt):
        if fmt == "e2m1":
            c = torch.randint(0, 256, (rows, C // 2), dtype=torch.uint8, device="cuda", generator=g)
            return c, torch.stack([val[(c & 15).long()], val[(c >> 4).long()]], -1).flatten(1)
        q = torch.randn((rows, C), device="cuda", generator=g).to(types[fmt])
        return q.view(torch.uint8), q.double()

    (a, va), (b, vb) = operand(I, a_fmt), operand(J, b_fmt)
    kind = {(True, False): lib.FP4_GEMM_F8F6F4_A8, (False, True): lib.FP4_GEMM_F8F6F4_B8, (True, True): lib.FP4_GEMM_F8F6F4_A8B8}[
        (a_fmt != "e2m1", b_fmt != "e2m1")]
    kind |= (lib.binding.FP4_GEMM_A_E5M2 if a_fmt == "e5m2" else 0) | (lib.binding.FP4_GEMM_B_E5M2 if b_fmt == "e5m2" else 0)
    out = torch.full((I, J), float("nan"), device="cuda")
    assert pair_launches(lambda: lib.fp4_gemm(ctx, a, b, gemm_kind=kind, out=out)) == 1
    ctx.status.zero_()
    lib.fp4_gemm(ctx, a, b, gemm_kind=kind, out=out)
    torch.cuda.synchronize()
    assert ctx.read_status() == 0
    err, mag = (out.double() - va @ vb.T).abs(), va.abs() @ vb.abs().T
    assert bool((err <= C / 32 * 2.0 ** -23 * mag).all())


@pytest.mark.parametrize("hot", [0, 100])
def test_pairs_of_ctas_with_a_residual(lib, hot):
    """Pairs with the rows of the weight gradient's compensation and (hot columns) with the forward's dense tail, 63 and 25 row
    blocks: against the codes' products in float64.  The residual's part may differ by the 4e-6 of its summed magnitudes
    that the tensor cores' additions are allowed, or by those of an fp32 sum entry by entry, its entries times 2^-24; the
    two branches are fp32 numbers, four of whose roundings are allowed on top.  The tail is added to the FP4 branch's
    accumulators: 6 blocks of 4 instructions, each of which cuts at most 2^-23 off the running sum."""
    M, K, N, alpha = 8064, 3200, 4096, 0.995
    g = torch.Generator(device="cuda").manual_seed(hot)
    A = torch.randn((M, K), device="cuda", generator=g)
    A[:, :32 * hot:32] *= 20.0
    A, W = A.bfloat16(), (torch.randn((K, N), device="cuda", generator=g) * 0.02).bfloat16()
    dY = (torch.randn((M, N), device="cuda", generator=g) * 1e-3).bfloat16()
    c = lib.Context.for_shape(M, K, N)
    y, sa, sw = lib.fp4_linear_fwd(c, A, W, alpha, out_f32=True)
    dA, dW = lib.fp4_linear_bwd(c, dY, W, sa, sw, out_f32=True, dge_on=False)
    again = [torch.empty_like(t) for t in (y, dA, dW)]
    assert pair_launches(lambda: lib.fp4_linear_fwd(c, A, W, alpha, sa, sw, out=again[0], out_f32=True)) == 1
    assert pair_launches(lambda: lib.fp4_linear_bwd(c, dY, W, sa, sw, out_f32=True, dge_on=False, dA=again[1], dW=again[2])) == 1
    six = torch.tensor(6.0, device="cuda")
    g1 = lib.fp4_quantize(c, dY, 0, prescale=sw.amax / six, codes_t=False)
    g2 = lib.fp4_quantize(c, dY, 1, prescale=sa.amax / six, codes=False)
    torch.cuda.synchronize()
    assert c.read_status() == 0
    hits = sa.csc_colptr.diff()
    assert int((hits >= M // 4).sum()) == hot                                   # the columns of the dense forms
    val = torch.tensor([0, .5, 1, 1.5, 2, 3, 4, 6, 0, -.5, -1, -1.5, -2, -3, -4, -6], dtype=torch.float64, device="cuda")
    dec = lambda c: torch.stack([val[(c & 15).long()], val[(c >> 4).long()]], -1).flatten(1)        # noqa: E731
    lo, hi = sa.thresholds.double().tolist()
    res = A.double() - A.double().clamp(lo, hi)

    def check(got, codes, vectors, residual, dense, entries, cuts=0):
        fp4 = dec(codes[0]) @ dec(codes[1]).T
        for v in vectors:
            fp4 *= v
        comp = residual @ dense if residual is not None else torch.zeros_like(fp4)
        allow = 4 * 2.0 ** -24 * (fp4.abs() + comp.abs()) + cuts * 2.0 ** -23 * fp4.abs()
        if residual is not None:
            allow += torch.maximum(torch.full_like(entries, 4e-6), (entries + 4) * 2.0 ** -24) * (residual.abs() @ dense.abs())
        assert bool(((got.double() - fp4 - comp).abs() <= allow).all())

    d_a, d_w, d_1, d_2 = ((q.amax / six).double() for q in (sa, sw, g1, g2))
    check(y, (sa.codes, sw.codes_t), (d_a[:, None], d_w), res, W.double(), sa.csr_rowptr.diff().double()[:, None],
          cuts=24 if hot else 0)
    check(dA, (g1.codes, sw.codes), (d_1[:, None],), None, None, None)
    check(dW, (sa.codes_t, g2.codes_t), (d_2,), res.T, dY.double(), hits.double()[:, None])
    c.close()


@pytest.mark.parametrize("kind", KINDS)
def test_extreme_codes_long_contraction(lib, ctx, kind):
    """All +-6 operands over the longest contraction of the workloads (16384): |acc| up to 589824."""
    rng = np.random.default_rng(5)
    I, J, C = 128, 128, 16384
    ca = np.where(rng.random((I, C)) < 0.5, 0x7, 0xF).astype(np.uint8)
    cb = np.full((J, C), 0x7, dtype=np.uint8)
    cb[1::2] = 0xF
    ca[0] = 0x7                          # one row with no cancellation at all
    got = _run(lib, ctx, ca, cb, kind).cpu().numpy().astype(np.float64)
    ref = O.gemm_codes(ca, cb)
    assert abs(ref[0, 0]) == 36.0 * C
    np.testing.assert_array_equal(got, ref)


@pytest.mark.parametrize("kind", KINDS)
def test_descales_fp32_and_bf16(lib, ctx, kind):
    rng = np.random.default_rng(9)
    I, J, C = 256, 384, 512
    ca, cb = _codes(rng, I, C), _codes(rng, J, C)
    ra = (rng.random(I) * 4 + 0.1).astype(np.float32)
    cam = (rng.random(J) * 0.1 + 0.01).astype(np.float32)
    acc = O.gemm_codes(ca, cb)
    six = np.float32(6)
    want32 = ((acc.astype(np.float32) * (ra / six)[:, None]).astype(np.float32) * (cam / six)[None, :]).astype(np.float32)
    out = _run(lib, ctx, ca, cb, kind, row_amax=torch.from_numpy(ra).cuda(), col_amax=torch.from_numpy(cam).cuda())
    np.testing.assert_array_equal(out.cpu().numpy(), want32)     # two float multiplies, in this order
    outb = _run(lib, ctx, ca, cb, kind, row_amax=torch.from_numpy(ra).cuda(), col_amax=torch.from_numpy(cam).cuda(),
                out_f32=False)
    wantb = torch.from_numpy(want32).to(torch.bfloat16)
    assert torch.equal(outb.cpu(), wantb)


@pytest.mark.parametrize("kind_name", ["FP4_GEMM_F8F6F4_A8", "FP4_GEMM_F8F6F4_B8", "FP4_GEMM_F8F6F4_A8B8"])
@pytest.mark.parametrize("shape", [(128, 256, 256), (384, 640, 1152), (256, 512, 4096)])
def test_mixed_e4m3_operands(lib, ctx, kind_name, shape):
    """E4M3 bytes as one or both operands of the byte-container kind (the W4A8 / W8A4 settings).
    The products are not all on one binary scale, so the fp32 accumulation is compared at the
    GEMM tolerance of 1e-3 of the summed magnitudes, and is in fact far closer."""
    I, J, C = shape
    kind = getattr(lib, kind_name)
    a8 = kind_name in ("FP4_GEMM_F8F6F4_A8", "FP4_GEMM_F8F6F4_A8B8")
    b8 = kind_name in ("FP4_GEMM_F8F6F4_B8", "FP4_GEMM_F8F6F4_A8B8")
    rng = np.random.default_rng(I + J + C + len(kind_name))

    def fp8(rows):
        c = rng.integers(0, 256, (rows, C), dtype=np.uint8)
        c[(c & 0x7F) == 0x7F] = 0x38                       # no NaN codes
        return c

    ca = fp8(I) if a8 else _codes(rng, I, C)
    cb = fp8(J) if b8 else _codes(rng, J, C)
    va = O.e4m3_decode(ca) if a8 else O.e2m1_decode(ca)
    vb = O.e4m3_decode(cb) if b8 else O.e2m1_decode(cb)
    a = torch.from_numpy(ca if a8 else O.pack_nibbles(ca)).cuda()
    b = torch.from_numpy(cb if b8 else O.pack_nibbles(cb)).cuda()
    ra = (rng.random(I) * 4 + 0.1).astype(np.float32)
    cam = (rng.random(J) * 0.1 + 0.01).astype(np.float32)
    ctx.status.zero_()
    raw = lib.fp4_gemm(ctx, a, b, gemm_kind=kind)
    out = lib.fp4_gemm(ctx, a, b, torch.from_numpy(ra).cuda(), torch.from_numpy(cam).cuda(), gemm_kind=kind)
    torch.cuda.synchronize()
    assert ctx.read_status() == 0
    ref = va @ vb.T
    mag = np.abs(va) @ np.abs(vb).T
    err = np.abs(raw.cpu().numpy().astype(np.float64) - ref)
    assert (err <= 1e-3 * mag).all()
    assert (err <= 2.0 ** -18 * mag).all()                 # what fp32 accumulation of exact products gives
    d_row = (ra / np.float32(448 if a8 else 6)).astype(np.float32)
    d_col = (cam / np.float32(448 if b8 else 6)).astype(np.float32)
    want = (raw.cpu().numpy() * d_row[:, None]).astype(np.float32) * d_col[None, :]
    np.testing.assert_array_equal(out.cpu().numpy(), want.astype(np.float32))   # the two de-scales, in this order


def test_argument_errors(lib, ctx):
    a = torch.zeros((128, 64), dtype=torch.uint8, device="cuda")
    with pytest.raises(lib.Fp4Error) as e:
        lib.fp4_gemm(ctx, a[:100], a)                     # I not a multiple of 128
    assert e.value.code == -2
    with pytest.raises(lib.Fp4Error) as e:
        lib.fp4_gemm(ctx, a, a, gemm_kind=7)
    assert e.value.code == -7


def test_a_wait_that_runs_out_raises_timeout_and_leaves_the_context_usable(lib):
    """Every device-side wait of the GEMM is bounded.  With the debug switches of the library the
    producer of the first CTA leaves out one fill of the shared-memory ring while the limit of the
    waits is 1 ms: the consumer's wait runs out, the kernel raises FP4_DEV_TIMEOUT, frees its tensor
    memory and returns; the next GEMM on the same context is exact again."""
    rng = np.random.default_rng(77)
    ca, cb = _codes(rng, 256, 4096), _codes(rng, 256, 4096)          # 16 fills per tile (MXF4), 32 (byte containers)
    want = O.gemm_codes(ca, cb)
    a = torch.from_numpy(O.pack_nibbles(ca)).cuda()
    b = torch.from_numpy(O.pack_nibbles(cb)).cuda()
    c = lib.Context(0, 64 << 20)
    for kind in KINDS:
        c.debug_set(lib.binding.FP4_DEBUG_WAIT_LIMIT_US, 1000)
        c.debug_set(lib.binding.FP4_DEBUG_SKIP_FILL, 6)
        c.status.zero_()
        lib.fp4_gemm(c, a, b, gemm_kind=kind)
        torch.cuda.synchronize()                                       # the kernel returned
        assert c.read_status() & lib.FP4_DEV_TIMEOUT
        c.debug_set(lib.binding.FP4_DEBUG_SKIP_FILL, -1)
        c.debug_set(lib.binding.FP4_DEBUG_WAIT_LIMIT_US, 0)
        c.status.zero_()
        out = lib.fp4_gemm(c, a, b, gemm_kind=kind)
        torch.cuda.synchronize()
        assert c.read_status() == 0
        np.testing.assert_array_equal(out.cpu().numpy().astype(np.float64), want)
    c.close()
