"""Repeated calls are replayed as CUDA graphs inside the library: a replay must do what plain launches do
(a context in profiling mode enqueues every call), on whatever the buffers hold at that time."""
import numpy as np
import pytest
import torch

from paper_2501_17116_b200 import workloads as WL

pytestmark = pytest.mark.gpu


def _dev(bits):
    return torch.from_numpy(bits.view(np.int16)).cuda().view(torch.bfloat16)


def _layer(lib, ctx, A, W, dY, alpha, sa, sw, y, da, dw, reuse_w):
    lib.fp4_linear_fwd(ctx, A, W, alpha, saved_a=sa, saved_w=sw, reuse_w=reuse_w, out=y)
    lib.fp4_linear_bwd(ctx, dY, W, sa, sw, dA=da, dW=dw)


@pytest.mark.parametrize("M,K,N,alpha", [(128, 128, 128, 1.0), (256, 384, 640, 0.99), (1024, 512, 384, 0.97)])
def test_replays_follow_the_buffers(lib, M, K, N, alpha):
    """Ten steps over the same buffers with new contents each: weights kept on two of three, overlap and the
    form of the quantile switched on the way."""
    fast, plain = (lib.Context.for_shape(M, K, N) for _ in range(2))
    plain.profile_enable()
    cap = lib.tail_capacity(M, K, alpha)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    A, W, dY = torch.empty((M, K), **bf), torch.empty((K, N), **bf), torch.empty((M, N), **bf)
    bufs = [(lib.QTensor(M, K, 0, "cuda", cap), lib.QTensor(K, N, 1, "cuda"), torch.empty((M, N), **bf),
             torch.empty((M, K), **bf), torch.empty((K, N), **bf)) for _ in range(2)]
    for step in range(10):
        a, w, dy = WL.small_case(M, K, N, seed=step)
        A.copy_(_dev(a))
        dY.copy_(_dev(dy))
        reuse_w = step % 3 != 0
        if not reuse_w:
            W.copy_(_dev(w))
        mode = lib.FP4_QUANTILE_ABS if step in (6, 9) else lib.FP4_QUANTILE_SIGNED
        counts = []
        for c, (sa, sw, y, da, dw) in zip((fast, plain), bufs):
            c.set_quantile_mode(mode)
            c.set_overlap(step != 7)
            before = c.launch_count()
            _layer(lib, c, A, W, dY, alpha, sa, sw, y, da, dw, reuse_w)
            counts.append(c.launch_count() - before)
        torch.cuda.synchronize()
        assert fast.read_status() == plain.read_status() == 0
        assert counts[0] == counts[1] > 0
        for got, want in zip(bufs[0][2:], bufs[1][2:]):
            assert torch.equal(got, want), step
        for name in ("codes", "codes_t", "amax"):
            assert torch.equal(getattr(bufs[0][0], name), getattr(bufs[1][0], name)), (step, name)
    fast.close()
    plain.close()


def test_more_calls_than_a_context_remembers(lib):
    """700 calls with outputs of their own, each repeated often enough to be captured, then again in
    another order: graphs leave and come back while the stream is busy."""
    ctx = lib.Context.for_shape(128, 256, 128)
    x = _dev(WL.small_case(128, 256, 128, seed=5)[0])
    want = lib.fp4_quantize(ctx, x, 0, alpha=0.99)
    outs = [lib.QTensor(128, 256, 0, "cuda", want.sparse_cap) for _ in range(700)]
    for _ in range(2):
        for q in outs:
            for _ in range(4):
                lib.fp4_quantize(ctx, x, 0, alpha=0.99, out=q)
    for q in outs:
        q.codes.zero_()
        q.csc_val.zero_()
    for q in reversed(outs):
        lib.fp4_quantize(ctx, x, 0, alpha=0.99, out=q)
    torch.cuda.synchronize()
    assert ctx.read_status() == 0
    for q in outs:
        assert torch.equal(q.codes, want.codes) and torch.equal(q.csc_val, want.csc_val)
    ctx.close()
