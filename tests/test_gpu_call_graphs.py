"""Repeated calls are replayed as CUDA graphs inside the library: a replay must do what plain launches do
(a context in profiling mode enqueues every call), on whatever the buffers hold at that time."""
import time

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


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("M,K,N,alpha", [(128, 128, 128, 1.0), (256, 384, 640, 0.99), (1024, 512, 384, 0.97)])
def test_replays_follow_the_buffers(lib, M, K, N, alpha, own_stream):
    """Steps over the same buffers with new contents each, on the legacy stream and on one of the caller's.  Every
    setting comes five times in a row, so that its calls are captured and replayed, and then again after others:
    the weight quantised or kept, the form of the clamp (a replay of the other form would show), the side streams."""
    stream = torch.cuda.Stream() if own_stream else torch.cuda.default_stream()
    fast, plain = (lib.Context.for_shape(M, K, N) for _ in range(2))
    plain.profile_enable()
    cap = lib.tail_capacity(M, K, alpha)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    A, W, dY = torch.empty((M, K), **bf), torch.empty((K, N), **bf), torch.empty((M, N), **bf)
    bufs = [(lib.QTensor(M, K, 0, "cuda", cap), lib.QTensor(K, N, 1, "cuda"), torch.empty((M, N), **bf),
             torch.empty((M, K), **bf), torch.empty((K, N), **bf)) for _ in range(2)]
    torch.cuda.synchronize()
    signed, magnitude = lib.FP4_QUANTILE_SIGNED, lib.FP4_QUANTILE_ABS
    settings = [(signed, False, True), (magnitude, False, True), (signed, True, True), (signed, False, False),
                (magnitude, True, False), (signed, False, True), (magnitude, False, True)]
    step = 0
    with torch.cuda.stream(stream):
        for mode, reuse_w, overlap in settings:
            for _ in range(5):
                step += 1
                a, w, dy = WL.small_case(M, K, N, seed=step)
                A.copy_(_dev(a))
                dY.copy_(_dev(dy))
                if not reuse_w:
                    W.copy_(_dev(w))
                counts = []
                for c, (sa, sw, y, da, dw) in zip((fast, plain), bufs):
                    c.set_quantile_mode(mode)
                    c.set_overlap(overlap)
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


def test_many_calls_with_outputs_of_their_own(lib):
    """700 calls with outputs of their own, each repeated often enough to be captured, then again in
    another order."""
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


def test_a_cycle_of_more_calls_than_a_context_remembers(lib):
    """1200 different calls (by alpha, on the same buffers) that come round again and again: most are replayed, seen by
    the host time of a call beside that of calls that never came before.  Later the calls change for good: the old
    graphs leave, the new ones take their place, and the results are still those of the call that was made last."""
    M = 128
    ctx = lib.Context.for_shape(M, M, M)
    a, w, _ = WL.small_case(M, M, M, seed=5)
    A, W = _dev(a), _dev(w)
    y = torch.empty((M, M), dtype=torch.bfloat16, device="cuda")
    sa, sw = lib.QTensor(M, M, 0, "cuda", lib.tail_capacity(M, M, 0.9)), lib.QTensor(M, M, 1, "cuda")

    def host_us(alphas):
        """Host time per call: batches that the launch queue holds, the GPU idle before each."""
        t = 0.0
        for i in range(0, len(alphas), 40):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for al in alphas[i:i + 40]:
                lib.fp4_linear_fwd(ctx, A, W, al, saved_a=sa, saved_w=sw, out=y)
            t += time.perf_counter() - t0
        return 1e6 * t / len(alphas)

    cycle = [0.99 - 1e-9 * i for i in range(1200)]
    for _ in range(4):
        host_us(cycle)
    again, new = host_us(cycle), host_us([0.98 - 1e-9 * i for i in range(400)])
    assert again < 0.7 * new, (again, new)
    other = [0.97 - 1e-9 * i for i in range(1200)]
    for _ in range(8):
        host_us(other)
    assert host_us(other) < 0.7 * new
    for al in (0.99, 0.97, 0.9, 0.97):
        lib.fp4_linear_fwd(ctx, A, W, al, saved_a=sa, saved_w=sw, out=y)
        want, _, _ = lib.fp4_linear_fwd(ctx, A, W, al)
        assert torch.equal(y, want)
    assert ctx.read_status() == 0
    ctx.close()
