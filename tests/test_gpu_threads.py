"""Host threads that share a context take turns: calls of several threads on one stream give what the same calls of
one thread give, while graphs are captured, settings switched and host-buffer steps pipelined in between."""
import threading

import numpy as np
import pytest
import torch

from paper_2501_17116_b200 import workloads as WL

pytestmark = pytest.mark.gpu


def _bf16(bits):
    return torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16)


def _together(*work):
    """Runs the functions in a thread each, started at once; raises what any of them raised."""
    gate, failed = threading.Barrier(len(work)), []

    def body(f):
        try:
            torch.cuda.set_device(0)
            gate.wait(timeout=60)
            f()
        except BaseException as e:                   # noqa: BLE001
            failed.append(e)

    threads = [threading.Thread(target=body, args=(f,)) for f in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join(timeout=240)
    assert not any(t.is_alive() for t in threads)
    if failed:
        raise failed[0]


def test_layers_of_several_threads(lib):
    """Three threads, a layer each, thirty steps on one context and one stream."""
    shapes, alpha, steps = [(256, 384, 640), (128, 512, 256), (512, 256, 384)], 0.99, 30
    ctx = lib.Context(0, max(int(lib.load_library().fp4_workspace_bytes(*s)) for s in shapes))
    layers, want = [], []
    for i, (M, K, N) in enumerate(shapes):
        A, W, dY = (_bf16(b).cuda() for b in WL.small_case(M, K, N, seed=60 + i))
        sa, sw = lib.QTensor(M, K, 0, "cuda", lib.tail_capacity(M, K, alpha)), lib.QTensor(K, N, 1, "cuda")
        outs = [[torch.empty(s, dtype=torch.bfloat16, device="cuda") for s in ((M, N), (M, K), (K, N))] for _ in range(steps)]
        one = lib.Context.for_shape(M, K, N)
        y, _, _ = lib.fp4_linear_fwd(one, A, W, alpha, saved_a=sa, saved_w=sw)
        da, dw = lib.fp4_linear_bwd(one, dY, W, sa, sw)
        torch.cuda.synchronize()
        one.close()
        want.append((y, da, dw))
        layers.append((A, W, dY, sa, sw, outs))

    def steps_of(A, W, dY, sa, sw, outs):
        def run():
            for i, (y, da, dw) in enumerate(outs):
                if i % 3 == 0:                       # outputs of their own: never captured
                    lib.fp4_linear_fwd(ctx, A, W, alpha, saved_a=sa, saved_w=sw, out=y)
                    lib.fp4_linear_bwd(ctx, dY, W, sa, sw, dA=da, dW=dw)
                else:                                # the same outputs again and again: captured, then replayed
                    lib.fp4_linear_fwd(ctx, A, W, alpha, saved_a=sa, saved_w=sw, out=outs[1][0])
                    lib.fp4_linear_bwd(ctx, dY, W, sa, sw, dA=outs[1][1], dW=outs[1][2])
        return run

    _together(*(steps_of(*layer) for layer in layers))
    torch.cuda.synchronize()
    assert ctx.read_status() == 0
    for (*_, outs), wanted in zip(layers, want):
        for i in [1] + list(range(0, steps, 3)):
            for got, w in zip(outs[i], wanted):
                assert torch.equal(got, w), i
    ctx.close()


def test_host_steps_of_two_threads(lib):
    """Two threads send host-buffer steps of different shapes into one context."""
    shapes, alpha, steps = [(256, 256, 384), (128, 512, 128)], 0.99, 20
    library = lib.load_library()
    ctx = lib.Context(0, max(int(library.fp4_step_host_workspace_bytes(M, K, N, alpha)) for M, K, N in shapes))
    jobs = []
    for i, (M, K, N) in enumerate(shapes):
        ins = [_bf16(b).pin_memory() for b in WL.small_case(M, K, N, seed=80 + i)]
        outs = [[torch.empty(s, dtype=torch.bfloat16).pin_memory() for s in ((M, N), (M, K), (K, N))] for _ in range(steps + 1)]
        lib.fp4_linear_step_host(ctx, *ins, alpha, *outs[-1])
        jobs.append((ins, outs))

    def steps_of(ins, outs):
        def run():
            for i, o in enumerate(outs[:-1]):
                assert lib.fp4_linear_step_host(ctx, *ins, alpha, *o, read_status=i % 4 == 0) == 0
        return run

    _together(*(steps_of(*job) for job in jobs))
    torch.cuda.synchronize()
    for _, outs in jobs:
        for o in outs[:-1]:
            for got, want in zip(o, outs[-1]):
                assert torch.equal(got.view(torch.int16), want.view(torch.int16))
    ctx.close()


def test_a_setting_switched_by_another_thread(lib):
    """One thread quantises the same tensor over and over while another switches the form of the clamp: every result
    is that of one form, and what is replayed afterwards is the form that is set."""
    M, K, alpha = 256, 512, 0.97
    x = _bf16(WL.small_case(M, K, 128, seed=3)[0]).cuda()
    forms = (lib.FP4_QUANTILE_SIGNED, lib.FP4_QUANTILE_ABS)
    ctx = lib.Context.for_shape(M, K, 128)
    want = []
    for form in forms:
        one = lib.Context.for_shape(M, K, 128)
        one.set_quantile_mode(form)
        want.append(lib.fp4_quantize(one, x, 0, alpha=alpha).thresholds.clone())
        torch.cuda.synchronize()
        one.close()
    assert not torch.equal(*want)
    q, seen, stop = lib.QTensor(M, K, 0, "cuda", lib.tail_capacity(M, K, alpha)), [], threading.Event()

    def quantise():
        try:
            for _ in range(300):
                lib.fp4_quantize(ctx, x, 0, alpha=alpha, out=q)
                seen.append(q.thresholds.clone())
        finally:
            stop.set()

    def switch():
        while not stop.is_set():
            for form in forms:
                ctx.set_quantile_mode(form)

    _together(quantise, switch)
    torch.cuda.synchronize()
    assert all(any(torch.equal(s, w) for w in want) for s in seen)
    for form, w in list(zip(forms, want)) * 3:
        ctx.set_quantile_mode(form)
        for _ in range(2):
            lib.fp4_quantize(ctx, x, 0, alpha=alpha, out=q)
            assert torch.equal(q.thresholds, w)
    assert ctx.read_status() == 0
    ctx.close()
