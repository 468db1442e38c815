"""The bounded device-side waits, made to run out without any fault.

Every wait of the convolution kernels (on an mbarrier, or of a split weight gradient on its sibling CTAs) has a time
limit; when it runs out the CTA records the time-out, drains its copies, frees its tensor memory and exits, and
pt_poll_device_status returns PT_ERR_TIMEOUT. The tests shorten the limit to a few milliseconds, make ONE tiny launch
leave out one arrival through the library's test hook (no trap, no bad address, no unbounded loop), and check the
status, the time it took, and that the next ordinary launches on the same context -- which need the SMs' whole tensor
memory and, for the weight gradient, the same arrival counters -- still match the oracle.
"""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_1901_09290_b200 import binding as B
from paper_1901_09290_b200 import workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu

LIMIT_MS = 20


def _inputs(N, H, C, K, R, seed):
    x = W.gen_act(N, H, H, C, seed)
    w = W.bf16_round(W.gen_weight(K, R, R, C, seed + 1))
    dy = W.gen_dy(N, H, H, K, seed + 2)
    return x, w, dy


def _expect_timeout(ctx, launch):
    B.pt_test_set_wait_limit(ctx, LIMIT_MS)
    try:
        t0 = time.perf_counter()
        launch()
        with pytest.raises(B.PtError) as e:
            ctx.poll()
        dt = time.perf_counter() - t0
        assert e.value.status == 5, e.value                     # PT_ERR_TIMEOUT
        assert dt < 2.0, f"the wait took {dt:.2f} s to give up at a {LIMIT_MS} ms limit"
    finally:
        B.pt_test_skip_next_arrive(ctx, 0)
        B.pt_test_set_wait_limit(ctx, 0)
    ctx.poll()                                                  # the status word was cleared by the failing poll


def test_split_weight_gradient_wait_runs_out_and_the_context_recovers():
    ctx = Hh.ctx()
    N, H, C, K, R = 8, 16, 16, 32, 3                            # config-1 size
    x, w, dy = _inputs(N, H, C, K, R, W.BASE_SEED + 61)
    d = B.make_conv_desc(N, H, H, C, K, R, R, 1, 1, algo=2)
    ctas, waits = B.pt_conv_wgrad_ctas(ctx, d)
    assert waits and ctas > 1, "the shape must split its reduction over CTAs for this test"
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    dw = torch.zeros((K, R, R, C), dtype=torch.float32, device="cuda")
    ws = Hh.conv_ws(d, B.PT_CONV_WGRAD)

    def launch():
        B.pt_test_skip_next_arrive(ctx, 1)
        B.pt_conv_wgrad(ctx, d, xd, dyd, dw, ws)

    _expect_timeout(ctx, launch)
    # the same split launch again (same counters after the reset), several times, and a launch that takes all 512 TMEM
    # columns on every SM: a CTA that had kept its tensor memory would make these wait for ever (they are bounded too)
    ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, 1, 1)
    for _ in range(3):
        dw.fill_(7680.0)
        B.pt_conv_wgrad(ctx, d, xd, dyd, dw, ws)
        torch.cuda.synchronize()
        ctx.poll()
        Hh.check_conv(dw, C, ref, what="wgrad after a time-out")
    xb, wb, dyb = _inputs(4, 28, 256, 256, 1, W.BASE_SEED + 62)
    y, dx, dwb, _ = Hh.run_conv_all(4, 28, 28, 256, 256, 1, 1, 0, xb, wb, dyb, algo=2)
    Hh.check_conv(y, 256, oracle.conv_fwd(xb.numpy(), wb.numpy(), 1, 0), what="fwd after a time-out")
    Hh.check_conv(dwb, 256, oracle.conv_wgrad(xb.numpy(), dyb.numpy(), 1, 1, 1, 0), what="wide wgrad after a time-out")


# the forms that other layers choose: filter rows at both strides, packed rows, rows of blocks
@pytest.mark.parametrize("form,N,H,C,K,stride,ld", [("TAPS", 6, 14, 70, 40, 1, 8), ("TAPS", 6, 15, 20, 130, 2, 8), ("PACKED", 8, 16, 13, 27, 1, 16), ("ROWS", 8, 16, 40, 27, 1, 8),
                                                    ("PIXELS", 8, 16, 40, 27, 1, 8)])
def test_every_form_of_the_weight_gradient_gives_up_and_recovers(form, N, H, C, K, stride, ld):
    ctx = Hh.ctx()
    P = (H + 2 - 3) // stride + 1
    x, dy = W.gen_act(N, H, H, C, W.BASE_SEED + 69), W.gen_dy(N, P, P, K, W.BASE_SEED + 70)
    up = lambda n: -(-n // ld) * ld
    d = B.make_conv_desc(N, H, H, C, K, 3, 3, stride, 1, up(C), up(K), algo=2)
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    want = getattr(B, "PT_FORM_WGRAD_" + form)
    B.pt_test_form(ctx, want)
    try:
        ctas, waits = B.pt_conv_wgrad_ctas(ctx, d)
        assert waits and ctas > 1
        dw = torch.zeros((K, 3, 3, C), dtype=torch.float32, device="cuda")
        ws = Hh.conv_ws(d, B.PT_CONV_WGRAD)

        def launch():
            B.pt_test_skip_next_arrive(ctx, 1)
            B.pt_conv_wgrad(ctx, d, xd, dyd, dw, ws)

        _expect_timeout(ctx, launch)
        ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), 3, 3, stride, 1)
        for _ in range(3):
            dw.fill_(7680.0)
            B.pt_conv_wgrad(ctx, d, xd, dyd, dw, ws)
            torch.cuda.synchronize()
            ctx.poll()
            assert B.pt_test_last_form(ctx) == want
            Hh.check_conv(dw, C, ref, what="wgrad after a time-out")
    finally:
        B.pt_test_form(ctx, B.PT_FORM_ANY)


# one and two accumulators an issuer, with and without statistics; a CTA of one output row and of several
@pytest.mark.parametrize("N,H,K,stats", [(2, 128, 20, False), (12, 128, 90, True)])
def test_stem_wait_runs_out_and_the_context_recovers(N, H, K, stats):
    ctx = Hh.ctx()
    x, w = W.gen_act(N, H, H, 3, W.BASE_SEED + 71), W.bf16_round(W.gen_weight(K, 7, 7, 3, W.BASE_SEED + 72))
    d = B.make_conv_desc(N, H, H, 3, K, 7, 7, 2, 3, algo=2)
    xd, wd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(w, d.ldw)
    y = torch.zeros((N, H // 2, H // 2, d.ldy), dtype=torch.bfloat16, device="cuda")
    ws = Hh.conv_ws(d, B.PT_CONV_FWD)
    st = torch.empty(B.pt_conv_fwd_stats_bytes(ctx, d) // 4, device="cuda")
    run = lambda out: B.pt_conv_fwd_stats(ctx, d, xd, wd, out, st, ws) if stats else B.pt_conv_fwd(ctx, d, xd, wd, out, ws)

    def launch():
        B.pt_test_skip_next_arrive(ctx, 6)
        run(y)

    _expect_timeout(ctx, launch)
    ref = oracle.conv_fwd(x.numpy(), w.numpy(), 2, 3)
    for _ in range(3):
        yo = Hh.out_buffer((N, H // 2, H // 2), K, d.ldy, False)
        run(yo)
        torch.cuda.synchronize()
        ctx.poll()
        assert B.pt_test_last_form(ctx) == B.PT_FORM_STEM
        Hh.check_conv(yo, K, ref, what="stem after a time-out")
    # a launch that takes all 512 columns of every SM's tensor memory
    xb, wb, dyb = _inputs(4, 28, 256, 256, 1, W.BASE_SEED + 73)
    dwb = Hh.run_conv_all(4, 28, 28, 256, 256, 1, 1, 0, xb, wb, dyb, algo=2)[2]
    Hh.check_conv(dwb, 256, oracle.conv_wgrad(xb.numpy(), dyb.numpy(), 1, 1, 1, 0), what="wide wgrad after a time-out")


def test_pipeline_barrier_wait_runs_out_and_the_context_recovers():
    ctx = Hh.ctx()
    N, H, C, K, R = 8, 16, 16, 32, 1                            # a 1x1 layer: the pixel-linear kernel
    x, w, dy = _inputs(N, H, C, K, R, W.BASE_SEED + 63)
    d = B.make_conv_desc(N, H, H, C, K, R, R, 1, 0, algo=2)
    xd, wd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(w, d.ldw)
    y = torch.zeros((N, H, H, d.ldy), dtype=torch.bfloat16, device="cuda")

    def launch():
        B.pt_test_skip_next_arrive(ctx, 2)
        B.pt_conv_fwd(ctx, d, xd, wd, y, None)

    _expect_timeout(ctx, launch)
    ref = oracle.conv_fwd(x.numpy(), w.numpy(), 1, 0)
    for _ in range(3):
        yo = Hh.out_buffer((N, H, H), K, d.ldy, False)
        B.pt_conv_fwd(ctx, d, xd, wd, yo, None)
        torch.cuda.synchronize()
        ctx.poll()
        Hh.check_conv(yo, K, ref, what="fwd after a time-out")


def test_halo_pipeline_wait_runs_out_and_the_context_recovers():
    ctx = Hh.ctx()
    N, H, C, K, R = 8, 16, 72, 40, 3                            # two chunks per tile, a producer warp per ring
    x, w, dy = _inputs(N, H, C, K, R, W.BASE_SEED + 65)
    d = B.make_conv_desc(N, H, H, C, K, R, R, 1, 1, algo=2)
    xd, wd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(w, d.ldw)
    y = torch.zeros((N, H, H, d.ldy), dtype=torch.bfloat16, device="cuda")

    def launch():
        B.pt_test_skip_next_arrive(ctx, 5)
        B.pt_conv_fwd(ctx, d, xd, wd, y, None)

    _expect_timeout(ctx, launch)
    ref = oracle.conv_fwd(x.numpy(), w.numpy(), 1, 1)
    for _ in range(3):
        yo = Hh.out_buffer((N, H, H), K, d.ldy, False)
        B.pt_conv_fwd(ctx, d, xd, wd, yo, None)
        torch.cuda.synchronize()
        ctx.poll()
        Hh.check_conv(yo, K, ref, what="fwd after a time-out")


@pytest.mark.parametrize("C", [24, 371])                        # whole rows by bulk copies; channel slabs by TMA boxes
def test_batch_norm_wait_runs_out_and_the_context_recovers(C):
    ctx = Hh.ctx()
    N, H, ld = 32, 28, W.pad8(C)
    gen = torch.Generator(device="cuda").manual_seed(W.BASE_SEED + 66)
    x = torch.randn((N, H, H, ld), generator=gen, device="cuda").to(torch.bfloat16)
    g, b, sm, si = torch.ones(C, device="cuda"), torch.zeros(C, device="cuda"), torch.empty(C, device="cuda"), torch.empty(C, device="cuda")
    y, again = torch.zeros_like(x), torch.zeros_like(x)
    d = B.make_bn_desc(N, H, H, C, ld)
    ws = torch.empty(B.pt_bn_workspace_bytes(ctx, d), dtype=torch.uint8, device="cuda")
    run = lambda out: B.pt_bn_relu_fwd(ctx, d, x, None, g, b, None, None, sm, si, out, ws)
    run(y)

    def launch():
        B.pt_test_skip_next_arrive(ctx, 3)
        run(again)

    _expect_timeout(ctx, launch)
    for _ in range(3):
        run(again)
        torch.cuda.synchronize()
        ctx.poll()
        assert torch.equal(y, again)


def test_channel_gate_wait_runs_out_and_the_context_recovers():
    ctx = Hh.ctx()
    npix, C, S = 50000, 222, 211
    gen = torch.Generator(device="cuda").manual_seed(W.BASE_SEED + 67)
    ld, lds = W.pad8(C), W.pad8(S)
    node = torch.randn((npix, ld), generator=gen, device="cuda").to(torch.bfloat16)
    idx = torch.randperm(C, generator=gen, device="cuda")[:S].to(torch.int32)
    out = torch.zeros((npix, lds), dtype=torch.bfloat16, device="cuda")

    def launch():
        B.pt_test_skip_next_arrive(ctx, 4)
        B.pt_channel_gather(ctx, node, ld, C, idx, S, out, lds, npix)

    _expect_timeout(ctx, launch)
    for _ in range(3):
        B.pt_channel_gather(ctx, node, ld, C, idx, S, out, lds, npix)
        torch.cuda.synchronize()
        ctx.poll()
        assert torch.equal(out[:, :S], node[:, idx.long()])


def test_regulariser_value_does_not_depend_on_an_unpolled_time_out():
    """A weight gradient that gave up leaves its arrival counters behind until the status is polled: nothing else may count with them,
    however many launches have gone round the ring of counters meanwhile."""
    ctx = B.Context(0)                                          # a ring of its own
    N, H, C, K, R = 8, 16, 16, 32, 3
    x, w, dy = _inputs(N, H, C, K, R, W.BASE_SEED + 68)
    d = B.make_conv_desc(N, H, H, C, K, R, R, 1, 1, algo=2)
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    dw = torch.zeros((K, R, R, C), device="cuda")
    ws = torch.empty(B.pt_conv_workspace_bytes(ctx, d, B.PT_CONV_WGRAD), dtype=torch.uint8, device="cuda")
    wt, sq_o, sq_i = w.cuda().contiguous(), torch.zeros(K, device="cuda"), torch.zeros(C, device="cuda")
    v = torch.zeros_like(wt)
    arr = B.layer_array([B.make_layer(wt, dw, v, None, K, C, R * R, d.ldw, True, True, sq_o, sq_i, None, None)])
    lws = torch.empty(max(256, B.pt_group_lasso_workspace_bytes(ctx, arr)), dtype=torch.uint8, device="cuda")
    reg = torch.zeros(1, dtype=torch.float64, device="cuda")
    B.pt_test_set_wait_limit(ctx, LIMIT_MS)
    try:
        B.pt_test_skip_next_arrive(ctx, 1)
        B.pt_conv_wgrad(ctx, d, xd, dyd, dw, ws)
        torch.cuda.synchronize()
        bad = torch.zeros((), dtype=torch.int64, device="cuda")
        B.pt_group_lasso_norms(ctx, arr, reg, lws)
        ref = reg.clone()
        for _ in range(16500):                                  # (the ring has 16384 counters)
            reg.fill_(-1.0)
            B.pt_group_lasso_norms(ctx, arr, reg, lws)
            bad += (reg != ref).sum()
        assert int(bad) == 0
        with pytest.raises(B.PtError):
            ctx.poll()
    finally:
        B.pt_test_set_wait_limit(ctx, 0)
        ctx.close()
