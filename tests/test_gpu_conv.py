"""Parity of the CUDA convolutions (through the C ABI) with the fp64 oracle on the same seeded inputs."""
import numpy as np
import pytest
import torch

import oracle
from paper_1901_09290_b200 import binding as B
from paper_1901_09290_b200 import workloads as W
from tests import helpers as Hh

pytestmark = pytest.mark.gpu

ALGOS = [0, 1]

# (N, H, W, C, K, R, stride)  -- odd and tiny channel counts, ragged pixel tails, stride 2, 7x7
SMALL = [
    (2, 5, 7, 1, 1, 1, 1), (2, 5, 7, 3, 7, 3, 1), (1, 1, 1, 8, 11, 1, 1), (3, 16, 16, 11, 27, 3, 1),
    (2, 16, 16, 16, 16, 1, 1), (2, 9, 9, 27, 8, 3, 2), (2, 8, 8, 7, 93, 1, 2), (1, 23, 23, 3, 16, 7, 2),
    (2, 14, 14, 93, 77, 3, 1), (1, 12, 10, 130, 70, 1, 1), (1, 7, 7, 260, 300, 3, 1),
    # few-channel stride-2 stems (space-to-depth path): 7x7, 5x5, 3x3; C = 1, 3, 4; non-square image
    (2, 32, 32, 3, 16, 7, 2), (1, 16, 20, 3, 55, 7, 2), (2, 12, 12, 1, 9, 5, 2), (2, 16, 16, 4, 24, 3, 2),
]


def _case(N, H, Wd, C, K, R, stride, seed):
    pad = R // 2
    x = W.gen_act(N, H, Wd, C, seed)
    w = W.bf16_round(W.gen_weight(K, R, R, C, seed + 1))
    P, Q = (H + 2 * pad - R) // stride + 1, (Wd + 2 * pad - R) // stride + 1
    dy = W.gen_dy(N, P, Q, K, seed + 2)
    return x, w, dy, pad


@pytest.mark.parametrize("algo", ALGOS)
@pytest.mark.parametrize("shape", SMALL)
def test_small_and_odd_shapes(shape, algo):
    N, H, Wd, C, K, R, stride = shape
    x, w, dy, pad = _case(*shape, seed=W.BASE_SEED + 11)
    y32, dx32, dw, _ = Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=algo, out_f32=1)
    y16, dx16, dw2, _ = Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=algo, out_f32=0)
    yr = oracle.conv_fwd(x.numpy(), w.numpy(), stride, pad)
    dxr = oracle.conv_dgrad(dy.numpy(), w.numpy(), H, Wd, stride, pad)
    Hh.check_conv(y32, K, yr, what="fwd f32")
    Hh.check_conv(dx32, C, dxr, what="dgrad f32")
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad), what="wgrad")
    Hh.check_conv(y16, K, yr, what="fwd bf16")
    Hh.check_conv(dx16, C, dxr, what="dgrad bf16")
    # the bf16 output is the fp32 result rounded to nearest even, nothing else
    assert torch.equal(y16[..., :K], y32[..., :K].to(torch.bfloat16))
    assert torch.equal(dx16[..., :C], dx32[..., :C].to(torch.bfloat16))
    assert torch.equal(dw, dw2)


@pytest.mark.parametrize("algo", ALGOS)
def test_config1_single_layer_with_zero_groups(algo):
    """Batch 8, 16->32 channels, 16x16, 3x3: zero input channels / zero upstream-gradient channels give
    exactly-zero weight-gradient columns / rows (Eq. 4)."""
    N, H, C, K, R = 8, 16, 16, 32, 3
    seed = W.BASE_SEED + 1
    g = np.random.default_rng(seed)
    kz, cz = np.sort(g.permutation(K)[:5]), np.sort(g.permutation(C)[:3])
    x, w, dy, pad = _case(N, H, H, C, K, R, 1, seed)
    x[..., cz] = 0
    dy[..., kz] = 0
    w[kz] = 0
    w[:, :, :, cz] = 0
    y, dx, dw, _ = Hh.run_conv_all(N, H, H, C, K, R, 1, pad, x, w, dy, algo=algo)
    Hh.check_conv(y, K, oracle.conv_fwd(x.numpy(), w.numpy(), 1, pad), what="fwd")
    Hh.check_conv(dx, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, H, 1, pad), what="dgrad")
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, 1, pad), what="wgrad")
    dwc = dw.cpu()
    assert torch.all(dwc[kz] == 0) and torch.all(dwc[:, :, :, cz] == 0)
    assert torch.all(y.float().cpu()[..., kz] == 0) and torch.all(dx.float().cpu()[..., cz] == 0)


@pytest.mark.parametrize("algo", ALGOS)
def test_config3_pruned_bottleneck(algo):
    """ResNet-50 stage-3 bottleneck at batch 64, 28x28, pruned to 371 -> 93 -> 77 -> 371: full-tensor parity."""
    net = W.with_sizes(W.bottleneck_stage3(), [371, 93, 77])
    for li, l in enumerate(net.layers):
        seed = W.layer_seed(3, li)
        x, w, dy, pad = _case(64, l.H, l.H, l.C, l.K, l.R, l.stride, seed)
        y, dx, dw, _ = Hh.run_conv_all(64, l.H, l.H, l.C, l.K, l.R, l.stride, pad, x, w, dy, algo=algo)
        Hh.check_conv(y, l.K, oracle.conv_fwd(x.numpy(), w.numpy(), l.stride, pad), what=l.name + " fwd")
        Hh.check_conv(dx, l.C, oracle.conv_dgrad(dy.numpy(), w.numpy(), l.H, l.H, l.stride, pad), what=l.name + " dgrad")
        Hh.check_conv(dw, l.C, oracle.conv_wgrad(x.numpy(), dy.numpy(), l.R, l.R, l.stride, pad), what=l.name + " wgrad")


# (N, H, W, C, K, R, extra pitch of y) of the stem's kernel that reads the image itself: the narrowest and widest rows, every channel count, 3x3
# to 7x7 filters, one and two 64-channel chunks, one and two accumulators an issuer, CTAs of one and several output rows, of several images
@pytest.mark.parametrize("shape", [(2, 6, 128, 3, 16, 7, 0), (1, 2, 250, 1, 9, 3, 8), (3, 10, 200, 4, 65, 5, 0), (30, 42, 130, 2, 128, 3, 0), (31, 22, 160, 3, 55, 7, 8),
                                   (200, 2, 224, 3, 20, 7, 0), (2, 224, 224, 3, 70, 7, 0)])
def test_stem_straight_from_the_image(shape):
    N, H, Wd, C, K, R, ey = shape
    x, w, _, pad = _case(N, H, Wd, C, K, R, 2, seed=W.BASE_SEED + 47)
    d = B.make_conv_desc(N, H, Wd, C, K, R, R, 2, pad, 8, W.pad8(K) + ey, W.pad8(C), 0, 2)
    P, Q = (H + 2 * pad - R) // 2 + 1, (Wd + 2 * pad - R) // 2 + 1
    xd, wd = Hh.to_dev_padded(x, 8), Hh.to_dev_padded(w, d.ldw)
    y, y2 = Hh.out_buffer((N, P, Q), K, d.ldy, 0), Hh.out_buffer((N, P, Q), K, d.ldy, 0)
    c = B.Context(0)
    before = c.launch_count()
    B.pt_conv_fwd(c, d, xd, wd, y, Hh.conv_ws(d, B.PT_CONV_FWD))
    assert c.launch_count() == before + 1                        # (the space-to-depth copy would be two launches more)
    stats = torch.full((B.pt_conv_fwd_stats_bytes(c, d) // 4,), float("nan"), device="cuda")
    parts = B.pt_conv_fwd_stats(c, d, xd, wd, y2, stats, Hh.conv_ws(d, B.PT_CONV_FWD))
    torch.cuda.synchronize()
    c.poll()
    Hh.check_conv(y, K, oracle.conv_fwd(x.numpy(), w.numpy(), 2, pad), what="stem")
    assert torch.equal(y, y2)
    sums = stats[:parts * 2 * d.ldy].view(parts, 2, d.ldy).double().sum(0)
    v = y[..., :K].double()
    # fp32 chains of a few hundred values, combined in fp64
    assert torch.all((sums[0, :K] - v.sum((0, 1, 2))).abs() <= 1e-5 * v.abs().sum((0, 1, 2)))
    assert torch.all((sums[1, :K] - (v * v).sum((0, 1, 2))).abs() <= 1e-5 * (v * v).sum((0, 1, 2)))
    c.close()


def test_stem_behind_the_kernel_that_writes_its_image():
    """The stem's kernel starts before its predecessor has ended (a batch norm, which releases its dependents early): every pass sees the image of
    its own predecessor, whatever the same addresses held the pass before."""
    N, H, C, K, R = 16, 128, 3, 40, 7
    c = B.Context(0)
    gen = torch.Generator(device="cuda").manual_seed(W.BASE_SEED + 50)
    src = [torch.randn((N, H, H, 8), generator=gen, device="cuda").to(torch.bfloat16) for _ in range(2)]
    w = Hh.to_dev_padded(W.bf16_round(W.gen_weight(K, R, R, C, W.BASE_SEED + 51)), 8)
    d = B.make_conv_desc(N, H, H, C, K, R, R, 2, 3, 8, W.pad8(K), 8, 0, 2)
    bn = B.make_bn_desc(N, H, H, C, 8)
    g, b, sm, si = torch.ones(C, device="cuda"), torch.zeros(C, device="cuda"), torch.empty(C, device="cuda"), torch.empty(C, device="cuda")
    wsb = torch.empty(B.pt_bn_workspace_bytes(c, bn), dtype=torch.uint8, device="cuda")
    ws = torch.empty(B.pt_conv_workspace_bytes(c, d, B.PT_CONV_FWD), dtype=torch.uint8, device="cuda")
    image = torch.empty_like(src[0])
    ys = [torch.zeros((N, H // 2, H // 2, d.ldy), dtype=torch.bfloat16, device="cuda") for _ in range(40)]
    for i, y in enumerate(ys):
        B.pt_bn_relu_fwd(c, bn, src[i & 1], None, g, b, None, None, sm, si, image, wsb)
        B.pt_conv_fwd(c, d, image, w, y, ws)
    torch.cuda.synchronize()
    c.poll()
    assert B.pt_test_last_form(c) == B.PT_FORM_STEM
    for i in range(2):
        B.pt_bn_relu_fwd(c, bn, src[i], None, g, b, None, None, sm, si, image, wsb)
        torch.cuda.synchronize()
        alone = torch.zeros_like(ys[0])
        B.pt_conv_fwd(c, d, image, w, alone, ws)
        torch.cuda.synchronize()
        assert all(torch.equal(y, alone) for y in ys[i::2])
    assert not torch.equal(ys[0], ys[1])
    c.close()


# (N, H, W, C, K, R, pad) of the stride-2 forward by parity planes, taken whether they pay or not, and in the form of the library's choice: rows of 16, 32 and 64 lanes, one and several
# chunks, resident and streamed weights, several channel tiles, odd sizes, no padding, an even filter
@pytest.mark.parametrize("shape", [(150, 32, 32, 9, 17, 3, 1), (110, 33, 31, 32, 20, 3, 1), (80, 30, 60, 40, 33, 3, 0), (50, 56, 56, 70, 100, 3, 1), (100, 16, 130, 130, 24, 3, 1),
                                   (60, 40, 42, 17, 300, 3, 1), (170, 24, 40, 20, 12, 2, 0), (120, 26, 34, 24, 40, 5, 2),
                                   (2, 15, 14, 70, 300, 3, 1), (1, 7, 9, 8, 8, 4, 1), (3, 9, 70, 200, 40, 3, 0), (2, 56, 56, 260, 210, 3, 1)])
def test_stride_2_forward_by_planes(shape):
    c = Hh.ctx()
    B.pt_test_form(c, B.PT_FORM_PLANES)
    try:
        _stride_2_forward(shape)
        assert B.pt_test_last_form(c) == B.PT_FORM_PLANES
    finally:
        B.pt_test_form(c, B.PT_FORM_ANY)
    _stride_2_forward(shape)
    with pytest.raises(B.PtError):
        B.pt_test_form(c, B.PT_FORM_STEM)


def _stride_2_forward(shape):
    N, H, Wd, C, K, R, pad = shape
    x = W.gen_act(N, H, Wd, C, W.BASE_SEED + 48)
    w = W.bf16_round(W.gen_weight(K, R, R, C, W.BASE_SEED + 49))
    P, Q = (H + 2 * pad - R) // 2 + 1, (Wd + 2 * pad - R) // 2 + 1
    d = B.make_conv_desc(N, H, Wd, C, K, R, R, 2, pad, algo=2)
    c = Hh.ctx()
    y = Hh.out_buffer((N, P, Q), K, d.ldy, 0)
    B.pt_conv_fwd(c, d, Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(w, d.ldw), y, Hh.conv_ws(d, B.PT_CONV_FWD))
    torch.cuda.synchronize()
    c.poll()
    # (the oracle for images of either end and the middle; fp64 torch for all)
    ref = torch.nn.functional.conv2d(x.double().permute(0, 3, 1, 2), w.double().permute(0, 3, 1, 2), stride=2, padding=pad).permute(0, 2, 3, 1).numpy()
    Hh.check_conv(y, K, ref, what="fwd")
    # bf16 is the rounding of the fp32 output, and the statistics are those of the stored values
    xd, wd, d32 = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(w, d.ldw), B.make_conv_desc(N, H, Wd, C, K, R, R, 2, pad, out_f32=1, algo=2)
    y32, ys = Hh.out_buffer((N, P, Q), K, d.ldy, True), Hh.out_buffer((N, P, Q), K, d.ldy, False)
    B.pt_conv_fwd(c, d32, xd, wd, y32, Hh.conv_ws(d32, B.PT_CONV_FWD))
    stats = torch.full((B.pt_conv_fwd_stats_bytes(c, d) // 4,), float("nan"), device="cuda")
    parts = B.pt_conv_fwd_stats(c, d, xd, wd, ys, stats, Hh.conv_ws(d, B.PT_CONV_FWD))
    torch.cuda.synchronize()
    c.poll()
    assert torch.equal(y32[..., :K].to(torch.bfloat16), y[..., :K]) and torch.equal(ys[..., :K], y[..., :K])
    st, v = stats[: parts * 2 * d.ldy].view(parts, 2, d.ldy).double().sum(0), y[..., :K].double().reshape(-1, K)
    # (fp32 sums of at most P Q N values each: the bounds of the statistics' own test)
    assert torch.allclose(st[0, :K], v.sum(0), rtol=1e-5, atol=1e-5 * v.abs().sum(0).max().item()) and torch.allclose(st[1, :K], (v * v).sum(0), rtol=1e-5)
    for n in (0, N // 2, N - 1):
        np.testing.assert_allclose(ref[n:n + 1], oracle.conv_fwd(x[n:n + 1].numpy(), w.numpy(), 2, pad), rtol=1e-9, atol=1e-9)


# (N, H, W, C, K, R, stride): stride-2 weight gradients with few input channels (the generic kernel and the stem path):
# odd and even tap groups, K above and below 64, 5x5 and 7x7 stems
STRIDED_SMALL_C = [
    (2, 16, 16, 20, 36, 3, 2), (2, 18, 18, 64, 128, 3, 2), (3, 16, 16, 7, 70, 5, 2), (2, 32, 32, 3, 16, 7, 2), (2, 12, 12, 1, 9, 5, 2),
    (4, 20, 20, 33, 100, 2, 2),
]


@pytest.mark.parametrize("shape", STRIDED_SMALL_C)
def test_strided_weight_gradient_with_few_input_channels(shape):
    N, H, Wd, C, K, R, stride = shape
    x, w, dy, pad = _case(N, H, Wd, C, K, R, stride, seed=W.BASE_SEED + 53)
    dw = Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=2)[2]
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad), what="wgrad")
    assert torch.equal(dw, Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=2)[2])


# (N, H, W, C, K, R, pad): stride-1 filters with several taps and at most 64 input channels -- the weight gradient that
# stages row blocks and pairs taps: two dy boxes (K > 64), several tap groups with an odd last one (K = 200), 25 taps,
# a wide image, an even filter, padding 0 and padding larger than (R - 1) / 2
ROW_BLOCK = [
    (3, 12, 12, 20, 100, 3, 1), (2, 10, 14, 64, 200, 3, 1), (2, 9, 9, 6, 10, 5, 2), (1, 8, 120, 9, 12, 3, 1),
    (2, 11, 11, 13, 21, 3, 0), (2, 7, 7, 5, 9, 3, 2), (2, 6, 6, 33, 40, 2, 0), (64, 20, 20, 38, 38, 3, 1),
    # 1x1 filters on large maps take the same kernel (single tap, K > 128 in one tile)
    (3, 30, 30, 59, 143, 1, 0), (2, 28, 28, 7, 19, 1, 0), (2, 40, 33, 64, 250, 1, 0),
    # more than 64 input channels (the generic kernel): ragged channel tiles, 25 taps, a 28x28 map
    (2, 14, 14, 93, 77, 3, 1), (2, 15, 16, 130, 40, 3, 1), (3, 14, 20, 213, 242, 3, 1), (2, 16, 16, 128, 100, 5, 2), (8, 28, 28, 113, 111, 3, 1),
]


@pytest.mark.parametrize("shape", ROW_BLOCK)
def test_row_block_weight_gradient(shape):
    N, H, Wd, C, K, R, pad = shape
    seed = W.BASE_SEED + 41
    x = W.gen_act(N, H, Wd, C, seed)
    w = W.bf16_round(W.gen_weight(K, R, R, C, seed + 1))
    P, Q = H + 2 * pad - R + 1, Wd + 2 * pad - R + 1
    dy = W.gen_dy(N, P, Q, K, seed + 2)
    y, dx, dw, _ = Hh.run_conv_all(N, H, Wd, C, K, R, 1, pad, x, w, dy, algo=2)
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, 1, pad), what="wgrad")
    Hh.check_conv(y, K, oracle.conv_fwd(x.numpy(), w.numpy(), 1, pad), what="fwd")
    Hh.check_conv(dx, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, Wd, 1, pad), what="dgrad")
    again = Hh.run_conv_all(N, H, Wd, C, K, R, 1, pad, x, w, dy, algo=2)[2]
    assert torch.equal(dw, again)
    d = B.make_conv_desc(N, H, Wd, C, K, R, R, 1, pad, algo=2)
    rows, took = _wgrad_of_form(Hh.ctx(), d, Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy), B.PT_FORM_WGRAD_ROWS, 0)
    assert (took == B.PT_FORM_WGRAD_ROWS) == (C <= 64)
    Hh.check_conv(rows, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, 1, pad), what="wgrad, row blocks")


@pytest.mark.parametrize("shape", [(2, 16, 16, 20, 36, 3, 1), (2, 14, 14, 37, 70, 3, 1), (2, 8, 8, 7, 33, 1, 1), (2, 16, 16, 41, 20, 3, 2)])
def test_pad_lanes_up_to_a_multiple_of_16_are_zero(shape):
    """With channel pitches that are multiples of 16 (as the training harness uses) the bf16 outputs are stored in whole
    32-byte sectors: the pad lanes receive zeros, never stale accumulator columns."""
    N, H, Wd, C, K, R, stride = shape
    pad = R // 2
    x, w, dy, _ = _case(N, H, Wd, C, K, R, stride, seed=W.BASE_SEED + 23)
    ldx, ldy, ldw = W.pad16(C), W.pad16(K), W.pad8(C)
    d = B.make_conv_desc(N, H, Wd, C, K, R, R, stride, pad, ldx, ldy, ldw, 0, 2)
    P, Q = (H + 2 * pad - R) // stride + 1, (Wd + 2 * pad - R) // stride + 1
    xd, wd, dyd = Hh.to_dev_padded(x, ldx), Hh.to_dev_padded(w, ldw), Hh.to_dev_padded(dy, ldy)
    y = Hh.out_buffer((N, P, Q), K, ldy, 0)
    dx = Hh.out_buffer((N, H, Wd), C, ldx, 0)
    B.pt_conv_fwd(Hh.ctx(), d, xd, wd, y, Hh.conv_ws(d, B.PT_CONV_FWD))
    B.pt_conv_dgrad(Hh.ctx(), d, dyd, wd, dx, Hh.conv_ws(d, B.PT_CONV_DGRAD))
    torch.cuda.synchronize()
    Hh.ctx().poll()
    Hh.check_conv(y, K, oracle.conv_fwd(x.numpy(), w.numpy(), stride, pad), what="fwd")
    Hh.check_conv(dx, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, Wd, stride, pad), what="dgrad")
    assert torch.all(y[..., K:] == 0) and torch.all(dx[..., C:] == 0)


# (N, H, W, C, K, R, stride, extra pitch of x, of dy): the weight gradient loads pad lanes (here NaN) up to a multiple of 16 channels where
# the pitch has them, up to a multiple of 8 where not; both kernels, the space-to-depth stem
@pytest.mark.parametrize("shape", [(3, 12, 12, 19, 33, 3, 1, 8, 8), (3, 12, 12, 33, 19, 3, 1, 0, 16), (2, 14, 14, 70, 103, 3, 1, 8, 0),
                                   (2, 16, 16, 106, 41, 3, 2, 16, 32), (2, 10, 10, 130, 300, 1, 1, 24, 8), (2, 32, 32, 3, 19, 7, 2, 0, 8)])
def test_weight_gradient_of_nan_pad_lanes(shape):
    N, H, Wd, C, K, R, stride, ex, ey = shape
    x, w, dy, pad = _case(N, H, Wd, C, K, R, stride, seed=W.BASE_SEED + 29)
    d = B.make_conv_desc(N, H, Wd, C, K, R, R, stride, pad, W.pad8(C) + ex, W.pad8(K) + ey, W.pad8(C), 0, 2)
    dw = torch.full((K, R, R, C), 7680.0, device="cuda")
    B.pt_conv_wgrad(Hh.ctx(), d, Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy), dw, Hh.conv_ws(d, B.PT_CONV_WGRAD))
    torch.cuda.synchronize()
    Hh.ctx().poll()
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad), what="wgrad")


def _wgrad_of_form(c, d, xd, dyd, form, limit):
    """The weight gradient in the given form (PT_FORM_ANY: the library's choice) at a CTA limit, computed twice, and the form that it took."""
    B.pt_test_form(c, form)
    B.pt_set_wgrad_cta_limit(c, limit)
    try:
        ws = torch.empty(max(16, B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD)), dtype=torch.uint8, device="cuda")
        dw = torch.full((d.K, d.R, d.S, d.C), 7680.0, device="cuda")
        again = torch.full_like(dw, 7680.0)
        B.pt_conv_wgrad(c, d, xd, dyd, dw, ws)
        B.pt_conv_wgrad(c, d, xd, dyd, again, ws)
        torch.cuda.synchronize()
        c.poll()
    finally:
        B.pt_test_form(c, B.PT_FORM_ANY)
        B.pt_set_wgrad_cta_limit(c, 0)
    assert torch.equal(dw, again)
    return dw, B.pt_test_last_form(c)


# (N, H, W, C, K, R, S, stride, pad) of the filter-row form of the weight gradient: one and two blocks of channels on either side and just
# past them, units that leave rows over, both parities (odd and even sizes, no padding, more padding than the filter), filters of 2, 4, 5 and
# 8 columns, other than square, a wide image, a single output row
@pytest.mark.parametrize("shape", [(5, 14, 14, 65, 64, 3, 3, 1, 1), (4, 28, 28, 106, 129, 3, 3, 1, 1), (3, 13, 9, 160, 40, 3, 3, 1, 0), (2, 6, 100, 70, 20, 3, 3, 1, 1),
                                   (4, 28, 28, 106, 103, 3, 3, 2, 1), (3, 15, 17, 20, 70, 3, 3, 2, 1), (3, 15, 16, 33, 65, 3, 3, 2, 0), (2, 17, 12, 90, 30, 5, 5, 2, 2),
                                   (3, 12, 12, 66, 50, 2, 2, 2, 0), (3, 16, 16, 60, 130, 4, 4, 2, 3), (2, 24, 24, 64, 40, 8, 8, 2, 3), (2, 9, 20, 90, 24, 1, 5, 1, 2),
                                   (2, 3, 30, 80, 64, 3, 3, 1, 0), (64, 14, 14, 77, 77, 3, 3, 1, 1), (64, 28, 28, 38, 38, 3, 3, 2, 1)])
def test_filter_row_weight_gradient(shape):
    N, H, Wd, C, K, R, S, stride, pad = shape
    x = W.gen_act(N, H, Wd, C, W.BASE_SEED + 43)
    P, Q = (H + 2 * pad - R) // stride + 1, (Wd + 2 * pad - S) // stride + 1
    dy = W.gen_dy(N, P, Q, K, W.BASE_SEED + 44)
    ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), R, S, stride, pad)
    c = B.Context(0)
    d = B.make_conv_desc(N, H, Wd, C, K, R, S, stride, pad, W.pad8(C), W.pad16(K), W.pad8(C), 0, 2)
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    for limit in (0, 49, 3):                                    # (all SMs, a share of them, one CTA per filter row)
        for form in (B.PT_FORM_WGRAD_TAPS, B.PT_FORM_WGRAD_PIXELS, B.PT_FORM_ANY):
            dw, took = _wgrad_of_form(c, d, xd, dyd, form, limit)
            assert took == form or form == B.PT_FORM_ANY
            Hh.check_conv(dw, C, ref, what=f"wgrad at limit {limit}, form {took}")
    c.close()


# (N, H, W, C, K, R, S, pad, ldx, ldy) of the packed form: either pitch on either side, one and two blocks of dy, rows that do not divide into
# groups of four or two pixels, all padding and none, one to five filter rows and columns, an image of one column group, many images
@pytest.mark.parametrize("shape", [(5, 12, 12, 11, 13, 3, 3, 1, 16, 16), (40, 32, 32, 16, 16, 3, 3, 1, 16, 16), (3, 9, 13, 8, 20, 3, 3, 1, 16, 32), (4, 14, 15, 27, 9, 3, 3, 1, 32, 16),
                                   (20, 16, 16, 32, 32, 3, 3, 1, 32, 32), (3, 10, 11, 17, 31, 3, 3, 2, 32, 32), (3, 11, 10, 16, 7, 3, 3, 0, 16, 16), (2, 8, 9, 13, 12, 4, 5, 2, 16, 32),
                                   (2, 7, 21, 30, 30, 1, 2, 0, 32, 32), (3, 2, 3, 5, 6, 3, 3, 1, 16, 16), (2, 56, 56, 19, 19, 3, 3, 1, 32, 32), (2, 200, 6, 9, 9, 5, 3, 2, 16, 16)])
def test_packed_weight_gradient(shape):
    N, H, Wd, C, K, R, S, pad, ldx, ldy = shape
    x = W.gen_act(N, H, Wd, C, W.BASE_SEED + 45)
    P, Q = H + 2 * pad - R + 1, Wd + 2 * pad - S + 1
    dy = W.gen_dy(N, P, Q, K, W.BASE_SEED + 46)
    ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), R, S, 1, pad)
    c = B.Context(0)
    d = B.make_conv_desc(N, H, Wd, C, K, R, S, 1, pad, ldx, ldy, W.pad8(C), 0, 2)
    xd, dyd = Hh.to_dev_padded(x, ldx), Hh.to_dev_padded(dy, ldy)
    for limit in (0, 49, 5, 1):
        for form in (B.PT_FORM_WGRAD_PACKED, B.PT_FORM_ANY):
            dw, took = _wgrad_of_form(c, d, xd, dyd, form, limit)
            assert took == form or form == B.PT_FORM_ANY
            Hh.check_conv(dw, C, ref, what=f"wgrad at limit {limit}, form {took}")
    c.close()


def _dw_of_products(x, dy, R, S, stride, pad):
    """dw from every product of an output pixel's dy with the pixel of x that a tap has there, zeros outside the image among them (0 x Inf is a
    NaN), in fp64."""
    N, P, Q, K = dy.shape
    xp = torch.nn.functional.pad(x.double(), (0, 0, pad, pad + stride, pad, pad + stride))
    dw = torch.empty((K, R, S, x.shape[3]), dtype=torch.float64)
    for r in range(R):
        for s in range(S):
            v = xp[:, r:r + stride * (P - 1) + 1:stride, s:s + stride * (Q - 1) + 1:stride]
            dw[:, r, s] = (dy.double()[..., :, None] * v[..., None, :]).sum((0, 1, 2))
    return dw


# Infinities and NaN at the edges of the images, where a row of pixels meets the next one, a unit's last row the rows behind it or a column
# group the next: they reach the sums that they are part of and no other, in every form, however the splits exchange their sums
# (N, H, W, C, K, R, S, stride, pad, ldx, ldy, form)
@pytest.mark.parametrize("shape", [(3, 10, 9, 70, 40, 3, 3, 1, 1, 72, 40, "TAPS"), (2, 9, 12, 66, 130, 3, 3, 1, 0, 80, 136, "TAPS"), (3, 11, 14, 20, 70, 3, 3, 2, 1, 24, 72, "TAPS"),
                                   (40, 7, 8, 68, 24, 3, 3, 2, 1, 72, 24, "TAPS"), (3, 10, 9, 70, 40, 3, 3, 1, 1, 72, 40, "PIXELS"), (3, 11, 14, 20, 70, 3, 3, 2, 1, 24, 72, "PIXELS"),
                                   (3, 9, 13, 8, 20, 3, 3, 1, 1, 16, 32, "PACKED"), (40, 10, 11, 30, 9, 3, 3, 1, 1, 32, 16, "PACKED"), (2, 8, 9, 13, 12, 4, 5, 1, 2, 16, 32, "PACKED"),
                                   (3, 10, 13, 20, 33, 3, 3, 1, 1, 24, 40, "ROWS"), (3, 9, 9, 41, 30, 3, 3, 1, 1, 48, 32, "ROWS"), (40, 7, 9, 12, 21, 5, 5, 1, 2, 16, 24, "ROWS"),
                                   (2, 30, 30, 9, 12, 1, 1, 1, 0, 16, 16, "ROWS"), (2, 38, 32, 3, 16, 7, 7, 2, 3, 8, 16, "ANY"), (3, 12, 12, 4, 9, 3, 3, 2, 1, 8, 16, "ANY")])
def test_infinities_and_nan_reach_their_own_weight_gradients_only(shape):
    N, H, Wd, C, K, R, S, stride, pad, ldx, ldy, form = shape
    P, Q = (H + 2 * pad - R) // stride + 1, (Wd + 2 * pad - S) // stride + 1
    x, dy = W.gen_act(N, H, Wd, C, W.BASE_SEED + 91), W.gen_dy(N, P, Q, K, W.BASE_SEED + 92)
    inf, nan = float("inf"), float("nan")
    # one pixel in a channel of its own each: the corners of the first and the last image, the middles of the edges, an inner one
    spots = [(0, 0, 0, inf), (N - 1, H - 1, Wd - 1, inf), (0, H - 1, 0, -inf), (0, 0, Wd - 1, nan), (0, H // 2, 0, inf), (N - 1, H // 2, Wd - 1, -inf), (0, 0, Wd // 2, nan), (0, H - 1, Wd // 2, inf),
             (N // 2, H // 2, Wd // 2, nan)]
    for c, (n, h, w_, v) in zip(range(C - 1, 0, -1), spots):      # (channel 0 stays finite)
        x[n, h, w_, c] = v
    for k, (n, p, q, v) in zip(range(K - 1, 1, -1), [(0, 0, 0, inf), (N - 1, P - 1, Q - 1, nan), (N // 2, P // 2, Q // 2, -inf)]):
        dy[n, p, q, k] = v
    ref = _dw_of_products(x, dy, R, S, stride, pad)
    c = B.Context(0)
    d = B.make_conv_desc(N, H, Wd, C, K, R, S, stride, pad, ldx, ldy, W.pad8(C), 0, 2)
    xd, dyd = Hh.to_dev_padded(x, ldx), Hh.to_dev_padded(dy, ldy)
    want = B.PT_FORM_ANY if form == "ANY" else getattr(B, "PT_FORM_WGRAD_" + form)
    for limit in (0, 40, 1):
        B.pt_test_form(c, want)
        B.pt_set_wgrad_cta_limit(c, limit)
        ws = torch.empty(max(16, B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD)), dtype=torch.uint8, device="cuda")
        dw = torch.full((K, R, S, C), 7680.0, device="cuda")
        B.pt_conv_wgrad(c, d, xd, dyd, dw, ws)
        torch.cuda.synchronize()
        c.poll()
        assert want == B.PT_FORM_ANY or B.pt_test_last_form(c) == want
        got = dw.cpu().double()
        for what in (torch.isnan, torch.isposinf, torch.isneginf):
            assert torch.equal(what(got), what(ref)), (limit, what.__name__, int((what(got) & ~what(ref)).sum()), int((what(ref) & ~what(got)).sum()))
        fin = torch.isfinite(ref)
        assert fin.any() and (~fin).any()
        err = (got - ref)[fin]
        # (fp32 sums of products of bf16 values: the bound of the other tests, of the finite part)
        assert err.norm() <= 5e-3 * ref[fin].norm()
    c.close()


def test_wgrad_is_run_to_run_identical():
    N, H, C, K, R = 4, 14, 27, 19, 3
    x, w, dy, pad = _case(N, H, H, C, K, R, 1, W.BASE_SEED + 5)
    a = Hh.run_conv_all(N, H, H, C, K, R, 1, pad, x, w, dy)[2].cpu()
    b = Hh.run_conv_all(N, H, H, C, K, R, 1, pad, x, w, dy)[2].cpu()
    assert torch.equal(a, b)


@pytest.mark.parametrize("limit", [1, 7, 37])
def test_wgrad_with_a_cta_limit(limit):
    """The weight gradient may be held to fewer CTAs (to run beside other kernels): same result class, bounded by the limit."""
    c = Hh.ctx()
    try:
        B.pt_set_wgrad_cta_limit(c, limit)
        for (N, H, C, K, R) in [(4, 14, 93, 77, 3), (8, 28, 130, 70, 1), (3, 16, 11, 27, 3)]:
            x, w, dy, pad = _case(N, H, H, C, K, R, 1, W.BASE_SEED + 31 + limit)
            dw = Hh.run_conv_all(N, H, H, C, K, R, 1, pad, x, w, dy, algo=2)[2]
            Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, 1, pad), what=f"wgrad limit {limit}")
        with pytest.raises(B.PtError):
            B.pt_set_wgrad_cta_limit(c, -1)
    finally:
        B.pt_set_wgrad_cta_limit(c, 0)


def test_wgrad_cta_query_follows_the_limit():
    """pt_conv_wgrad_ctas reports tiles x splits at the current limit: never above a limit it can meet, whole multiples of
    the tile count, and an unsplit launch (more tiles than the limit) is reported as not waiting."""
    c = Hh.ctx()
    try:
        for (N, H, C, K, R, stride) in [(64, 14, 213, 242, 3, 1), (64, 56, 46, 59, 3, 1), (64, 28, 418, 113, 1, 1), (64, 7, 434, 495, 3, 1),
                                        (64, 224, 3, 55, 7, 2)]:
            d = B.make_conv_desc(N, H, H, C, K, R, R, stride, R // 2, 8 if C <= 4 else W.pad16(C), W.pad16(K))
            B.pt_set_wgrad_cta_limit(c, 1)
            tiles, waits = B.pt_conv_wgrad_ctas(c, d)
            assert tiles >= 1 and not waits
            prev = 0
            for lim in (8, 24, 49, 74, 148):
                B.pt_set_wgrad_cta_limit(c, lim)
                n, waits = B.pt_conv_wgrad_ctas(c, d)
                assert n % tiles == 0 and n >= prev
                assert (n <= lim and waits == (n > tiles)) or (n == tiles and not waits)
                prev = n
        assert B.pt_conv_wgrad_ctas(c, B.make_conv_desc(2, 8, 8, 16, 16, 3, 3, 1, 1, algo=1)) == (0, False)
    finally:
        B.pt_set_wgrad_cta_limit(c, 0)


def test_invalid_arguments_are_rejected_before_launch():
    c = Hh.ctx()
    buf = torch.zeros(4096, dtype=torch.bfloat16, device="cuda")
    good = B.make_conv_desc(1, 4, 4, 8, 8, 3, 3, 1, 1)
    for field, val in (("ldx", 9), ("ldy", 4), ("ldw", 12), ("C", 0), ("stride", 0), ("algo", 7)):
        d = B.make_conv_desc(1, 4, 4, 8, 8, 3, 3, 1, 1)
        setattr(d, field, val)
        with pytest.raises(B.PtError) as e:
            B.pt_conv_fwd(c, d, buf, buf, buf)
        assert e.value.status == 1
    with pytest.raises(B.PtError):
        B.pt_conv_fwd(c, good, None, buf, buf)
    d = B.make_conv_desc(2, 8, 8, 8, 8, 3, 3, 1, 1, algo=1)
    with pytest.raises(B.PtError) as e:       # the SIMT wgrad needs a workspace
        B.pt_conv_wgrad(c, d, buf, buf, torch.zeros(8 * 9 * 8, device="cuda"), None)
    assert e.value.status == 3
    c.poll()


@pytest.mark.parametrize("stride", [1, 2])
def test_tcgen05_path_takes_all_three_passes_when_forced(stride):
    """algo = 2 forces the tcgen05 kernels: the calls must not fall back silently."""
    N, H, C, K, R = 3, 12, 40, 24, 3
    x, w, dy, pad = _case(N, H, H, C, K, R, stride, W.BASE_SEED + 9)
    y, dx, dw, d = Hh.run_conv_all(N, H, H, C, K, R, stride, pad, x, w, dy, algo=2, out_f32=1)
    Hh.check_conv(y, K, oracle.conv_fwd(x.numpy(), w.numpy(), stride, pad), what="fwd tcgen05")
    Hh.check_conv(dx, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, H, stride, pad), what="dgrad tcgen05")
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad), what="wgrad tcgen05")
    # a 9x9 filter has more taps than the tcgen05 path's tap table: forcing it must fail loudly, auto must fall back
    d9 = B.make_conv_desc(1, 12, 12, 8, 8, 9, 9, 1, 4, algo=2)
    buf = torch.zeros(1 << 16, dtype=torch.bfloat16, device="cuda")
    with pytest.raises(B.PtError) as e:
        B.pt_conv_fwd(Hh.ctx(), d9, buf, buf, buf)
    assert e.value.status == 2


# Weight gradients whose splits meet as a thread-block cluster: lane quarters that are partly or wholly empty (C or K just above and
# below 32, 64 and 128), an odd last tap, one and several channel tiles, two to eight splits (the CTA limit), and accumulators larger
# than the shared memory of the owners (several rounds: 8 x 512 columns)
@pytest.mark.parametrize("N,H,C,K,R,stride", [(4, 12, 31, 33, 3, 1), (4, 12, 33, 129, 3, 1), (8, 9, 64, 256, 3, 1), (5, 10, 65, 127, 3, 1),
                                              (6, 14, 300, 260, 1, 1), (8, 15, 128, 96, 3, 2), (16, 8, 256, 128, 1, 1), (3, 28, 40, 20, 1, 1)])
def test_weight_gradient_splits_as_a_cluster(N, H, C, K, R, stride):
    c = Hh.ctx()
    x, w, dy, pad = _case(N, H, H, C, K, R, stride, W.BASE_SEED + C)
    ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad)
    d = B.make_conv_desc(N, H, H, C, K, R, R, stride, pad, algo=2)
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    try:
        for lim in (0, 2, 7, 40):
            B.pt_set_wgrad_cta_limit(c, lim)
            dw = torch.full((K, R, R, C), 7680.0, device="cuda")
            B.pt_conv_wgrad(c, d, xd, dyd, dw, Hh.conv_ws(d, B.PT_CONV_WGRAD))
            torch.cuda.synchronize()
            c.poll()
            Hh.check_conv(dw, C, ref, what=f"wgrad at limit {lim}")
            again = torch.full_like(dw, 7680.0)
            B.pt_conv_wgrad(c, d, xd, dyd, again, Hh.conv_ws(d, B.PT_CONV_WGRAD))
            torch.cuda.synchronize()
            assert torch.equal(dw, again)                        # fixed order of the sums
    finally:
        B.pt_set_wgrad_cta_limit(c, 0)


# (N, H, W, C, K, R, stride) at the edges of the launch variants: pixel rows of 16, 32 and 64 staged channels and outputs of at most 32
# (one or several tiles per CTA); last chunks of 16, 17, 32 and 33 channels with a ring per issuer; outputs two pixels apart with one and
# several column tiles, with and without room for 16-channel vectors, odd heights and widths, parities that no tap reaches
VARIANTS = [
    (4, 20, 20, 15, 33, 3, 1), (80, 20, 20, 16, 17, 3, 1), (80, 20, 20, 17, 31, 3, 1), (40, 20, 20, 32, 16, 3, 1), (40, 20, 20, 33, 32, 3, 1),
    (76, 32, 32, 80, 40, 1, 1), (76, 32, 32, 81, 24, 1, 1), (76, 32, 32, 32, 96, 1, 1), (76, 32, 32, 33, 97, 1, 1),
    (100, 34, 34, 70, 24, 3, 2), (100, 34, 34, 30, 20, 3, 2), (52, 34, 34, 290, 16, 3, 2),
    (3, 9, 11, 70, 65, 1, 2), (2, 16, 16, 300, 40, 1, 2), (2, 10, 8, 23, 100, 1, 2), (400, 28, 28, 16, 72, 1, 2),
]


@pytest.mark.parametrize("shape", VARIANTS)
def test_launch_variants(shape):
    N, H, Wd, C, K, R, stride = shape
    x, w, dy, pad = _case(*shape, seed=W.BASE_SEED + 71)
    y16, dx16, dw, _ = Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=2, out_f32=0)
    y32, dx32, _, _ = Hh.run_conv_all(N, H, Wd, C, K, R, stride, pad, x, w, dy, algo=2, out_f32=1)
    Hh.check_conv(y16, K, oracle.conv_fwd(x.numpy(), w.numpy(), stride, pad), what="fwd")
    Hh.check_conv(dx16, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, Wd, stride, pad), what="dgrad")
    Hh.check_conv(dw, C, oracle.conv_wgrad(x.numpy(), dy.numpy(), R, R, stride, pad), what="wgrad")
    # the same sums, rounded once more
    assert torch.equal(y16[..., :K], y32[..., :K].to(torch.bfloat16)) and torch.equal(dx16[..., :C], dx32[..., :C].to(torch.bfloat16))


# a 1x1 filter of stride 2 with padding 1 reaches the odd pixels only: the pixels of parity (0, 0) are among the zeros
@pytest.mark.parametrize("N,H,W_,C,K", [(2, 16, 16, 40, 24), (3, 18, 32, 130, 70)])
def test_data_gradient_of_a_padded_1x1_at_stride_2(N, H, W_, C, K):
    c = Hh.ctx()
    w, dy = W.bf16_round(W.gen_weight(K, 1, 1, C, W.BASE_SEED + 81)), W.gen_dy(N, H // 2 + 1, W_ // 2 + 1, K, W.BASE_SEED + 82)
    d = B.make_conv_desc(N, H, W_, C, K, 1, 1, 2, 1, algo=2)
    dx = Hh.out_buffer((N, H, W_), C, d.ldx, False)
    B.pt_conv_dgrad(c, d, Hh.to_dev_padded(dy, d.ldy), Hh.to_dev_padded(w, d.ldw), dx, None)
    torch.cuda.synchronize()
    c.poll()
    Hh.check_conv(dx, C, oracle.conv_dgrad(dy.numpy(), w.numpy(), H, W_, 2, 1), what="dgrad")


def test_a_round_of_many_layers_costs_the_host_no_more_per_call_than_one_layer():
    """The launch shape of a weight gradient is chosen once per descriptor: going round the layers of a network must not choose it again."""
    import time
    c = B.Context(0)
    # small maps and batches, where every candidate is weighed
    descs = [B.make_conv_desc(N, H, H, C, K, 3, 3, 1, 1) for N in (2, 3, 4, 6, 8) for H in (14, 28, 32) for C in (20, 31, 48, 64) for K in (17, 60, 128)]
    for d in descs:
        B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD)

    def per_call(ds):
        best = 1e9
        for _ in range(5):
            t0 = time.perf_counter()
            for d in ds:
                B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD)
            best = min(best, (time.perf_counter() - t0) / len(ds))
        return best

    many, one = per_call(descs), per_call([descs[-1]] * len(descs))
    c.close()
    assert len(descs) == 180
    # (with 128 places of one plan each, the round took 2.4 times as long per call as the repeated layer)
    assert many < 1.6 * one, (many, one)


def test_a_workspace_sized_at_one_cta_limit_serves_every_smaller_one():
    c = B.Context(0)
    for N, H, C, K, R, stride in [(9, 56, 41, 9, 3, 1), (6, 32, 3, 60, 3, 1), (14, 7, 30, 503, 3, 1), (24, 28, 18, 228, 3, 2), (64, 112, 3, 55, 7, 2),
                                  (4, 16, 300, 200, 1, 1), (11, 28, 1373, 458, 1, 1), (2, 9, 64, 256, 3, 1)]:
        d = B.make_conv_desc(N, H, H, C, K, R, R, stride, R // 2, ldx=8 if C <= 4 else None)
        need = []
        for limit in [0] + list(range(147, 0, -1)):
            B.pt_set_wgrad_cta_limit(c, limit)
            need.append(B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD))
        assert all(a >= b for a, b in zip(need, need[1:])), (N, H, C, K, R)
    # the workspace of the largest limit, at every limit: what a launch uses stays inside it
    N, H, C, K = 9, 56, 41, 9
    d = B.make_conv_desc(N, H, H, C, K, 3, 3, 1, 1)
    x, _, dy, _ = _case(N, H, H, C, K, 3, 1, W.BASE_SEED + 83)
    xd, dyd = Hh.to_dev_padded(x, d.ldx), Hh.to_dev_padded(dy, d.ldy)
    B.pt_set_wgrad_cta_limit(c, 0)
    n = B.pt_conv_workspace_bytes(c, d, B.PT_CONV_WGRAD)
    buf = torch.full((n + 4096,), 77, dtype=torch.uint8, device="cuda")
    ref = oracle.conv_wgrad(x.numpy(), dy.numpy(), 3, 3, 1, 1)
    for limit in (0, 140, 110, 74, 49, 36, 24, 12, 6, 2, 1):
        B.pt_set_wgrad_cta_limit(c, limit)
        dw = torch.empty((K, 3, 3, C), device="cuda")
        B.pt_conv_wgrad(c, d, xd, dyd, dw, buf[:n])
        torch.cuda.synchronize()
        c.poll()
        Hh.check_conv(dw, C, ref, what=f"wgrad at limit {limit}")
        assert torch.all(buf[n:] == 77)
    c.close()


def test_a_limit_on_the_weight_gradients_leaves_the_data_gradients_alone():
    """Only the data gradients' own limit makes their launches smaller; neither changes a result."""
    c = B.Context(0)
    N, H, C = 64, 56, 64
    gen = torch.Generator(device="cuda").manual_seed(W.BASE_SEED + 84)
    d = B.make_conv_desc(N, H, H, C, C, 3, 3, 1, 1)
    dy = torch.randn((N, H, H, C), generator=gen, device="cuda").to(torch.bfloat16)
    w = torch.randn((C, 3, 3, C), generator=gen, device="cuda").to(torch.bfloat16)

    def run(wgrad_limit, dgrad_limit):
        B.pt_set_wgrad_cta_limit(c, wgrad_limit)
        if dgrad_limit:
            B.pt_set_dgrad_cta_limit(c, dgrad_limit)
        dx = torch.empty_like(dy)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = 1e9
        for _ in range(5):
            a.record()
            for _ in range(40):
                B.pt_conv_dgrad(c, d, dy, w, dx, None)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return dx, best

    run(0, 0)
    dx0, t0 = run(0, 0)
    dx1, t1 = run(49, 0)
    assert torch.equal(dx0, dx1) and t1 < 1.1 * t0, (t0, t1)
    dx2, t2 = run(49, 74)
    assert torch.equal(dx0, dx2) and t2 > 1.3 * t0, (t0, t2)      # (half of the SMs: about twice the time)
    with pytest.raises(B.PtError):
        B.pt_set_dgrad_cta_limit(c, -1)
    c.close()
