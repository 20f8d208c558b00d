"""The warm-start network's convolution kernels against the float64 CPU
reference: forward, data gradient (with the ReLU mask), filter and bias
gradients on ragged shapes, bitwise determinism, and the whole network's
parameter gradients."""
import numpy as np
import pytest
import torch

from oracle import cnn_reference as ref

pytestmark = pytest.mark.gpu

# N, H, W, C, K, R, S, stride, pad: tails in every GEMM dimension
SHAPES = [
    (2, 17, 23, 8, 32, 3, 3, 1, 1),
    (2, 33, 31, 8, 24, 3, 3, 2, 1),
    (1, 40, 40, 40, 72, 3, 3, 2, 1),
    (3, 16, 16, 128, 64, 3, 3, 1, 1),
    (2, 9, 13, 32, 8, 1, 1, 1, 0),
    (1, 66, 70, 64, 128, 3, 3, 1, 1),
    (1, 30, 30, 16, 16, 3, 3, 2, 0),
    (2, 15, 17, 16, 8, 1, 1, 2, 0),   # stride 2, 1 x 1: two parity classes see no tap
    (1, 21, 19, 8, 16, 5, 5, 2, 2),
    (1, 64, 64, 32, 64, 3, 3, 2, 1),  # the network's second layer at small size
]


def _bf16(a, dev):
    """(bf16 device tensor, the same values as float64 numpy)."""
    t = torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16)
    return t.to(dev), t.to(torch.float64).numpy()


def _inputs(shape, seed):
    N, H, W, C, K, R, S, stride, pad = shape
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((N, H, W, C))
    w = rng.standard_normal((K, R, S, C)) / np.sqrt(R * S * C)
    b = rng.standard_normal(K).astype(np.float32)
    P = (H + 2 * pad - R) // stride + 1
    Q = (W + 2 * pad - S) // stride + 1
    dy = rng.standard_normal((N, P, Q, K))
    return x, w, b, dy


@pytest.fixture(scope="module", params=["tcgen05", "mma_sync"])
def cnn(request):
    """The convolution module with the forward / data-gradient engine set to
    the tcgen05 tensor cores or the warp-level MMA (every test runs on both)."""
    from paper_2606_21381_gb300 import cnn as m
    m.use_tcgen05(request.param == "tcgen05")
    yield m
    assert m.sync_status() == 0
    m.use_tcgen05(True)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("relu", [False, True])
def test_conv_forward_matches_reference(cnn, shape, relu):
    dev = torch.device("cuda")
    x, w, b, _ = _inputs(shape, 1)
    xd, x64 = _bf16(x, dev)
    wd, w64 = _bf16(w, dev)
    bd = torch.from_numpy(b).to(dev)
    y, y32 = cnn.conv2d(xd, wd, bd, shape[7], shape[8], relu, want_f32=True)
    want = ref.conv_forward(x64, w64, b.astype(np.float64), shape[7], shape[8], relu)
    assert cnn.sync_status() == 0
    got32 = y32.cpu().numpy().astype(np.float64)
    scale = np.abs(want).max()
    assert np.abs(got32 - want).max() <= 1e-5 * scale
    # the bf16 output is the fp32 value rounded to nearest
    got = y.to(torch.float32).cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * scale)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("masked", [False, True])
def test_conv_backward_data_matches_reference(cnn, shape, masked):
    dev = torch.device("cuda")
    x, w, b, dy = _inputs(shape, 2)
    xd, x64 = _bf16(x, dev)
    wd, w64 = _bf16(w, dev)
    dyd, dy64 = _bf16(dy, dev)
    dx = cnn.conv2d_backward_data(dyd, wd, tuple(xd.shape), shape[7], shape[8],
                                  x_act=xd if masked else None)
    want, _, _ = ref.conv_grads(x64, w64, b.astype(np.float64), shape[7], shape[8], dy64)
    if masked:
        want = want * (x64 > 0)
    assert cnn.sync_status() == 0
    got = dx.to(torch.float32).cpu().numpy().astype(np.float64)
    scale = np.abs(want).max()
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * scale)


@pytest.mark.parametrize("shape", SHAPES)
def test_conv_backward_filter_matches_reference(cnn, shape):
    dev = torch.device("cuda")
    x, w, b, dy = _inputs(shape, 3)
    xd, x64 = _bf16(x, dev)
    _, w64 = _bf16(w, dev)
    dyd, dy64 = _bf16(dy, dev)
    dw, db = cnn.conv2d_backward_filter(dyd, xd, w.shape, shape[7], shape[8])
    _, want_w, want_b = ref.conv_grads(x64, w64, b.astype(np.float64), shape[7], shape[8], dy64)
    got_w = dw.cpu().numpy().astype(np.float64)
    assert np.abs(got_w - want_w).max() <= 1e-5 * np.abs(want_w).max() * np.sqrt(dy.size / dy.shape[-1])
    assert np.abs(db.cpu().numpy() - want_b).max() <= 1e-5 * np.abs(dy64).sum(axis=(0, 1, 2)).max()


def test_filter_gradient_spans_several_pixel_splits(cnn):
    # 2 x 64 x 64 output pixels = 4 splits of 2048 plus a ragged tail
    shape = (2, 65, 66, 8, 16, 3, 3, 1, 1)
    test_conv_backward_filter_matches_reference(cnn, shape)


def test_kernels_are_bitwise_deterministic(cnn):
    dev = torch.device("cuda")
    shape = (4, 64, 64, 32, 64, 3, 3, 1, 1)
    x, w, b, dy = _inputs(shape, 4)
    xd, _ = _bf16(x, dev)
    wd, _ = _bf16(w, dev)
    dyd, _ = _bf16(dy, dev)
    bd = torch.from_numpy(b).to(dev)
    outs = []
    for _ in range(2):
        y = cnn.conv2d(xd, wd, bd, 1, 1, True)
        dx = cnn.conv2d_backward_data(dyd, wd, tuple(xd.shape), 1, 1, x_act=xd)
        dw, db = cnn.conv2d_backward_filter(dyd, xd, w.shape, 1, 1)
        outs.append([t.clone() for t in (y, dx, dw, db)])
    for a, c in zip(*outs):
        assert torch.equal(a, c)


def test_relu_backward(cnn):
    dev = torch.device("cuda")
    rng = np.random.default_rng(5)
    dyd, dy64 = _bf16(rng.standard_normal(1000), dev)
    actd, act64 = _bf16(rng.standard_normal(1000), dev)
    got = cnn.relu_backward(dyd, actd).to(torch.float32).cpu().numpy()
    assert np.array_equal(got, np.where(act64 > 0, dy64, 0.0).astype(np.float32))


def _reference_network_grads(net, x64, dout64):
    """float64 CPU autograd through the same network, with activations
    rounded to bf16 where the kernels store them."""
    import torch.nn.functional as F
    ws = [torch.from_numpy(w.to(torch.bfloat16).to(torch.float64).cpu().numpy()).permute(0, 3, 1, 2)
          .contiguous().requires_grad_(True) for w in net.w]
    bs = [b.cpu().double().clone().requires_grad_(True) for b in net.b]
    a = torch.from_numpy(x64).permute(0, 3, 1, 2)
    for i, (_, _, _, stride, pad) in enumerate(net.specs):
        z = F.conv2d(a, ws[i], bs[i], stride=stride, padding=pad)
        if i < len(net.specs) - 1:
            a = torch.clamp(z, min=0.0)
            a = a + (a.to(torch.bfloat16).to(torch.float64) - a).detach()
        else:
            out = z
    (out * torch.from_numpy(dout64).permute(0, 3, 1, 2)).sum().backward()
    return [w.grad.permute(0, 2, 3, 1).numpy() for w in ws], [b.grad.numpy() for b in bs], \
        out.detach().permute(0, 2, 3, 1).numpy()


def test_network_gradients_match_reference(cnn):
    dev = torch.device("cuda")
    net = cnn.WarmStartNet(dev, seed=1)
    rng = np.random.default_rng(6)
    x = np.zeros((2, 64, 64, 8))
    x[..., :2] = rng.standard_normal((2, 64, 64, 2))
    xd, x64 = _bf16(x, dev)
    out, acts = net.forward(xd)
    dout = rng.standard_normal(tuple(out.shape)).astype(np.float32)
    doutd, dout64 = _bf16(dout, dev)
    grads = net.backward(doutd.to(torch.float32), acts)
    want_w, want_b, want_out = _reference_network_grads(net, x64, dout64)
    got_out = out.cpu().numpy()
    assert np.abs(got_out - want_out).max() <= 2e-2 * np.abs(want_out).max()
    for i, ((dw, db), ww, wb) in enumerate(zip(grads, want_w, want_b)):
        gw = dw.cpu().numpy().astype(np.float64)
        if i == 0:  # padding channels are zero in the input
            gw, ww = gw[..., :2], ww[..., :2]
        cos = (gw * ww).sum() / np.sqrt((gw * gw).sum() * (ww * ww).sum())
        assert cos > 0.999, (i, cos)
        assert np.linalg.norm(gw - ww) <= 3e-2 * np.linalg.norm(ww), i
        gb = db.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(gb - wb) <= 3e-2 * np.linalg.norm(wb) + 1e-6, i


# the edges of the patch kernels' plans: several column blocks and channel
# chunks, more chunks than shared memory holds, wide filters on both strides,
# padding past the filter, classes and images smaller than a tile
PATCH_SHAPES = [
    (1, 20, 18, 264, 136, 3, 3, 1, 1),
    (1, 9, 9, 1032, 16, 3, 3, 1, 1),
    (2, 40, 36, 32, 48, 5, 5, 2, 2),
    (1, 24, 25, 16, 8, 8, 8, 1, 3),
    (1, 37, 21, 72, 24, 7, 7, 2, 3),
    (1, 10, 11, 64, 16, 3, 3, 1, 4),
    (1, 13, 12, 136, 40, 1, 1, 2, 1),
    (5, 3, 2, 24, 200, 3, 2, 2, 1),
    (2, 70, 34, 40, 16, 3, 3, 1, 0),
    # eight channels, nine or ten taps
    (2, 35, 70, 8, 40, 3, 3, 1, 1),
    (3, 67, 41, 8, 64, 3, 3, 2, 1),
    (1, 20, 33, 8, 8, 2, 5, 2, 2),
    (1, 9, 100, 8, 24, 5, 2, 1, 0),
]


@pytest.mark.parametrize("shape", PATCH_SHAPES)
def test_patch_kernels_match_reference(cnn, shape):
    test_conv_forward_matches_reference(cnn, shape, True)
    test_conv_backward_data_matches_reference(cnn, shape, True)
    test_conv_backward_filter_matches_reference(cnn, shape)


@pytest.mark.parametrize("shape", SHAPES + PATCH_SHAPES)
def test_forward_without_the_fp32_copy_gives_the_same_bits(cnn, shape):
    dev = torch.device("cuda")
    x, w, b, _ = _inputs(shape, 1)
    xd, _ = _bf16(x, dev)
    wd, _ = _bf16(w, dev)
    bd = torch.from_numpy(b).to(dev)
    y, _ = cnn.conv2d(xd, wd, bd, shape[7], shape[8], True, want_f32=True)
    assert torch.equal(cnn.conv2d(xd, wd, bd, shape[7], shape[8], True), y)


def _at(shape, dtype, offset):
    """A contiguous CUDA tensor `offset` elements past a 16-byte boundary."""
    flat = torch.empty(int(np.prod(shape)) + 16, dtype=dtype, device="cuda")
    return flat[offset:offset + int(np.prod(shape))].view(shape)


@pytest.mark.parametrize("shape", [
    (1, 20, 33, 8, 24, 3, 3, 1, 1),   # eight channels, nine taps
    (1, 20, 18, 32, 40, 3, 3, 1, 1),  # tcgen05
    (1, 9, 13, 32, 8, 1, 1, 1, 0),    # a short reduction
])
def test_forward_into_outputs_that_are_only_pair_aligned(cnn, shape):
    # y 4-byte and y_f32 8-byte aligned: no kernel that stores 16-byte vectors
    from paper_2606_21381_gb300 import _lib
    dev = torch.device("cuda")
    x, w, b, _ = _inputs(shape, 1)
    xd, x64 = _bf16(x, dev)
    wd, w64 = _bf16(w, dev)
    bd = torch.from_numpy(b).to(dev)
    want = ref.conv_forward(x64, w64, b.astype(np.float64), shape[7], shape[8], True)
    scale = np.abs(want).max()
    s = cnn.conv_shape(xd, wd, shape[7], shape[8])
    for want32 in (False, True):
        y = _at(want.shape, torch.bfloat16, 2)
        y32 = _at(want.shape, torch.float32, 2) if want32 else None
        assert _lib.lib().osog_conv2d_forward(s, cnn._ptr(xd), cnn._ptr(wd), cnn._ptr(bd), 1, cnn._ptr(y),
                                              cnn._ptr(y32), cnn._stream(dev)) == 0
        got = y.to(torch.float32).cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * scale)
        if want32:
            assert np.abs(y32.cpu().numpy() - want).max() <= 1e-5 * scale


@pytest.mark.parametrize("shape", [(1, 21, 18, 40, 24, 3, 3, 1, 1), (2, 15, 17, 16, 40, 3, 3, 2, 1)])
@pytest.mark.parametrize("what", ["w", "x_act", "dx"])
def test_backward_data_of_operands_that_are_not_16_byte_aligned(cnn, shape, what):
    # filters 2 bytes, the mask and the result 4 bytes past a 16-byte boundary
    from paper_2606_21381_gb300 import _lib
    dev = torch.device("cuda")
    x, w, b, dy = _inputs(shape, 2)
    xd, x64 = _bf16(x, dev)
    wd, w64 = _bf16(w, dev)
    dyd, dy64 = _bf16(dy, dev)
    want, _, _ = ref.conv_grads(x64, w64, b.astype(np.float64), shape[7], shape[8], dy64)
    want = want * (x64 > 0)
    dx = torch.empty_like(xd)
    if what == "w":
        wd = _at(wd.shape, torch.bfloat16, 1).copy_(wd)
    elif what == "x_act":
        xd = _at(xd.shape, torch.bfloat16, 2).copy_(xd)
    else:
        dx = _at(xd.shape, torch.bfloat16, 2)
    s = cnn.conv_shape(xd, wd, shape[7], shape[8])
    w_t = torch.empty(wd.numel(), dtype=torch.bfloat16, device=dev)
    assert _lib.lib().osog_conv2d_backward_data(s, cnn._ptr(dyd), cnn._ptr(wd), cnn._ptr(xd), cnn._ptr(dx),
                                                cnn._ptr(w_t), cnn._stream(dev)) == 0
    got = dx.to(torch.float32).cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= 2.0 ** -8 * np.abs(want) + 1e-5 * np.abs(want).max())


@pytest.mark.parametrize("shape", [
    (1, 21, 18, 40, 24, 3, 3, 1, 1),
    (2, 40, 37, 16, 136, 3, 3, 2, 1),
    (1, 9, 30, 72, 16, 5, 2, 1, 2),
    (2, 35, 70, 8, 40, 3, 3, 1, 1),  # eight channels, nine taps
    (1, 67, 41, 8, 24, 3, 3, 2, 1),
    (1, 32, 16, 24, 16, 3, 3, 1, 1),  # whole tiles
])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_filter_gradient_of_activations_that_are_not_finite(cnn, shape, value):
    # at the corners and edges of the image: exactly the entries that such a pixel
    # is a factor of are not finite, the others are as accurate as ever
    dev = torch.device("cuda")
    x, w, b, dy = _inputs(shape, 3)
    H, W = shape[1:3]
    for c, (h, v) in enumerate([(0, 0), (H - 1, W - 1), (H - 1, W // 2), (H // 2, W - 1), (H - 2, W - 2)]):
        x[0, h, v, c] = value
    xd, x64 = _bf16(x, dev)
    _, w64 = _bf16(w, dev)
    dyd, dy64 = _bf16(dy, dev)
    dw, db = cnn.conv2d_backward_filter(dyd, xd, w.shape, shape[7], shape[8])
    _, want_w, want_b = ref.conv_grads(x64, w64, b.astype(np.float64), shape[7], shape[8], dy64)
    got_w = dw.cpu().numpy().astype(np.float64)
    fin = np.isfinite(want_w)
    assert np.array_equal(np.isfinite(got_w), fin)
    np.testing.assert_array_equal(got_w[~fin], want_w[~fin])
    assert np.abs(got_w[fin] - want_w[fin]).max() <= 1e-5 * np.abs(want_w[fin]).max() * np.sqrt(dy.size / dy.shape[-1])
    assert np.abs(db.cpu().numpy() - want_b).max() <= 1e-5 * np.abs(dy64).sum(axis=(0, 1, 2)).max()


def test_long_filter_gradients_are_as_accurate_as_the_general_kernel():
    # 131,072 pixels in a layer wide enough to fill the chip with nine splits: the
    # accumulators' rounding grows with the pixels added in one (2048 in the general
    # kernel), so the norm of the error stays below its, but for the order of the
    # products (a quarter at most)
    from paper_2606_21381_gb300 import cnn as m
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((32, 64, 64, 512), generator=g, device="cuda").clamp_(min=0).to(torch.bfloat16)
    dy = (torch.randn((32, 64, 64, 512), generator=g, device="cuda") + 0.5).to(torch.bfloat16)
    want = dy.reshape(-1, 512).double().t() @ x.reshape(-1, 512).double()
    err = []
    for engine in (False, True):
        m.use_tcgen05(engine)
        dw, db = m.conv2d_backward_filter(dy, x, (512, 1, 1, 512), 1, 0)
        err.append((dw.reshape(512, 512).double() - want).norm().item())
        assert (db.double() - dy.double().sum((0, 1, 2))).abs().max() <= 2e-6 * dy.double().abs().sum((0, 1, 2)).max()
    assert err[1] <= 1.25 * err[0]


# filter gradients whose CTAs add several tiles, with the blocks (of output and input
# channels and of taps) that share the 152 SMs: stages are used again (two of them; one,
# for wide filters on stride 2), accumulators go on over tiles, and CTAs with and without
# the bias gradient run side by side
MANY_TILES = [
    ((6, 48, 40, 136, 264, 3, 3, 1, 1), 18, (16, 8)),
    ((9, 70, 66, 72, 16, 7, 7, 2, 3), 9, (16, 8)),
    ((20, 50, 50, 32, 64, 3, 3, 1, 1), 1, (16, 8)),
    ((3, 200, 400, 8, 16, 3, 3, 1, 1), 0, (8, 32)),  # eight channels, nine taps: 304 CTAs
    ((3, 200, 400, 8, 64, 3, 3, 1, 1), 0, (8, 32)),
]


@pytest.mark.parametrize("shape,blocks,tile", MANY_TILES)
def test_filter_gradients_of_several_tiles_a_cta(cnn, shape, blocks, tile):
    N, H, W, _, _, R, S, stride, pad = shape
    P, Q = (H + 2 * pad - R) // stride + 1, (W + 2 * pad - S) // stride + 1
    tiles = N * -(-P // tile[0]) * -(-Q // tile[1])
    splits = max(152 // blocks, -(-N * P * Q // 1920)) if blocks else 304
    assert tiles >= 2.4 * splits
    test_conv_backward_filter_matches_reference(cnn, shape)


# both sides of the forward kernels' dispatch and of the column blocks: eight channels
# with 16, 25 and 28 taps, 136 and 200 output channels
@pytest.mark.parametrize("shape", [
    (1, 20, 18, 8, 24, 4, 4, 1, 2), (2, 15, 17, 8, 40, 5, 5, 2, 2), (1, 20, 18, 8, 24, 4, 7, 1, 3),
    (1, 18, 20, 16, 136, 3, 3, 1, 1), (2, 9, 21, 72, 200, 3, 3, 2, 1),
])
def test_forward_routes_match_reference(cnn, shape):
    test_conv_forward_matches_reference(cnn, shape, True)
    test_forward_without_the_fp32_copy_gives_the_same_bits(cnn, shape)


# few tiles: the taps spread over the idle SMs, one to a CTA and several
@pytest.mark.parametrize("shape", [(1, 7, 10, 8, 24, 7, 7, 2, 7), (2, 12, 7, 16, 48, 5, 5, 1, 0),
                                   (1, 30, 22, 40, 136, 8, 3, 1, 2)])
def test_filter_gradients_of_a_few_tiles(cnn, shape):
    test_conv_backward_filter_matches_reference(cnn, shape)
