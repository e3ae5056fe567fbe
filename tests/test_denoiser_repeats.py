"""The gradient sums of the denoiser have a fixed order: the same inputs give the same bits, call after call,
in the weight and bias gradients of every kernel and in whole training steps."""
import pytest
import torch

from paper_1608_05238_gb300 import _build
from paper_1608_05238_gb300 import denoise_ops as ops
from paper_1608_05238_gb300.denoise_ops import Act
from paper_1608_05238_gb300.denoiser import UNet, r64, sample_scale

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    ops.lib()


def _act(B, H, W, C, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    t = torch.zeros(B, H, W, r64(C), dtype=torch.bfloat16, device="cuda")
    t[..., :C] = torch.randn(B, H, W, C, generator=g, device="cuda").bfloat16()
    return t


# cout > 64: one tap a block (32, 11, 8 and 16 splits, a ragged second row tile); cout <= 64, W % 64 == 0: nine taps a
# block (152 and 50 splits); 1x1 (128 splits)
@pytest.mark.parametrize("B,H,W,cin,cout,taps", [(8, 64, 64, 64, 96, 9), (8, 64, 64, 384, 128, 9), (8, 32, 32, 256, 256, 9),
                                                 (4, 64, 64, 70, 130, 9), (8, 128, 128, 33, 32, 9), (4, 64, 64, 160, 64, 9),
                                                 (8, 128, 128, 32, 33, 1)])
def test_weight_and_bias_gradients_repeat(B, H, W, cin, cout, taps):
    x, dz = _act(B, H, W, cin, 1), _act(B, H, W, cout, 2)

    def both():
        dw, db = torch.zeros(cout, taps, cin, device="cuda"), torch.zeros(cout, device="cuda")
        ops.wgrad_nhwc(Act(dz, cout), Act(x, cin), taps, dw, db=db)
        one = torch.zeros(cout, device="cuda")
        ops.bias_grad(Act(dz, cout), one)
        return dw, db, one

    ref = both()
    for _ in range(6):
        assert all(torch.equal(a, b) for a, b in zip(ref, both()))
    ops.check()
    # against 64 bits: FP32 sums of P products of about unit size, in K steps of 16 and ranges of them, err by less
    # than P / 16 roundings of the running sum's size (sqrt P); 2^-24 P / 16 sqrt P in all
    P = B * H * W
    z, xx = dz[..., :cout].double(), torch.nn.functional.pad(x[..., :cin].double(), (0, 0, 1, 1, 1, 1))
    tol = 2.0 ** -24 * P / 16 * P ** 0.5
    for tap in range(taps):
        ky, kx = divmod(tap, 3) if taps == 9 else (1, 1)
        ex = torch.einsum("bhwn,bhwc->nc", z, xx[:, ky:ky + H, kx:kx + W])
        assert (ref[0][:, tap].double() - ex).abs().max() <= tol
    for b in ref[1:]:
        assert (b.double() - z.sum((0, 1, 2))).abs().max() <= tol


@pytest.mark.parametrize("B,H,W,cin,cout,taps", [(1, 8, 32, 128, 128, 9), (1, 4, 16, 40, 33, 9), (1, 1, 64, 64, 32, 9)])
def test_one_split_repeats(B, H, W, cin, cout, taps):
    """Few pixels: one block sums a tile and adds it straight onto what stands there."""
    x, dz = _act(B, H, W, cin, 6), _act(B, H, W, cout, 7)
    out = []
    for _ in range(4):
        dw, db = torch.full((cout, taps, cin), 0.5, device="cuda"), torch.full((cout,), 0.25, device="cuda")
        ops.wgrad_nhwc(Act(dz, cout), Act(x, cin), taps, dw, db=db)
        out.append((dw, db))
    ops.check()
    assert all(torch.equal(a, b) for o in out[1:] for a, b in zip(out[0], o))


@pytest.mark.parametrize("B,H,W,cin,cout", [(4, 64, 64, 128, 128), (2, 64, 128, 33, 32), (1, 8, 32, 64, 128)])
def test_sums_beside_a_convolution_are_the_same(B, H, W, cin, cout):
    """dn_wgrad_begin, a convolution, dn_wgrad_end beside it (many splits of both kernels, and one): the bits of the
    one call, and the convolution's own result; a second end adds nothing."""
    x, dz = _act(B, H, W, cin, 8), _act(B, H, W, cout, 9)
    ref = [torch.zeros(cout, 9, cin, device="cuda"), torch.zeros(cout, device="cuda")]
    ops.wgrad_nhwc(Act(dz, cout), Act(x, cin), 9, ref[0], db=ref[1])
    g = torch.Generator(device="cuda").manual_seed(10)
    wd = (0.05 * torch.randn((cin + 15) // 16 * 16, 9, r64(cout), generator=g, device="cuda")).bfloat16()
    dx, dx2 = torch.zeros(B, H, W, r64(cin), dtype=torch.bfloat16, device="cuda"), None
    ops.conv(dz, wd, cin, dx, cin=cout)
    for _ in range(5):
        got = [torch.zeros_like(r) for r in ref]
        dx2 = torch.zeros_like(dx)
        p = ops.wgrad_begin(Act(dz, cout), Act(x, cin), 9, got[0], got[1])
        ops.conv(dz, wd, cin, dx2, cin=cout)
        ops.wgrad_end(p, True)
        ops.wgrad_end(p, False)
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1]) and torch.equal(dx, dx2)
    ops.check()


def test_wgrad_of_transposed_copies_repeats():
    B, H, W, cin, cout = 4, 64, 64, 96, 128
    x, dz = _act(B, H, W, cin, 3), _act(B, H, W, cout, 4)
    zT, xT = ops.to_ct(Act(dz, cout), False), ops.to_ct(Act(x, cin), True)
    out = []
    for _ in range(6):
        dw = torch.zeros(cout, 9, cin, device="cuda")
        ops.wgrad(zT, xT, B, H, W, 9, cout, cin, dw)
        out.append(dw)
    assert all(torch.equal(out[0], d) for d in out[1:])


@pytest.mark.parametrize("B,H,W,C", [(3, 128, 256, 9), (8, 128, 128, 17)])
def test_training_steps_repeat(B, H, W, C):
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand(B, C, H, W, generator=g, device="cuda")
    t = (x + 0.3 * torch.randn(B, C, H, W, generator=g, device="cuda")).contiguous()
    runs = []
    for _ in range(2):
        net = UNet(in_ch=C, base=32, seed=1)
        losses = [net.train_step(x, sample_scale(x), t, 1e-3).clone() for _ in range(4)]
        ops.check()
        runs.append(losses + [v for lay in net.layers.values() for v in (lay.w, lay.b, lay.m, lay.v)])
    assert all(torch.equal(a, b) for a, b in zip(*runs))


def test_gradients_can_be_captured():
    """The weight gradient's scratch and its launches ahead in a CUDA graph: replays give the eager bits, and each
    adds once more."""
    B, H, W, cin, cout = 4, 64, 64, 128, 128
    x, dz = _act(B, H, W, cin, 12), _act(B, H, W, cout, 13)
    wd = (0.05 * torch.randn(cin, 9, r64(cout), device="cuda")).bfloat16()
    dx = torch.zeros(B, H, W, r64(cin), dtype=torch.bfloat16, device="cuda")
    dw, db, one = (torch.zeros(cout, 9, cin, device="cuda"), torch.zeros(cout, device="cuda"),
                   torch.zeros(cout, device="cuda"))

    def grads():
        p = ops.wgrad_begin(Act(dz, cout), Act(x, cin), 9, dw, db)
        ops.conv(dz, wd, cin, dx, cin=cout)
        ops.wgrad_end(p, True)
        ops.bias_grad(Act(dz, cout), one)

    grads()
    ref = [t.clone() for t in (dw, db, one, dx)]
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream), torch.cuda.graph(graph, stream=stream):
        grads()
    torch.cuda.current_stream().wait_stream(stream)
    for _ in range(3):
        for t in (dw, db, one, dx):
            t.zero_()
        graph.replay()
        assert all(torch.equal(a, b) for a, b in zip(ref, (dw, db, one, dx)))
    graph.replay()
    assert torch.equal(db, 2 * ref[1])
    ops.check()
