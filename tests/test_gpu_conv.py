"""The tcgen05 convolutions at the sizes where their geometry changes: one and several MMA tiles per
CTA, the flat position space (width up to 128) and the tiles beyond, split output channels, one and
several units of rows per CTA in the weight gradient, channel counts that leave parts of a block empty.

Inputs are exact in BF16, so against FP64 the only errors are the FP32 accumulations: relative to the
largest result 1e-5 for the FP32 outputs (as in the network's tests), plus 2^-8 relative for a BF16 one.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2209_14889_gb300 import lb
    return torch, lb


def _conv64(torch, x, w):
    """x [B, H, W, Ci], w [9, Co, Ci] (FP64) by shifted products."""
    B, H, W, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    return sum(torch.einsum("bhwc,oc->bhwo", xp[:, t // 3:t // 3 + H, t % 3:t % 3 + W], w[t]) for t in range(9))


SIZES = [(1, 1, 1, 16, 16), (2, 3, 128, 32, 24), (1, 2, 129, 16, 32), (3, 31, 33, 48, 40), (1, 70, 131, 144, 136),
         (4, 64, 64, 64, 64), (2, 130, 250, 96, 16), (5, 33, 127, 16, 128), (4, 256, 256, 32, 32)]


@pytest.mark.parametrize("B,H,W,Ci,Co", SIZES)
def test_forward_edges_vs_fp64(B, H, W, Ci, Co):
    torch, lb = _gpu()
    torch.manual_seed(B * H + W)
    x = torch.randn(B, H, W, Ci, device="cuda").to(torch.bfloat16)
    w = (torch.randn(9, Co, Ci, device="cuda") / (9 * Ci) ** 0.5).to(torch.bfloat16)
    b = torch.randn(Co, device="cuda")
    ref = _conv64(torch, x.double(), w.double()) + b.double()
    y = lb.conv3x3(x, w, b, act=False, out_f32=True)
    assert (y.double() - ref).abs().max() <= 1e-5 * ref.abs().max()
    z = lb.conv3x3(x, w, b, act=True, out_f32=False).double()
    ref = torch.where(ref > 0, ref, 0.1 * ref)
    assert torch.all((z - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * ref.abs().max())
    lb.conv_status()


@pytest.mark.parametrize("B,H,W,Ci,Co", SIZES)
def test_gradients_edges_vs_fp64(B, H, W, Ci, Co):
    torch, lb = _gpu()
    Co = (Co + 15) // 16 * 16                       # the data gradient takes multiples of 16
    torch.manual_seed(B + H * W)
    x = torch.randn(B, H, W, Ci, device="cuda").to(torch.bfloat16)
    gz = torch.randn(B, H, W, Co, device="cuda").to(torch.bfloat16)
    w = (torch.randn(9, Co, Ci, device="cuda") / (9 * Ci) ** 0.5).to(torch.bfloat16)
    ref = _conv64(torch, gz.double(), w.double().flip(0).transpose(1, 2))
    gx = lb.conv3x3_dgrad(gz, w).double()
    assert torch.all((gx - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * ref.abs().max())
    gw, gb = lb.conv3x3_wgrad(x, gz)
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    rw = torch.stack([torch.einsum("bhwo,bhwc->oc", gz.double(), xp[:, t // 3:t // 3 + H, t % 3:t % 3 + W])
                      for t in range(9)])
    assert (gw.double() - rw).abs().max() <= 1e-5 * rw.abs().max()
    rb = gz.double().sum((0, 1, 2))
    assert (gb.double() - rb).abs().max() <= 1e-5 * max(rb.abs().max().item(), 1.0)
    lb.conv_status()


def test_weight_gradient_of_few_output_channels_and_any_address():
    # Co = 8 (half an MMA column block) and results at addresses that are multiples of 4 bytes only
    torch, lb = _gpu()
    x = torch.randn(2, 9, 40, 32, device="cuda").to(torch.bfloat16)
    gz = torch.randn(2, 9, 40, 8, device="cuda").to(torch.bfloat16)
    gw, gb = lb.conv3x3_wgrad(x, gz)
    buf = torch.full((9 * 8 * 32 + 8 + 3,), 7.0, device="cuda")
    rc = lb.lib().lb_conv3x3_wgrad(x.data_ptr(), gz.data_ptr(), buf.data_ptr() + 4, buf.data_ptr() + 4 * (9 * 8 * 32 + 2),
                                   2, 9, 40, 32, 8, torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    torch.cuda.synchronize()
    n = 9 * 8 * 32
    assert torch.equal(buf[1:1 + n].reshape(gw.shape), gw) and torch.equal(buf[n + 2:n + 10], gb)
    assert buf[0] == 7.0 and buf[n + 1] == 7.0 and buf[n + 10] == 7.0


def test_data_gradient_of_two_to_the_31_pixels():
    # the size from which the mma.sync kernel takes the call: 64 GiB in, 64 GiB out; the gradient is
    # non-zero around the first and the last pixels and checked there
    torch, lb = _gpu()
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 160 << 30:
        pytest.skip("needs 160 GiB")
    torch.manual_seed(31)
    H, W, n = 32768, 65536, 20
    gz = torch.zeros(1, H, W, 16, dtype=torch.bfloat16, device="cuda")
    w = (torch.randn(9, 16, 16, device="cuda") / 12).to(torch.bfloat16)
    first, last = (torch.randn(1, n, n, 16, device="cuda").to(torch.bfloat16) for _ in range(2))
    gz[:, :n, :n] = first
    gz[:, -n:, -n:] = last
    gx = lb.conv3x3_dgrad(gz, w)
    wd = w.double().flip(0).transpose(1, 2)
    for part, got in ((first, gx[:, :n - 1, :n - 1]), (last, gx[:, 1 - n:, 1 - n:])):
        ref = _conv64(torch, part.double(), wd)
        ref = ref[:, :n - 1, :n - 1] if part is first else ref[:, 1:, 1:]
        assert ref.abs().max() > 1
        # as in test_gradients_edges_vs_fp64
        assert torch.all((got.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * ref.abs().max())
    del gz, gx
    torch.cuda.empty_cache()


@pytest.mark.parametrize("shift", [0, 1, 2, 4])
def test_network_output_at_any_address(shift):
    torch, lb = _gpu()
    n = lb.Net(1, 16, 24, seed=3)
    x = torch.randn(1, 16, 24, 16, device="cuda").to(torch.bfloat16)
    ref = n.forward(x)
    size = ref.numel() * 4
    buf = torch.full((size + 8,), 9, dtype=torch.uint8, device="cuda")
    assert lb.lib().lb_net_forward(n.n, x.data_ptr(), buf.data_ptr() + shift) == 0
    torch.cuda.synchronize()
    got = buf[shift:shift + size].clone().view(torch.float32).reshape(ref.shape)
    assert torch.equal(got, ref)
    assert (buf[:shift] == 9).all() and (buf[shift + size:] == 9).all()
    n.close()


@pytest.mark.parametrize("ldy,shift", [(25, 0), (25, 1), (24, 1), (27, 2), (24, 0)])
def test_outputs_at_odd_strides_and_addresses(ldy, shift):
    # both kernels store a BF16 output at any pixel stride and element address, and nothing beside it
    torch, lb = _gpu()
    B, H, W, Ci, Co = 2, 9, 21, 16, 24
    x = torch.randn(B, H, W, Ci, device="cuda").to(torch.bfloat16)
    w = (torch.randn(9, Co, Ci, device="cuda") / 12).to(torch.bfloat16)
    ref = _conv64(torch, x.double(), w.double())
    try:
        for kernel in (1, 0):
            lb.conv_kernel(kernel)
            buf = torch.full((B * H * W * ldy + shift + 8,), 7.0, dtype=torch.bfloat16, device="cuda")
            lb.conv3x3(x, w, None, out_f32=False, ldy=ldy, y=buf[shift:])
            torch.cuda.synchronize()
            y = buf[shift:shift + B * H * W * ldy].reshape(B, H, W, ldy)
            # as in test_forward_edges_vs_fp64
            assert torch.all((y[..., :Co].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * ref.abs().max())
            assert (y[..., Co:] == 7).all() and (buf[:shift] == 7).all() and (buf[-8:] == 7).all()
    finally:
        lb.conv_kernel(1)


def test_scratch_is_given_back():
    torch, lb = _gpu()
    x = torch.randn(1, 128, 128, 128, device="cuda").to(torch.bfloat16)
    gz = torch.randn(1, 128, 128, 96, device="cuda").to(torch.bfloat16)
    gw, gb = lb.conv3x3_wgrad(x, gz)                # partial sums of 9 x 128 x 96 for some tens of CTAs
    torch.cuda.synchronize()
    lb.conv_release()
    free0 = torch.cuda.mem_get_info()[0]
    again = lb.conv3x3_wgrad(x, gz)
    torch.cuda.synchronize()
    kept = free0 - torch.cuda.mem_get_info()[0]
    lb.conv_release()
    assert 0 < kept <= 64 << 20
    assert torch.cuda.mem_get_info()[0] >= free0
    assert torch.equal(again[0], gw) and torch.equal(again[1], gb)
