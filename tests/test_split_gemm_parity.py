"""The fp32 projections on tensor cores (three bf16 pieces per operand) at the edges of tiles, slices and fetch modes, against 64-bit products."""
import pytest
import torch
import torch.nn.functional as F

import __graft_entry__  # noqa: F401
import util
from paper_2205_14756_b200 import binding, inputs

pytestmark = pytest.mark.gpu

# Bound per element, in units of sum_k |a_k b_k|: the three products left out 2^-23; at most 16 truncating additions to an accumulator per chunk
# (256 k at most), each below 2^-23 of what it holds, and one rounding (2^-24) per chunk: 16 * 2^-23 + 2^-23 + 2^-22 < 2^-18.
BOUND = 2.0 ** -18


def check(got, x, w, bias=None):
    ref = torch.einsum("ok,bkn->bon", w.double(), x.double())
    size = torch.einsum("ok,bkn->bon", w.double().abs(), x.double().abs())
    if bias is not None:
        ref = ref + bias.double()[None, :, None]
        size = size + bias.double().abs()[None, :, None]
    assert torch.all((got.double() - ref).abs() <= BOUND * size)
    return float((got.double() - ref).norm() / ref.norm())


def offset(t, floats):
    """The same values `floats` floats past a 256-byte boundary: runs of eight that are 16- but not 32-byte aligned."""
    buf = torch.empty(t.numel() + floats, device="cuda")
    v = buf[floats:].view(t.shape)
    v.copy_(t)
    return v


# rows of tokens that are a multiple of eight, of four and of nothing; ragged tiles on either side; K below, at and beyond a slice of 64 and a
# chunk of 128; fewer tiles than SMs and several per SM
@pytest.mark.parametrize("B,N,C,Cout,d,off", [(1, 8192, 192, 576, 32, 0), (2, 4100, 72, 96, 16, 0), (3, 1023, 264, 192, 32, 0), (1, 1025, 520, 160, 16, 0), (5, 776, 128, 96, 32, 4),
                                              (40, 196, 64, 96, 32, 0), (1, 262144, 8, 32, 32, 0)])
def test_input_projection(B, N, C, Cout, d, off):
    g = torch.Generator(device="cuda").manual_seed(7)
    x, w = offset(torch.randn(B, C, N, generator=g, device="cuda"), off), offset(torch.randn(Cout, C, generator=g, device="cuda"), off)
    assert B * N * C * Cout >= 1 << 24
    y = torch.full((B, Cout // d, N, d), float("nan"), device="cuda")
    binding.msla_project_in(binding.MSLA_F32, x, w, y, B, C, Cout, N, d)
    torch.cuda.synchronize()
    # no less accurate than products and sums in fp32: about 2^-24 sqrt(K / 2) for an fp32 chain of K, 2e-7 at K = 64 .. 512
    assert check(y.permute(0, 1, 3, 2).reshape(B, Cout, N), x, w) <= 3e-7
    assert binding.msla_debug_wait_timeouts() == 0


@pytest.mark.parametrize("B,N,Cin,Cout,off", [(1, 8192, 384, 192, 0), (2, 4099, 80, 104, 0), (3, 1023, 264, 24, 0), (7, 130, 1032, 72, 4), (1, 65537, 32, 8, 0)])
def test_output_projection(B, N, Cin, Cout, off):
    g = torch.Generator(device="cuda").manual_seed(8)
    a, w = offset(torch.randn(B, N, Cin, generator=g, device="cuda"), off), torch.randn(Cout, Cin, generator=g, device="cuda")
    bias, y = torch.randn(Cout, generator=g, device="cuda"), torch.full((B, Cout, N), float("nan"), device="cuda")
    assert B * N * Cin * Cout >= 1 << 24
    binding.msla_project_out(binding.MSLA_F32, a, w, bias, y, B, Cin, Cout, N)
    torch.cuda.synchronize()
    assert check(y, a.transpose(1, 2), w, bias) <= 3e-7


# values at the ends of the exponent range: the largest finite ones stay finite in pieces, and channels of zeros beside them add nothing
def test_largest_values():
    B, N, C, Cout = 1, 4096, 64, 96
    x = torch.zeros(B, C, N, device="cuda")
    x[:, 0], x[:, 1] = torch.finfo(torch.float32).min, 1e-30
    w = torch.zeros(Cout, C, device="cuda")
    w[:, 0], w[:, 1] = torch.linspace(-1.0, 1.0, Cout, device="cuda"), 2.0 ** 99
    y = torch.empty(B, Cout // 32, N, 32, device="cuda")
    binding.msla_project_in(binding.MSLA_F32, x, w, y, B, C, Cout, N, 32)
    torch.cuda.synchronize()
    assert torch.isfinite(y).all()
    check(y.permute(0, 1, 3, 2).reshape(B, Cout, N), x, w)


# both layers of the FFN: bias, the three activations and the residual, on rows in every fetch mode
@pytest.mark.parametrize("B,C,H,W,Ch,act", [(1, 64, 48, 64, 256, "hardswish"), (2, 72, 33, 31, 288, "relu"), (1, 96, 30, 46, 200, "identity")])
def test_ffn_layers(B, C, H, W, Ch, act):
    s = inputs.FfnShape("split_ffn", "f32", B, C, H, W, Ch, C, seed=91)
    t = inputs.ffn_inputs(s)
    dd = {k: torch.from_numpy(v).double() for k, v in t.items()}
    f = {"hardswish": F.hardswish, "relu": F.relu, "identity": lambda v: v}[act]
    h = f(F.conv2d(dd["x"], dd["w1"].reshape(Ch, C, 1, 1), dd["b1"]))
    h = f(F.conv2d(h, dd["w_dw"].reshape(Ch, 1, 3, 3), dd["b_dw"], padding=1, groups=Ch))
    ref = (F.conv2d(h, dd["w2"].reshape(C, Ch, 1, 1), dd["b2"]) + dd["x"]).numpy()
    util.assert_close(util.run_ffn(s, t, act, True), ref, "f32", "fp32 FFN on tensor cores")
