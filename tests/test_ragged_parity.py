"""16-bit storage with token counts that are no multiple of 8: the tensor-core kernels run on rows padded to one
(GPU against the oracle, the bounds of ``util``)."""
import pytest

import __graft_entry__  # noqa: F401
import oracle
import util
from paper_2205_14756_b200 import binding, inputs

pytestmark = pytest.mark.gpu


# 49, 1, 3, 196 and 645 tokens (every residue that the copies treat apart: odd and even rows, rows shorter than a piece);
# batches whose last row ends inside a 16-byte piece; C_out > 256 / 2C' > 512 (apply and projection as two kernels)
@pytest.mark.parametrize("dtype,B,C,H,W,heads,d,c_out", [("bf16", 3, 64, 7, 7, 2, 32, 64), ("bf16", 1, 32, 1, 1, 1, 32, 32), ("f16", 2, 64, 1, 3, 4, 16, 64),
                                                         ("f16", 2, 96, 14, 14, 3, 32, 96), ("bf16", 2, 64, 15, 43, 4, 16, 40), ("bf16", 1, 64, 9, 17, 2, 32, 264),
                                                         ("bf16", 2, 288, 7, 7, 9, 32, 288), ("bf16", 1, 64, 21, 13, 3, 16, 264)])
def test_ragged_module(dtype, B, C, H, W, heads, d, c_out):
    s = inputs.ModuleShape("ragged", dtype, B, C, H, W, heads, d, seed=61)
    t = inputs.module_inputs(s)
    k = 2 * heads * d
    t["w_proj"] = inputs.quantise(inputs.normal(61, 9, c_out * k, k ** -0.5).reshape(c_out, k), dtype)
    bias = inputs.quantise(inputs.normal(61, 10, c_out, 0.5), dtype)
    ref = oracle.msla_forward(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_proj"], bias, heads=heads, d=d, eps=s.eps)
    util.assert_close(util.run_module(s, t, bias), ref, dtype, "ragged module", block=util.MODULE_BLOCK)
    assert binding.msla_debug_wait_timeouts() == 0


@pytest.mark.parametrize("dtype,B,C,H,W,Ch,c_out,residual", [("bf16", 2, 64, 7, 7, 128, 64, True), ("f16", 1, 64, 5, 9, 64, 136, False), ("bf16", 1, 32, 1, 1, 64, 32, True)])
def test_ragged_ffn(dtype, B, C, H, W, Ch, c_out, residual):
    s = inputs.FfnShape("ragged_ffn", dtype, B, C, H, W, Ch, c_out, seed=62)
    t = inputs.ffn_inputs(s)
    ref = oracle.ffn_dwconv(t["x"], t["w1"], t["w_dw"], t["w2"], t["b1"], t["b_dw"], t["b2"], act="hardswish", residual=residual)
    util.assert_close(util.run_ffn(s, t, "hardswish", residual), ref, dtype, "ragged FFN", block=util.MODULE_BLOCK)


@pytest.mark.parametrize("dtype,B,C,H,W,heads,d", [("bf16", 2, 64, 7, 9, 2, 32), ("f16", 1, 64, 14, 14, 4, 16), ("bf16", 1, 288, 5, 5, 9, 32)])
def test_ragged_block(dtype, B, C, H, W, heads, d):
    s = inputs.ModuleShape("ragged_block", dtype, B, C, H, W, heads, d, seed=63)
    t = inputs.module_inputs(s)
    f = inputs.ffn_inputs(inputs.FfnShape("ragged_block_ffn", dtype, B, C, H, W, 2 * C, C, seed=63))
    ref = oracle.evit_block(t["x"], t, f, heads=heads, d=d, act="hardswish")
    util.assert_close(util.run_block(s, t, f, 2 * C, "hardswish"), ref, dtype, "ragged block", block=util.MODULE_BLOCK)


# the two halves of the block on one workspace: the attention's padded output must not be read from memory that the FFN writes
@pytest.mark.parametrize("dtype,B,C,H,W,heads,d", [("bf16", 2, 64, 7, 9, 2, 32), ("f16", 3, 128, 14, 14, 8, 16), ("bf16", 1, 288, 5, 5, 9, 32),
                                                   ("bf16", 1, 64, 24, 24, 2, 32)])
def test_block_on_one_workspace(dtype, B, C, H, W, heads, d):
    import torch
    dt, code = util.TORCH_DTYPE[dtype], util.CODE[dtype]
    gen = torch.Generator(device="cuda").manual_seed(64)
    rnd = lambda *shape: (torch.randn(*shape, generator=gen, device="cuda") * shape[-1] ** -0.5).to(dt)
    keep = [rnd(3 * C, C), rnd(3 * C, 5, 5), rnd(3 * C, d), rnd(C, 2 * C)]
    fkeep = [rnd(4 * C, C), rnd(4 * C, 3, 3), rnd(C, 4 * C)]
    x = torch.randn(B, C, H, W, generator=gen, device="cuda").to(dt)
    attn, ffn = (lambda ws=None: binding.make_desc(B, C, H, W, heads, d, C, code, workspace=ws)), \
                (lambda ws=None: binding.make_ffn_desc(B, C, H, W, 4 * C, C, code, binding.MSLA_ACT_HARDSWISH, True, workspace=ws))
    na, nf = binding.msla_forward_workspace_bytes(attn()), binding.msla_ffn_workspace_bytes(ffn())
    scratch = lambda n: torch.zeros(n, dtype=torch.uint8, device="cuda")
    both = scratch(max(na, nf))
    outs = []
    for wa, wf in ((scratch(na), scratch(nf)), (both, both)):
        y, out = torch.empty_like(x), torch.empty_like(x)
        binding.msla_evit_block(attn(wa), binding.make_weights(*keep), ffn(wf), binding.make_ffn_weights(*fkeep), x, y, out)
        torch.cuda.synchronize()
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
