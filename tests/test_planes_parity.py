"""The 16-bit module on channel-blocked planes (many tokens, rows of whole pixel octets): GPU against the oracle at the sizes where
a tile, a border or a dispatch can go wrong.  All shapes lie above the size from which that path is taken."""
import numpy as np
import pytest

import __graft_entry__  # noqa: F401
import oracle
import util
from paper_2205_14756_b200 import binding, inputs

pytestmark = pytest.mark.gpu


# two image rows and a very wide image; rows of one octet; widths of 16 k + 8 and 16 k; ragged last tile rows; odd head counts (d = 16:
# half-empty blocks); runs of tiles that cross images and heads; 2C' > 512 (apply and projection apart); C_out != C with a bias
@pytest.mark.parametrize("dtype,B,C,H,W,heads,d,c_out", [("bf16", 1, 32, 2, 81920, 1, 32, 32), ("bf16", 320, 32, 66, 8, 1, 32, 32), ("f16", 2, 48, 235, 232, 3, 16, 48),
                                                         ("bf16", 1, 96, 239, 248, 3, 32, 40), ("bf16", 3, 64, 112, 256, 4, 16, 264), ("f16", 40, 288, 15, 32, 9, 32, 288),
                                                         ("f16", 21, 64, 66, 64, 2, 32, 64), ("bf16", 52, 288, 15, 24, 9, 32, 288)])
def test_planes_module(dtype, B, C, H, W, heads, d, c_out):
    s = inputs.ModuleShape("planes", dtype, B, C, H, W, heads, d, seed=81)
    t = inputs.module_inputs(s)
    k = 2 * heads * d
    t["w_proj"] = inputs.quantise(inputs.normal(81, 9, c_out * k, k ** -0.5).reshape(c_out, k), dtype)
    bias = inputs.quantise(inputs.normal(81, 10, c_out, 0.5), dtype)
    ref = oracle.msla_forward(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_proj"], bias, heads=heads, d=d, eps=s.eps)
    got = util.run_module(s, t, bias)
    util.assert_close(got, ref, dtype, "planes", block=util.MODULE_BLOCK)
    assert np.array_equal(got, util.run_module(s, t, bias))  # bit for bit from run to run
    assert binding.msla_debug_wait_timeouts() == 0


# three branches (two aggregation launches, the second without the un-aggregated scale), a 3x3 filter, fused and apart.  d = 32
# only: a query row of 16 entries has none above zero with probability 2^-16, and among 10^6 rows some have nothing but an entry
# of the size of the projected query's rounding error, whose quotient bf16 does not determine (the token-major kernels give the
# same value there); with 32 entries that takes 2^-32.
@pytest.mark.parametrize("C,H,W,heads,d,k1,k2", [(64, 240, 344, 2, 32, 5, 3), (192, 160, 176, 6, 32, 3, 5), (96, 240, 232, 3, 32, 3, 3)])
def test_planes_three_branches(C, H, W, heads, d, k1, k2):
    s = inputs.ModuleShape("planes3", "bf16", 1, C, H, W, heads, d, seed=82, n_scales=3, agg_kernel=k1, agg_kernel2=k2)
    t = inputs.module_inputs(s)
    ref = oracle.msla_forward3(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_dw2"], t["w_pw2"], t["w_proj"], heads=heads, d=d)
    util.assert_close(util.run_module(s, t), ref, "bf16", "planes, three branches", block=util.MODULE_BLOCK)


# d = 16: three branches and 3x3 filters.  The queries of scale 0 get a positive mean (a constant channel of x), so that no row is without
# an entry well above zero (see above).
@pytest.mark.parametrize("dtype,C,H,W,heads,n_scales,k1,k2", [("bf16", 64, 240, 344, 4, 3, 5, 3), ("f16", 96, 240, 232, 6, 3, 3, 5),
                                                              ("bf16", 80, 240, 280, 5, 2, 3, 5), ("f16", 32, 416, 400, 2, 2, 3, 5)])
def test_planes_of_narrow_heads(dtype, C, H, W, heads, n_scales, k1, k2):
    s = inputs.ModuleShape("planes16", dtype, 1, C, H, W, heads, 16, seed=85, n_scales=n_scales, agg_kernel=k1, agg_kernel2=k2)
    t = inputs.module_inputs(s)
    t["x"][:, 0] = 4.0
    t["w_qkv"].reshape(heads, 3, 16, C)[:, 0, :, 0] = 0.5
    if n_scales == 3:
        ref = oracle.msla_forward3(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_dw2"], t["w_pw2"], t["w_proj"], heads=heads, d=16)
    else:
        ref = oracle.msla_forward(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_proj"], heads=heads, d=16, eps=s.eps)
    util.assert_close(util.run_module(s, t), ref, dtype, "planes, d = 16", block=util.MODULE_BLOCK)
    assert binding.msla_debug_wait_timeouts() == 0


def test_planes_block():
    s = inputs.ModuleShape("planes_block", "bf16", 2, 64, 200, 208, 2, 32, seed=83)
    t = inputs.module_inputs(s)
    f = inputs.ffn_inputs(inputs.FfnShape("planes_block_ffn", "bf16", 2, 64, 200, 208, 128, 64, seed=83))
    ref = oracle.evit_block(t["x"], t, f, heads=2, d=32, act="hardswish")
    util.assert_close(util.run_block(s, t, f, 128, "hardswish"), ref, "bf16", "planes block", block=util.MODULE_BLOCK)


# bands of one image, each above the line: rows outside the band's own do not count in its states, queries start at a row
@pytest.mark.parametrize("c_out", [64, 264])
def test_planes_bands(c_out):
    from test_sharded import _run_bands
    s = inputs.ModuleShape("planes_bands", "bf16", 1, 64, 500, 344, 2, 32, seed=84)
    t = inputs.module_inputs(s)
    k = 2 * 64
    t["w_proj"] = inputs.quantise(inputs.normal(84, 9, c_out * k, k ** -0.5).reshape(c_out, k), "bf16")
    ref = oracle.msla_forward(t["x"], t["w_qkv"], t["w_dw"], t["w_pw"], t["w_proj"], heads=2, d=32)
    got, _ = _run_bands(t, s, 2, "bf16")
    util.assert_close(got, ref, "bf16", "planes bands", block=util.MODULE_BLOCK)
