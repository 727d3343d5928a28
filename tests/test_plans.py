"""What the library reserves and how it cuts a call, checked on the host: every call here is refused for a null pointer before
anything is launched, and the status says whether the planning before that check found anything wrong."""
import ctypes
import random

import __graft_entry__  # noqa: F401
from paper_2205_14756_b200 import binding

FAKE = 1 << 20            # an aligned address that nothing reads
NULL_POINTER = 1          # MSLA_ERR_INVALID_ARG; a plan that does not fit answers 4


def _desc(dtype, B, C, H, W, d, n_scales=2, nbytes=None):
    desc = binding.make_desc(B, C, H, W, C // d, d, C, dtype, n_scales=n_scales, agg_kernel2=3)
    desc.workspace, desc.workspace_bytes = FAKE, nbytes or 0
    return desc


def test_parts_of_a_host_call_fit_the_reservation_of_the_batch():
    """msla_forward_host runs a batch in parts; each must fit what msla_forward_host_workspace_bytes reserved for the whole."""
    lib, rng = binding.lib(), random.Random(1)
    shapes = [(2, 128, 128, 256, 32), (3, 256, 64, 112, 32), (2, 64, 256, 256, 32), (2, 64, 128, 384, 32), (16, 256, 64, 64, 32)]
    shapes += [(rng.randint(2, 64), 32 * rng.randint(2, 12), rng.randint(7, 512), rng.choice([rng.randint(7, 512), 16 * rng.randint(1, 32)]),
                rng.choice([16, 32])) for _ in range(4000)]
    w = binding.msla_weights()
    for B, C, H, W, d in shapes:
        if B * C * H * W > 40 << 20:
            continue
        for dtype in (binding.MSLA_BF16, binding.MSLA_F32):
            for n_scales in (2, 3):
                desc = _desc(dtype, B, C, H, W, d, n_scales)
                need = lib.msla_forward_host_workspace_bytes(ctypes.byref(desc))
                assert need > 0
                desc.workspace_bytes = need
                st = lib.msla_forward_host(ctypes.byref(desc), None, ctypes.byref(w), None, None)
                assert st == NULL_POINTER, (B, C, H, W, d, dtype, n_scales, lib.msla_last_error())


def test_a_host_call_that_its_parts_would_refuse_copies_nothing():
    """A null or misaligned weight is found before the first copy (on a machine without a GPU: before the device is looked for)."""
    import torch
    lib = binding.lib()
    B, C, H, W, d = 6, 64, 64, 96, 32
    x, out = torch.zeros(B, C, H, W, dtype=torch.bfloat16), torch.zeros(B, C, H, W, dtype=torch.bfloat16)
    need = binding.msla_forward_host_workspace_bytes(_desc(binding.MSLA_BF16, B, C, H, W, d))
    # real buffers: a GPU's where there is one (the call is refused all the same)
    device = "cuda" if torch.cuda.is_available() else "cpu"
    ws = torch.full((need + 256,), 0xA5, dtype=torch.uint8, device=device)
    wt = torch.zeros(1 << 20, dtype=torch.bfloat16, device=device)
    desc = _desc(binding.MSLA_BF16, B, C, H, W, d, nbytes=need)
    desc.workspace = (ws.data_ptr() + 255) // 256 * 256
    fields = ("w_qkv", "w_dw", "w_pw", "w_proj")
    for field, value, status in [("w_dw", None, 1), ("w_proj", None, 1), ("w_pw", wt.data_ptr() + 2, 3), ("b_proj", wt.data_ptr() + 8, 3)]:
        w = binding.msla_weights()
        for f in fields:
            setattr(w, f, wt.data_ptr())
        setattr(w, field, value)
        assert lib.msla_forward_host(ctypes.byref(desc), x.data_ptr(), ctypes.byref(w), out.data_ptr(), None) == status, field
    if device == "cuda":
        torch.cuda.synchronize()
    assert bool((ws == 0xA5).all())


def test_bands_fit_the_reservation_of_the_band_with_its_halo():
    """msla_band_states splits the band's own tokens, whose number of chunks may exceed that of the band with its halo."""
    lib, rng = binding.lib(), random.Random(2)
    shapes = [(2, 256, 54, 64, 32, 2, 0), (2, 256, 56, 64, 32, 2, 2), (1, 32, 9, 57, 32, 2, 2)]
    shapes += [(rng.randint(1, 40), 32 * rng.randint(1, 12), rng.randint(5, 300), rng.randint(1, 300), rng.choice([16, 32]), rng.choice([0, 2]),
                rng.choice([0, 2])) for _ in range(20000)]
    w = binding.msla_weights()
    for B, C, H, W, d, top, bottom in shapes:
        for dtype in (binding.MSLA_BF16, binding.MSLA_F32):
            desc = _desc(dtype, B, C, H, W, d)
            desc.workspace_bytes = lib.msla_forward_workspace_bytes(ctypes.byref(desc))
            st = lib.msla_band_states(ctypes.byref(desc), None, ctypes.byref(w), top, bottom, None, None)
            assert st == NULL_POINTER, (B, C, H, W, d, top, bottom, lib.msla_last_error())


def test_workspaces_do_not_shrink_as_feature_maps_grow():
    """A workspace sized for the largest batch, height and width serves every smaller one: whole forward, host call and FFN."""
    lib, rng = binding.lib(), random.Random(3)
    widths = [(256, 32, 2), (128, 16, 2), (384, 32, 2), (64, 32, 3), (96, 16, 3)]  # the third: apply and projection apart
    shapes = [(1, 128, 152, 1, 128, 160), (64, 14, 14, 64, 14, 16), (64, 7, 7, 64, 7, 8), (1, 250, 255, 1, 250, 256), (21, 66, 64, 22, 66, 64)]
    for _ in range(4000):
        B, H, W = rng.randint(1, 40), rng.randint(1, 260), rng.randint(1, 260)
        i, by = rng.randrange(3), rng.choice([1, 1, 2, 7, 8, 30])
        shapes.append((B, H, W) + tuple(v + (by if j == i else 0) for j, v in enumerate((B, H, W))))

    def answers(dtype, C, d, S, B, H, W):
        desc, ffn = _desc(dtype, B, C, H, W, d, S), binding.make_ffn_desc(B, C, H, W, C + 64, C, dtype)
        return [lib.msla_forward_workspace_bytes(ctypes.byref(desc)), lib.msla_forward_host_workspace_bytes(ctypes.byref(desc)),
                lib.msla_ffn_workspace_bytes(ctypes.byref(ffn))]

    for B0, H0, W0, B1, H1, W1 in shapes:
        for C, d, S in widths:
            for dtype in (binding.MSLA_BF16, binding.MSLA_F32):
                small, large = answers(dtype, C, d, S, B0, H0, W0), answers(dtype, C, d, S, B1, H1, W1)
                assert min(small) > 0 and all(a <= b for a, b in zip(small, large)), (B0, H0, W0, B1, H1, W1, C, d, S, dtype, small, large)


def test_a_block_that_its_second_half_would_refuse_runs_nothing():
    """The FFN's arguments are checked before the attention is launched (without a GPU: before the device is looked for)."""
    import torch
    lib = binding.lib()
    B, C, H, W, d = 1, 64, 8, 8, 32
    device = "cuda" if torch.cuda.is_available() else "cpu"
    x, y, out = (torch.zeros(B, C, H, W, dtype=torch.bfloat16, device=device) for _ in range(3))
    wt = torch.zeros(1 << 20, dtype=torch.bfloat16, device=device)
    ws = torch.full((8 << 20,), 0xA5, dtype=torch.uint8, device=device)
    base = (ws.data_ptr() + 255) // 256 * 256
    desc = _desc(binding.MSLA_BF16, B, C, H, W, d)
    desc.workspace, desc.workspace_bytes = base, lib.msla_forward_workspace_bytes(ctypes.byref(desc))
    w, fw = binding.msla_weights(), binding.msla_ffn_weights()
    w.w_qkv = w.w_dw = w.w_pw = w.w_proj = wt.data_ptr()
    for w2, short, status in [(None, 0, 1), (wt.data_ptr() + 2, 0, 3), (wt.data_ptr(), 1, 4)]:
        ffn = binding.make_ffn_desc(B, C, H, W, 4 * C, C, binding.MSLA_BF16, residual=True)
        need = lib.msla_ffn_workspace_bytes(ctypes.byref(ffn))
        ffn.workspace, ffn.workspace_bytes = base + (4 << 20), need - short
        assert need <= 3 << 20
        fw.w1, fw.w_dw, fw.w2 = wt.data_ptr(), wt.data_ptr(), w2
        assert lib.msla_evit_block(ctypes.byref(desc), ctypes.byref(w), ctypes.byref(ffn), ctypes.byref(fw), x.data_ptr(), y.data_ptr(),
                                   out.data_ptr(), None) == status
    if device == "cuda":
        torch.cuda.synchronize()
    assert bool((ws == 0xA5).all())


def test_plan_of_a_forward():
    """Which steps are one kernel, for every storage type, and the stages that the benchmark counts bytes for."""
    import bench
    plan = lambda dtype, C, H, W, heads, d, B=1: binding.msla_forward_plan(binding.make_desc(B, C, H, W, heads, d, C, dtype))
    apply, states = binding.MSLA_PLAN_FUSES_APPLY, binding.MSLA_PLAN_FUSES_STATES
    for dtype in (binding.MSLA_BF16, binding.MSLA_F16):
        assert plan(dtype, 256, 512, 512, 8, 32) == apply | states
        assert plan(dtype, 256, 512, 511, 8, 32) == apply           # rows of no whole octets
        assert plan(dtype, 256, 32, 32, 8, 32) == apply             # few tokens
        assert plan(dtype, 384, 256, 256, 12, 32) == states         # too many channels for the fused output kernel
        assert plan(dtype, 288, 7, 7, 9, 32) == 0
    assert plan(binding.MSLA_F32, 256, 512, 512, 8, 32) == 0
    assert plan(binding.MSLA_BF16, 60, 8, 8, 1, 32) == -1
    assert bench.plan_stages(0) == bench.STAGES and bench.plan_stages(apply) == bench.STAGES_FUSED
    assert bench.plan_stages(apply | states) == ("project_in", "aggregate_kv_state", "apply_project")
    assert bench.plan_stages(states) == ("project_in", "aggregate_kv_state", "apply", "project_out")
