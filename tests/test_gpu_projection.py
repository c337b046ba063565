"""The projection + combine kernel in its forms, at the edges of its rule: one wave of (head, 128-row tile) pairs and one
more, half a wave (32-column items), no slot, one slot and several slots, row tiles that end in one row.

Reference: the definition in 64 bits, with the parity bars (per row, so that no column item or slot chunk of one row can hide);
the warp-MMA kernels, an implementation that shares no kernel with these, are held against it as well."""
import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu

#  heads, requests, prefix tokens, longest suffix, schedule (0 = the rule, 2 = more slots)
SHAPES = [
    (16, 1, 200, 64, 0), (16, 128, 200, 64, 0), (16, 129, 3000, 64, 0), (16, 600, 300, 64, 0),      # few pairs
    (64, 130, 200, 64, 0), (128, 128, 64, 64, 0), (128, 33, 900, 64, 2), (128, 129, 300, 64, 0),    # around one wave
    (128, 385, 260, 64, 2), (48, 37, 4000, 64, 2),
]


@pytest.mark.parametrize("H,B,Ls,hi,schedule", SHAPES)
@pytest.mark.parametrize("fp32", [False, True])
def test_projection_forms(H, B, Ls, hi, schedule, fp32):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("projection", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=hi, seed=B + H))
    pc = I.build_pages(inp)
    sh = b.typhoon_mla_prepare_shared(b.make_dims(H), inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), inp.w_uk.cuda(), inp.w_uv.cuda())
    max_pages = pc.block_table.shape[1]
    ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, max_pages, 64), dtype=torch.uint8, device="cuda")
    args = (inp.q_nope.cuda(), inp.q_pe.cuda(), pc.ckv_pages.cuda(), pc.kpe_pages.cuda(), 64, pc.block_table.cuda(),
            pc.seq_lens.cuda(), inp.scale)

    def step(mode):
        out = torch.full((B, H, 128), float("nan"), dtype=torch.float32 if fp32 else torch.bfloat16, device="cuda")
        lse = torch.full((B, H), float("nan"), device="cuda")
        if fp32:
            b.typhoon_mla_decode_partial(sh, *args, out, lse, ws, mode=mode)
        else:
            b.typhoon_mla_decode(sh, *args, out, ws, mode=mode, lse_out=lse)
        b.typhoon_mla_check_status(sh)
        return out.float(), lse

    try:
        b.typhoon_mla_set_naive_schedule(schedule)
        got = {m: step(m) for m in (b.MODE_HYBRID, b.MODE_ABSORB)}
        b.typhoon_mla_set_kernel_path(b.PATH_WARP_MMA)
        got["warp MMA"] = step(b.MODE_HYBRID)
    finally:
        b.typhoon_mla_set_kernel_path(b.PATH_TCGEN05)
        b.typhoon_mla_set_naive_schedule(0)
    ref, ref_lse = G.reference64(inp)
    for what, (out, lse) in got.items():
        G.assert_parity(out.double().cpu().numpy(), ref, lse.double().cpu().numpy(), ref_lse, what=str(what))
    sh.free()
