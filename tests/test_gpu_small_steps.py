"""Absorb-only steps of few (request, head) rows: one kernel for merge, projection and rounding up to one row per SM, the
merge kernel and the GEMM above (rows 128 and 144 on either side of a B200's 148; with 16 heads and one request every 64
tokens are a chunk: 2, 32, 33 and 142 of them, on both sides of a pass of 32).  Also right behind the preparation of the prefix,
where the query absorption reads its weights before it waits.  Against the definition in 64 bits, with the parity bars; the
warp-MMA kernels, which merge with the same kernel up to one row per SM, are held against it as well."""
import dataclasses

import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu

SHAPES = [(H, B, Ls, hi) for H, B in [(16, 1), (16, 8), (16, 9), (16, 10), (48, 3), (64, 2), (128, 1), (128, 2), (32, 33)]
          for Ls, hi in [(0, 130), (1, 0), (64, 64), (2047, 200), (2113, 1), (9000, 64)]] + [(16, 1, 1984, 64), (16, 1, 2048, 64)]


@pytest.mark.parametrize("H,B,Ls,hi", SHAPES)
def test_absorb_only(H, B, Ls, hi):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("small", B=B, H=H, Ls=max(Ls, 1), suffix_lo=min(hi, 1), suffix_hi=hi, seed=B + H + Ls))
    inp = dataclasses.replace(inp, ckv_shared=inp.ckv_shared[:Ls], kpe_shared=inp.kpe_shared[:Ls])
    ckv, kpe = inp.ckv_shared.cuda(), inp.kpe_shared.cuda()
    pc = I.build_pages(inp)
    args = (inp.q_nope.cuda(), inp.q_pe.cuda(), pc.ckv_pages.cuda(), pc.kpe_pages.cuda(), 64, pc.block_table.cuda(),
            pc.seq_lens.cuda(), inp.scale)
    w_uk, w_uv = inp.w_uk.cuda(), inp.w_uv.cuda()
    ref, ref_lse = G.reference64(inp)
    sh = b.typhoon_mla_prepare_shared(b.make_dims(H), ckv, kpe, w_uk, w_uv)
    ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, pc.block_table.shape[1], 64), dtype=torch.uint8, device="cuda")
    sh.free()
    for path in (b.PATH_WARP_MMA, b.PATH_TCGEN05):
        o = torch.full((B, H, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        l = torch.full((B, H), float("nan"), device="cuda")
        torch.cuda.synchronize()
        try:
            b.typhoon_mla_set_kernel_path(path)
            sh = b.typhoon_mla_prepare_shared(b.make_dims(H), ckv, kpe, w_uk, w_uv)
            b.typhoon_mla_decode(sh, *args, o, ws, mode=b.MODE_ABSORB, lse_out=l)
            launches = b.typhoon_mla_last_launch_count()
        finally:
            b.typhoon_mla_set_kernel_path(b.PATH_TCGEN05)
        b.typhoon_mla_check_status(sh)
        sh.free()
        G.assert_parity(o.double().cpu().numpy(), ref, l.double().cpu().numpy(), ref_lse, what=f"path {path}")
        if path == b.PATH_TCGEN05:   # absorption, attention and one kernel behind them, or two
            assert launches <= (3 if B * H <= 148 else 4)
