"""Absorb-only steps of few (request, head) rows: one kernel for merge, projection and rounding up to one row per SM, the
merge kernel and the GEMM above (rows 128 and 144 on either side of a B200's 148 with both sides of every chunk batch: 2,
32, 33 and more chunks).  Also right behind the preparation of the prefix, where the query absorption reads its weights
before it waits.  Against the warp-MMA kernels; bars of two runs of the library."""
import pytest
import torch

from paper_2509_21081_b200 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,B", [(16, 1), (16, 8), (16, 9), (16, 10), (48, 3), (64, 2), (128, 1), (128, 2), (32, 33)])
@pytest.mark.parametrize("Ls,hi", [(0, 130), (1, 0), (64, 64), (2047, 200), (2113, 1), (9000, 64)])
def test_absorb_only(H, B, Ls, hi):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("small", B=B, H=H, Ls=max(Ls, 1), suffix_lo=min(hi, 1), suffix_hi=hi, seed=B + H + Ls))
    ckv, kpe = inp.ckv_shared[:Ls].cuda(), inp.kpe_shared[:Ls].cuda()
    pc = I.build_pages(inp)
    args = (inp.q_nope.cuda(), inp.q_pe.cuda(), pc.ckv_pages.cuda(), pc.kpe_pages.cuda(), 64, pc.block_table.cuda(),
            pc.seq_lens.cuda(), inp.scale)
    w_uk, w_uv = inp.w_uk.cuda(), inp.w_uv.cuda()
    out, lse = {}, {}
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
        finally:
            b.typhoon_mla_set_kernel_path(b.PATH_TCGEN05)
        b.typhoon_mla_check_status(sh)
        sh.free()
        out[path], lse[path] = o.float(), l
    got, ref = out[b.PATH_TCGEN05], out[b.PATH_WARP_MMA]
    assert torch.isfinite(got).all()
    assert (torch.linalg.norm(got - ref) / torch.linalg.norm(ref)).item() <= 5e-3
    assert (lse[b.PATH_TCGEN05] - lse[b.PATH_WARP_MMA]).abs().max().item() <= 2e-2
