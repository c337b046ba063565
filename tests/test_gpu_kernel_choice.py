"""What every absorb kernel has to do, on shapes that are shown to reach it (64 query rows per CTA, or 128 per pair of CTAs): latent and
rope keys interleaved in one page array, page ids outside the cache (in a tile that the pair kernel requests ahead), both forms of
the prefix's row groups, and page tables narrower than, as wide as and wider than the prefix.  Then the shared-prefix kernel for more
than 128 rows in the allocation-free entry point, and in ranges of many one-tile segments.  Against the definition in 64 bits."""
import numpy as np
import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu

ABSORB, HYBRID, NAIVE = 1, 2, 3


def _problem(H, B, Ls, lengths, mode, pairs, min_pages=0, stacked=True):
    from paper_2509_21081_b200 import binding as b
    from paper_2509_21081_b200.decoder import TyphoonMLADecoder
    inp = I.make_inputs(I.MLAConfig("choice", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=1, seed=H + B + Ls), suffix_lens=lengths)
    pc = I.build_pages(inp, poison=True, min_max_pages=min_pages)
    pages = pc.block_table.shape[1]
    assert b.typhoon_mla_workspace_plan(H, Ls, B, pages, mode=mode, stacked=stacked)[4] == pairs
    dec = TyphoonMLADecoder(H, inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), inp.w_uk.cuda(), inp.w_uv.cuda(), inp.scale, B, pages)
    return inp, pc, dec


def _lengths(B, hi):
    return [(37 * i * i + 11 * i) % (hi + 1) for i in range(B - 1)] + [hi]


# (heads, requests, prefix, longest suffix, mode, pair kernel)
CASES = [(128, 5, 200, 1000, HYBRID, 1), (128, 5, 200, 1000, ABSORB, 1), (16, 16, 6000, 700, ABSORB, 1), (64, 16, 2048, 900, ABSORB, 1),
         (16, 37, 200, 300, ABSORB, 0), (32, 64, 100, 150, ABSORB, 0), (96, 70, 300, 250, HYBRID, 0), (64, 70, 300, 700, HYBRID, 0)]


@pytest.mark.parametrize("H,B,Ls,hi,mode,pairs", CASES)
def test_interleaved_pages(H, B, Ls, hi, mode, pairs):
    from paper_2509_21081_b200 import binding as b
    inp, pc, dec = _problem(H, B, Ls, _lengths(B, hi), mode, pairs)
    fused = torch.cat([pc.ckv_pages, pc.kpe_pages], dim=-1).contiguous().cuda()     # [P, 64, 576]
    lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
    out = dec.decode(inp.q_nope.cuda(), inp.q_pe.cuda(), fused[..., :512], fused[..., 512:], pc.block_table.cuda(), pc.seq_lens.cuda(),
                     mode=mode, lse_out=lse)
    assert b.typhoon_mla_check_status(dec.shared) == 0
    ref, ref_lse = G.reference64(inp)
    G.assert_parity(out.float().cpu().double().numpy(), ref, lse.cpu().double().numpy(), ref_lse)
    dec.close()


@pytest.mark.parametrize("bad_id", ["num_pages", "minus_one", "huge"])
@pytest.mark.parametrize("H,B,Ls,hi,mode,pairs", CASES)
def test_page_ids_outside_the_cache(H, B, Ls, hi, mode, pairs, bad_id):
    from paper_2509_21081_b200 import binding as b
    inp, pc, dec = _problem(H, B, Ls, _lengths(B, hi), mode, pairs)
    bt = pc.block_table.clone()
    bad = {"num_pages": pc.ckv_pages.shape[0], "minus_one": -1, "huge": 1 << 22}[bad_id]
    bt[B - 1, (hi + 63) // 64 - 1] = bad      # the longest request's last tile, and its second page
    bt[B - 1, 1] = bad
    lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
    args = (inp.q_nope.cuda(), inp.q_pe.cuda(), pc.ckv_pages.cuda(), pc.kpe_pages.cuda())
    out = dec.decode(*args, bt.cuda(), pc.seq_lens.cuda(), mode=mode, lse_out=lse)
    assert b.typhoon_mla_check_status(dec.shared, clear=True, raise_on_error=False) == b.STATUS_BAD_PAGE
    o = out.float().cpu().double().numpy()
    assert np.isfinite(o).all()
    keep = np.ones((B, H), dtype=bool)
    keep[B - 1] = False
    ref, ref_lse = G.reference64(inp)
    G.assert_parity(o, ref, lse.cpu().double().numpy(), ref_lse, mask=keep)
    dec.decode(*args, pc.block_table.cuda(), pc.seq_lens.cuda(), mode=mode)
    assert b.typhoon_mla_check_status(dec.shared) == 0
    dec.close()


@pytest.mark.parametrize("H,B,Ls,hi,pages,pairs", [(64, 16, 2048, 1900, 31, 1), (64, 16, 2048, 1900, 32, 1), (64, 16, 2048, 1900, 33, 0),
                                                   (16, 37, 1100, 150, 3, 0), (48, 5, 1100, 150, 3, 1), (128, 3, 1100, 150, 3, 1)])
def test_row_groups_and_table_widths(H, B, Ls, hi, pages, pairs):
    from paper_2509_21081_b200 import binding as b
    inp, pc, dec = _problem(H, B, Ls, _lengths(B, hi), ABSORB, pairs, min_pages=pages)
    ref, ref_lse = G.reference64(inp)
    try:
        for stacked in (True, False):
            b.typhoon_mla_set_stacked_absorb(stacked)
            lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
            out = dec.decode(inp.q_nope.cuda(), inp.q_pe.cuda(), pc.ckv_pages.cuda(), pc.kpe_pages.cuda(), pc.block_table.cuda(),
                             pc.seq_lens.cuda(), mode=ABSORB, lse_out=lse)
            assert b.typhoon_mla_check_status(dec.shared) == 0
            G.assert_parity(out.float().cpu().double().numpy(), ref, lse.cpu().double().numpy(), ref_lse, what=f"stacked {stacked}")
    finally:
        b.typhoon_mla_set_stacked_absorb(True)
        dec.close()


@pytest.mark.parametrize("H,B,Ls", [(32, 200, 1500), (16, 300, 130)])
def test_allocation_free_entry_point_above_128_rows(H, B, Ls):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("noalloc", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=0, seed=H + B))
    w_uk, w_uv = inp.w_uk.cuda(), inp.w_uv.cuda()
    sh = b.typhoon_mla_prepare_shared(b.make_dims(H), inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), w_uk, w_uv)
    out = torch.full((B, H, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H), float("nan"), dtype=torch.float32, device="cuda")
    b.typhoon_mla_naive_shared_noalloc(sh, inp.q_nope.cuda(), inp.q_pe.cuda(), inp.scale, out, lse)
    assert b.typhoon_mla_check_status(sh) == 0
    ref, ref_lse = G.reference64(inp)
    G.assert_parity(out.float().cpu().double().numpy(), ref, lse.cpu().double().numpy(), ref_lse)
    sh.free()


def test_many_one_tile_segments_per_range():
    from paper_2509_21081_b200 import binding as b
    H, B, Ls = 128, 1024, 100
    assert b.typhoon_mla_naive_plan(H, B, Ls)[0] == 128 and b.typhoon_mla_naive_plan(H, B, Ls, 2)[1] == 18    # seven or eight heads each
    inp = I.make_inputs(I.MLAConfig("segments", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=2, seed=5))
    ref, ref_lse = G.reference64(inp)
    try:
        for schedule in (0, 2):
            b.typhoon_mla_set_naive_schedule(schedule)
            out, lse, _ = G.run_gpu(inp, HYBRID)
            G.assert_parity(out, ref, lse, ref_lse, what=f"schedule {schedule}")
    finally:
        b.typhoon_mla_set_naive_schedule(0)
