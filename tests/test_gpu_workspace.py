"""A decoder's workspace serves every step of at most the batch and page-table width it was sized for: batches on both sides of 128
(request, head) rows and of 128 query rows, narrower tables, and a batch whose own choice of partials would not fit (16 heads,
185 of 200 requests over 20000 tokens).  Against the definition in 64 bits; nothing is written behind the workspace."""
import dataclasses

import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Ls,max_batch,max_pages,lengths,batches", [
    (16, 4096, 8, 16, (0, 900), (1, 3, 4, 5, 7, 8)), (128, 1000, 8, 4, (1, 256), (5, 6)), (64, 256, 32, 4, (0, 256), (1, 2, 3, 20, 24)),
    (64, 300, 130, 3, (0, 150), (127, 128, 129)), (16, 20000, 200, 1, (0, 64), (185,)), (32, 500, 256, 2, (0, 128), (200, 255))])
def test_smaller_steps(H, Ls, max_batch, max_pages, lengths, batches):
    from paper_2509_21081_b200 import binding as b
    from paper_2509_21081_b200.decoder import TyphoonMLADecoder
    inp = I.make_inputs(I.MLAConfig("ws", B=max(batches), H=H, Ls=Ls, suffix_lo=lengths[0], suffix_hi=lengths[1], seed=H + Ls))
    pc = I.build_pages(inp, page_size=64, poison=True)
    dec = TyphoonMLADecoder(H, inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), inp.w_uk.cuda(), inp.w_uv.cuda(), inp.scale, max_batch, max_pages)
    size = dec.workspace.numel()
    ws = torch.empty(size + 4096, dtype=torch.uint8, device="cuda")
    ws[size:] = 0x5A
    dec.workspace = ws[:size]
    ref, ref_lse = G.reference64(inp)
    qn, qp, cp, kp, bt, sl = (x.cuda() for x in (inp.q_nope, inp.q_pe, pc.ckv_pages, pc.kpe_pages, pc.block_table, pc.seq_lens))
    assert bt.shape[1] <= max_pages
    wide = torch.full((bt.shape[0], max_pages), -1, dtype=torch.int32, device="cuda")
    wide[:, :bt.shape[1]] = bt
    for B in batches:
        for table in (bt, wide):
            for mode in (b.MODE_AUTO, b.MODE_ABSORB, b.MODE_HYBRID):
                lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
                out = dec.decode(qn[:B], qp[:B], cp, kp, table[:B].contiguous(), sl[:B], mode=mode, lse_out=lse)
                assert b.typhoon_mla_check_status(dec.shared) == 0
                G.assert_parity(out.float().cpu().double().numpy(), ref[:B], lse.cpu().double().numpy(), ref_lse[:B], what=f"B {B} mode {mode}")
    assert bool((ws[size:] == 0x5A).all())
    dec.close()


def test_narrower_tables_of_a_tree_step():
    """A root of more than 128 rows and two branches: sized for nine pages per request, run with one, four and nine, and without a table."""
    from paper_2509_21081_b200 import binding as b
    H, B, pages = 16, 140, 9
    root = I.make_inputs(I.MLAConfig("root", B=B, H=H, Ls=700, suffix_lo=0, suffix_hi=64 * pages, seed=11))
    branch = I.make_inputs(I.MLAConfig("branch", B=1, H=H, Ls=300, suffix_lo=0, suffix_hi=0, seed=12))
    w_uk, w_uv = root.w_uk.cuda(), root.w_uv.cuda()
    sh = [b.typhoon_mla_prepare_shared(b.make_dims(H), x.ckv_shared.cuda(), x.kpe_shared.cuda(), w_uk, w_uv) for x in (root, branch)]
    levels = [([sh[0]], [0, B]), ([sh[1], None], [0, 60, B])]
    ws = torch.empty(b.typhoon_mla_tree_workspace_bytes(levels, B, pages, 64), dtype=torch.uint8, device="cuda")
    for p in (0, 1, 4, pages):
        lens = [min(n, 64 * p) for n in root.suffix_lens]
        cut = lambda xs: [x[:n] for x, n in zip(xs, lens)]  # noqa: E731
        both = [torch.cat([y, x]) for x, y in zip(cut(root.ckv_suffix), [branch.ckv_shared] * 60 + [branch.ckv_shared[:0]] * (B - 60))]
        rope = [torch.cat([y, x]) for x, y in zip(cut(root.kpe_suffix), [branch.kpe_shared] * 60 + [branch.kpe_shared[:0]] * (B - 60))]
        ref, ref_lse = G.reference64(dataclasses.replace(root, ckv_suffix=both, kpe_suffix=rope))
        pc = I.build_pages(dataclasses.replace(root, suffix_lens=lens, ckv_suffix=cut(root.ckv_suffix), kpe_suffix=cut(root.kpe_suffix)),
                           min_max_pages=p)
        out = torch.empty(B, H, 128, dtype=torch.bfloat16, device="cuda")
        lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
        paged = [x.cuda() for x in (pc.ckv_pages, pc.kpe_pages)] if p else [None, None]
        table, seq = (pc.block_table.cuda(), pc.seq_lens.cuda()) if p else (None, None)
        b.typhoon_mla_decode_tree(levels, root.q_nope.cuda(), root.q_pe.cuda(), *paged, 64, table, seq, root.scale, out, ws, lse_out=lse)
        assert b.typhoon_mla_check_status(sh[0]) == 0
        G.assert_parity(out.float().cpu().double().numpy(), ref, lse.cpu().double().numpy(), ref_lse, what=f"{p} pages")
    for x in sh:
        x.free()
