"""A decoder's workspace serves every step of at most the batch and page-table width it was sized for: batches on both sides of 128
(request, head) rows and of 128 query rows, narrower tables, and a batch whose own choice of partials would not fit (16 heads,
185 of 200 requests over 20000 tokens).  Against the definition in 64 bits; nothing is written behind the workspace."""
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
