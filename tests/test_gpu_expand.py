"""Prefix expansion at the edges of its work split: fewer units than SMs, ranges that cross from one row tile to the next,
one token of padding and one of data in the last tile.  Against the product in 64 bits: fp32 sums of 512 products rounded to
bf16 are within one unit in the last place (2^-8 relative), plus 512 * 2^-24 of the absolute sum where terms cancel."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,Ls", [(16, 1), (16, 129), (16, 1281), (48, 5000), (128, 127), (128, 300)])
def test_expansion(H, Ls):
    from paper_2509_21081_b200 import binding as b
    gen = torch.Generator(device="cuda").manual_seed(H + Ls)
    ckv, kpe = (torch.randn(Ls, n, generator=gen, device="cuda").to(torch.bfloat16) for n in (512, 64))
    w_uk, w_uv = ((torch.randn(H, 128, 512, generator=gen, device="cuda") * 512 ** -0.5).to(torch.bfloat16) for _ in range(2))
    sh = b.typhoon_mla_prepare_shared(b.make_dims(H), ckv, kpe, w_uk, w_uv)
    k, v = b.typhoon_mla_shared_export(sh)
    b.typhoon_mla_check_status(sh)
    Lp = k.shape[1] * 64
    rows = torch.zeros(Lp, 512, dtype=torch.float64, device="cuda")
    rows[:Ls] = ckv.double()
    for h in range(H):
        got_k = k[h].double().permute(0, 2, 1, 3).reshape(Lp, 128)
        got_v = v[h].double().permute(0, 2, 1).reshape(Lp, 128)
        for got, w in ((got_k, w_uk[h].double()), (got_v, w_uv[h].double())):
            ref, mag = rows @ w.T, rows.abs() @ w.abs().T
            assert ((got - ref).abs() <= ref.abs() * 2 ** -8 + mag * 2 ** -15).all()
    sh.free()
