"""8-bit cache, 64-row query tile, one and two pairs of conversion warps per tensor: tile counts per CTA below, at and above
the rule's 16, odd ones, and ranges that cut heads so that segments start at odd ring positions.  Against attention in 64
bits over the exported codes; what is left are 16-bit queries and probabilities: the 16-bit path's bars."""
import pytest
import torch

from tests.gpu_harness import captured_step, worst_row

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("H,B,Ls", [(128, 5, 15 * 64), (128, 64, 16 * 64), (128, 3, 17 * 64 + 1), (16, 33, 151 * 64 + 1), (48, 64, 3400)])
def test_conversion_pairs(H, B, Ls, schedule):
    from paper_2509_21081_b200 import binding as b
    gen = torch.Generator(device="cuda").manual_seed(Ls)

    def rand(*shape, mul=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda") * mul).to(torch.bfloat16)

    ckv, kpe = rand(Ls, 512), rand(Ls, 64)
    sh = b.typhoon_mla_prepare_shared_fp8(b.make_dims(H), ckv, kpe, rand(H, 128, 512, mul=512 ** -0.5), rand(H, 128, 512, mul=512 ** -0.5))
    qn, qp = rand(B, H, 128), rand(B, H, 64)
    out = torch.full((B, H, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H), float("nan"), device="cuda")
    try:
        b.typhoon_mla_set_naive_schedule(schedule)
        ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, 0, 64), dtype=torch.uint8, device="cuda")
        b.typhoon_mla_decode(sh, qn, qp, None, None, 64, None, None, 192 ** -0.5, out, ws, mode=b.MODE_NAIVE, lse_out=lse)
    finally:
        b.typhoon_mla_set_naive_schedule(0)
    b.typhoon_mla_check_status(sh)
    kc, vc, sc = b.typhoon_mla_shared_export_fp8(sh)
    ref, ref_lse = torch.empty(B, H, 128, dtype=torch.float64, device="cuda"), torch.empty(B, H, dtype=torch.float64, device="cuda")
    for h in range(H):
        k = kc[h, :Ls].view(torch.float8_e4m3fn).float().double() * sc[0, h].double()
        v = vc[h].view(torch.float8_e4m3fn).float().double().permute(0, 2, 1).reshape(-1, 128)[:Ls] * sc[1, h].double()
        logits = (qn[:, h].double() @ k.T + qp[:, h].double() @ kpe.double().T) * 192 ** -0.5
        ref_lse[:, h] = torch.logsumexp(logits, -1)
        ref[:, h] = torch.softmax(logits, -1) @ v
    assert (torch.linalg.norm(out.double() - ref) / torch.linalg.norm(ref)).item() <= 5e-3
    assert worst_row(out, ref) <= 2e-2                     # (the row bar of the parity tests)
    assert (lse.double() - ref_lse).abs().max().item() <= 2e-2
    sh.free()


@pytest.mark.parametrize("B,Ls,pairs", [(128, 700, 1), (65, 4096, 1), (300, 700, 1), (64, 700, 1), (64, 4096, 2)])
def test_one_pair_per_tensor_runs_without_spills(B, Ls, pairs):
    """The instances with one pair of conversion warps per tensor keep everything in registers (at most 128 with 512
    threads); only the 640-thread one, at 96, does not."""
    from paper_2509_21081_b200 import binding as b
    H = 128
    z = lambda *shape: torch.zeros(*shape, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    sh = b.typhoon_mla_prepare_shared_fp8(b.make_dims(H), z(Ls, 512), z(Ls, 64), z(H, 128, 512), z(H, 128, 512))
    qn, qp, out = z(B, H, 128), z(B, H, 64), z(B, H, 128)
    ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, 0, 64), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    _, kernels = captured_step(lambda: b.typhoon_mla_decode(sh, qn, qp, None, None, 64, None, None, 192 ** -0.5, out, ws, mode=b.MODE_NAIVE))
    naive = [k for k in kernels if "naive_attn_sm100" in k["name"]]
    assert len(naive) == 1 and naive[0]["threads"] == 384 + 128 * pairs
    assert pairs == 2 or naive[0]["local_bytes"] == 0
    sh.free()


@pytest.mark.parametrize("B,Ls,walks", [(64, 1600, False), (64, 1900, True), (40, 2500, True), (65, 1200, False), (100, 1500, True)])
def test_absorb_branch_beside_an_8bit_prefix(B, Ls, walks):
    """Beside a shared-prefix kernel on 128 of 148 SMs that lasts long enough the query absorption walks through the heads on
    the other 20 (the 8-bit kernel's tiles are slower than the 16-bit one's); with one stream it takes a CTA per head.
    Same products either way: same bits."""
    from paper_2509_21081_b200 import binding as b
    H, pages = 128, 2
    gen = torch.Generator(device="cuda").manual_seed(B)

    def rand(*shape, mul=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda") * mul).to(torch.bfloat16)

    sh = b.typhoon_mla_prepare_shared_fp8(b.make_dims(H), rand(Ls, 512), rand(Ls, 64), rand(H, 128, 512, mul=0.044),
                                          rand(H, 128, 512, mul=0.044))
    table = torch.arange(B * pages, dtype=torch.int32, device="cuda").view(B, pages)
    lens = (torch.arange(B, dtype=torch.int32, device="cuda") * 37) % (64 * pages + 1)
    args = (rand(B, H, 128), rand(B, H, 64), rand(B * pages, 64, 512), rand(B * pages, 64, 64), 64, table, lens, 192 ** -0.5)
    ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, pages, 64), dtype=torch.uint8, device="cuda")
    got = {}
    for overlap in (True, False):
        out = torch.full((B, H, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        try:
            b.typhoon_mla_set_overlap(overlap)
            b.typhoon_mla_decode(sh, *args, out, ws, mode=b.MODE_HYBRID)
            b.typhoon_mla_check_status(sh)
            got[overlap] = out
            _, kernels = captured_step(lambda: b.typhoon_mla_decode(sh, *args, out, ws, mode=b.MODE_HYBRID))
        finally:
            b.typhoon_mla_set_overlap(True)
        grid = [k["grid"] for k in kernels if "q_absorb" in k["name"]]
        assert grid == [(21, 1) if walks and overlap else (1, 129)]   # (with the block that orders the requests)
    assert torch.isfinite(got[True]).all() and torch.equal(got[True], got[False])
    sh.free()
