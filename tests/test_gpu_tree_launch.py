"""Trees whose prefixes share a launch: every group's rows against an ordinary step of those rows alone.

Sizes: one tile and a ragged second one, one row and a full 64-row / 128-row group, more prefixes than one launch holds, a
group too large to share a launch (129 rows) and one with 8-bit storage beside the shared ones.  Both sides round the
probabilities and the result to 16 bits and differ in the order of fp32 sums and in the reference exponents only: the bars
are those of two runs of the library (relative Frobenius 5e-3, log-sum-exp 2e-2)."""
import pytest
import torch

from tests.gpu_harness import worst_row

pytestmark = pytest.mark.gpu

CASES = {
    "two": (16, [(1, 64, False), (63, 65, False)]),
    "half and full row tiles": (32, [(64, 700, False), (65, 129, False), (128, 1, False)]),
    "more than one launch": (16, [(1 + i % 5, 1 + 97 * i, False) for i in range(19)]),
    "beside unshared ones": (16, [(129, 300, False), (3, 500, False), (20, 260, True), (17, 1000, False)]),
}


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("case", sorted(CASES))
def test_prefixes_that_share_a_launch(case, schedule):
    from paper_2509_21081_b200 import binding as b
    H, groups = CASES[case]
    gen = torch.Generator(device="cuda").manual_seed(7)

    def rand(*shape, mul=1.0):
        return (torch.randn(*shape, generator=gen, device="cuda") * mul).to(torch.bfloat16)

    dims, B = b.make_dims(H), sum(g[0] for g in groups)
    w_uk, w_uv = rand(H, 128, 512, mul=512 ** -0.5), rand(H, 128, 512, mul=512 ** -0.5)
    qn, qp = rand(B, H, 128), rand(B, H, 64)
    root = b.typhoon_mla_prepare_shared(dims, rand(333, 512), rand(333, 64), w_uk, w_uv)
    parts, begin = [], [0]
    for rows, tokens, fp8 in groups:
        prepare = b.typhoon_mla_prepare_shared_fp8 if fp8 else b.typhoon_mla_prepare_shared
        parts.append(prepare(dims, rand(tokens, 512), rand(tokens, 64), w_uk, w_uv))
        begin.append(begin[-1] + rows)

    def tree(levels, r0, r1):
        ws = torch.empty(b.typhoon_mla_tree_workspace_bytes(levels, r1 - r0, 0, 64), dtype=torch.uint8, device="cuda")
        out = torch.full((r1 - r0, H, 128), float("nan"), dtype=torch.bfloat16, device="cuda")
        lse = torch.full((r1 - r0, H), float("nan"), device="cuda")
        b.typhoon_mla_decode_tree(levels, qn[r0:r1], qp[r0:r1], None, None, 64, None, None, 192 ** -0.5, out, ws, lse_out=lse)
        return out.float(), lse

    try:
        b.typhoon_mla_set_naive_schedule(schedule)
        got, got_lse = tree([([root], [0, B]), (parts, begin)], 0, B)
        flat, flat_lse = tree([(parts, begin)], 0, B)
        b.typhoon_mla_check_status(root)
    finally:
        b.typhoon_mla_set_naive_schedule(0)
    for i, part in enumerate(parts):
        r0, r1 = begin[i], begin[i + 1]
        o1, l1 = tree([([part], [0, r1 - r0])], r0, r1)                 # this prefix alone
        o0, l0 = tree([([root], [0, r1 - r0])], r0, r1)                 # the root alone, merged in fp32 here
        l = torch.logaddexp(l0, l1)
        o = o0 * torch.exp(l0 - l)[..., None] + o1 * torch.exp(l1 - l)[..., None]
        for a, c, la, lc in ((flat[r0:r1], o1, flat_lse[r0:r1], l1), (got[r0:r1], o, got_lse[r0:r1], l)):
            assert torch.isfinite(a).all()
            assert (torch.linalg.norm(a - c) / torch.linalg.norm(c)).item() <= 5e-3
            assert worst_row(a, c) <= 2e-2                 # (the row bar of the parity tests)
            assert (la - lc).abs().max().item() <= 2e-2
    for h in parts + [root]:
        h.free()
