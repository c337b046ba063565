"""More than 64 heads beside a shared-prefix launch of at most 128 rows and a narrow page table: the absorb kernel of 64 rows per CTA in
two head groups (the second with 16, 32, 48 and all 64 of its rows), suffixes around its 64-token tiles, and both sides of the line
to the pair kernel.  Against the definition in 64 bits."""
import pytest

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [80, 96, 112, 128])
@pytest.mark.parametrize("lengths", [[0, 1, 15, 16, 17, 63, 64], [64] * 65, [0, 1, 64, 65, 127, 128, 129, 192, 255, 256] * 7, [64, 128, 256, 33]])
def test_head_groups_of_short_suffixes(H, lengths):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("groups", B=len(lengths), H=H, Ls=130, suffix_lo=0, suffix_hi=1, seed=H + len(lengths)), suffix_lens=lengths)
    ref, ref_lse = G.reference64(inp)
    for page in (64, 128):
        out, lse, _ = G.run_gpu(inp, b.MODE_HYBRID, page_size=page)
        G.assert_parity(out, ref, lse, ref_lse, what=f"{H} heads, {len(lengths)} requests, pages of {page}")
