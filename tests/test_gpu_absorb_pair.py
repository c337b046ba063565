"""The absorb attention kernel that takes 128 query rows per CTA pair (more than 64 heads): lengths around its 16-token groups,
64-token halves and 128-token tiles (one, two and more tiles), row counts that fill the pair, leave the odd CTA with a part or (96
heads, one request) with rows of nobody, both page sizes with NaN behind every length, and (late > 1) rope keys that grow from tile to tile,
so that references are raised behind the first.  Against the definition in 64 bits, with the parity bars."""
import dataclasses

import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu

LENGTHS = [0, 1, 15, 16, 17, 48, 63, 64, 65, 80, 112, 113, 127, 128, 129, 144, 191, 192, 193, 255, 256, 257, 385, 1000]


@pytest.mark.parametrize("H,page,Ls,late", [(128, 64, 300, 1), (128, 128, 129, 8), (80, 64, 64, 1), (96, 128, 1, 1), (112, 64, 1153, 8),
                                            (16, 64, 1100, 8), (64, 128, 1025, 1)])
@pytest.mark.parametrize("B", [len(LENGTHS), 1])
def test_lengths_and_rows(H, page, Ls, late, B):
    from paper_2509_21081_b200 import binding as b
    lens = LENGTHS if B > 1 else [129]
    cfg = I.MLAConfig("pair", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=1, seed=H + Ls)
    inp = I.make_inputs(cfg, suffix_lens=lens)
    # (in the rope keys, which enter the products as they are: larger queries would also scale the error that the 16-bit rounding
    # of the absorbed query, 2^-9 / sqrt(3) of a logit's standard deviation, makes in every weight, 4 sqrt(2) times that in the
    # worst of some thousand rows: 5e-2 at 8 times the size, above the row bar)
    grow = lambda x: torch.cat([x[:128], x[128:256] * late, x[256:] * (2 * late)])  # noqa: E731
    inp = dataclasses.replace(inp, kpe_shared=grow(inp.kpe_shared), kpe_suffix=[grow(x) for x in inp.kpe_suffix])
    ref, ref_lse = G.reference64(inp)
    for mode in (b.MODE_ABSORB, b.MODE_HYBRID):
        out, lse, _ = G.run_gpu(inp, mode, page_size=page)
        G.assert_parity(out, ref, lse, ref_lse, what=f"{mode} {H} {page} {Ls}")
