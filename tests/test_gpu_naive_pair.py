"""The shared-prefix kernel for more than 128 query rows (256 per CTA pair): row counts on both sides of the CTAs' 128 and the
pair's 256 rows and of a warp's 32, prefixes of less than a tile to some tiles (ranges that begin and end inside heads, segments of
one tile), every work decomposition, and (late > 1) rope keys that grow along the prefix, so that references are raised by either
warpgroup behind the first tile.  Against the definition in 64 bits, with the parity bars."""
import dataclasses

import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests import gpu_harness as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,B,Ls,late", [(16, 129, 1, 1), (16, 160, 127, 1), (48, 161, 128, 1), (16, 200, 129, 8), (128, 255, 300, 8), (32, 256, 1000, 8),
                                         (16, 257, 2500, 8), (64, 300, 513, 1), (16, 385, 64, 1), (16, 513, 1300, 8), (16, 800, 700, 1)])
def test_rows_and_tiles(H, B, Ls, late):
    from paper_2509_21081_b200 import binding as b
    inp = I.make_inputs(I.MLAConfig("pair", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=3, seed=H + Ls + B))
    # (in the rope keys, which enter the products as they are, not in the queries: see the absorb kernel's test)
    kpe = inp.kpe_shared
    kpe = torch.cat([kpe[:128], kpe[128:256] * late, kpe[256:512] * (2 * late), kpe[512:] * (3 * late)])
    inp = dataclasses.replace(inp, kpe_shared=kpe)
    ref, ref_lse = G.reference64(inp)
    outs = []
    try:
        for schedule in (0, 1, 2):
            b.typhoon_mla_set_naive_schedule(schedule)
            out, lse, _ = G.run_gpu(inp, b.MODE_HYBRID)
            G.assert_parity(out, ref, lse, ref_lse, what=f"schedule {schedule}")
            outs.append(out)
    finally:
        b.typhoon_mla_set_naive_schedule(0)
    assert (outs[0] == G.run_gpu(inp, b.MODE_HYBRID)[0]).all()
