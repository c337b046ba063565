"""CPU-only tests of the library's host side: the shared object loads and exports every symbol the
header declares; cost model and Eq. 1 agree with the paper's printed constants; the crossover rule
behaves as the paper describes.  No compute entry point is called (no GPU here)."""
import ctypes
import json
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GOLD = os.path.join(ROOT, "tests", "golden")


@pytest.fixture(scope="module")
def b():
    from paper_2509_21081_b200 import build
    build.build()
    from paper_2509_21081_b200 import binding
    return binding


def _declared(header):
    hdr = open(os.path.join(ROOT, "include", header)).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    return set(re.findall(r"\b(typhoon_mla_[a-z_0-9]+)\s*\(", hdr))


def test_exports_every_declared_symbol(b):
    public, internal = _declared("typhoon_mla.h"), _declared("typhoon_mla_internal.h")
    assert {"typhoon_mla_prepare_shared", "typhoon_mla_decode", "typhoon_mla_free", "typhoon_mla_workspace_bytes",
            "typhoon_mla_choose_mode", "typhoon_mla_check_status", "typhoon_mla_status_string"} <= public
    # process-wide switches and measurement hooks are not part of the public header
    assert not {n for n in public if n.startswith("typhoon_mla_set_") and n not in
                ("typhoon_mla_set_hw_model", "typhoon_mla_set_absorb_efficiency")}
    assert not {n for n in public if "profile" in n or "debug" in n}
    lib = ctypes.CDLL(b.LIB_PATH)
    for n in sorted(public | internal):
        assert hasattr(lib, n), f"{n} declared in a header but not exported"
    # and nothing is exported that no header declares
    import subprocess
    out = subprocess.run(["nm", "-D", "--defined-only", b.LIB_PATH], capture_output=True, text=True).stdout
    exported = {ln.split()[-1] for ln in out.splitlines() if " T typhoon_mla_" in ln}
    assert exported <= (public | internal), exported - (public | internal)


def test_status_strings(b):
    assert b._lib.typhoon_mla_status_string(0) == b"ok"
    assert b"workspace" in b._lib.typhoon_mla_status_string(3)


def test_eq1_printed_value(b):
    g = json.load(open(os.path.join(GOLD, "eq1_batch_threshold.json")))
    bt = b.typhoon_mla_batch_threshold(b.make_dims(128), g["S_q"], g["T"], g["M"])
    assert int(bt) == g["B_theta_printed"]
    assert abs(b.typhoon_mla_batch_threshold(b.make_dims(128), 2, g["T"], g["M"]) - bt / 2) < 1e-9
    # no head-count dependence in Eq. 1
    assert b.typhoon_mla_batch_threshold(b.make_dims(64), 1, g["T"], g["M"]) == bt


def test_table1_printed_constants(b):
    g = json.load(open(os.path.join(GOLD, "table1_constants.json")))
    d = b.make_dims(g["dims"]["H"])
    B, Ls, Ln = 7, 1000, 300
    mn, wn = b.typhoon_mla_cost_model(d, b.COST_NAIVE, B, 1, Ls, Ln)
    ma, wa = b.typhoon_mla_cost_model(d, b.COST_ABSORB, B, 1, Ls, Ln)
    mt, wt = b.typhoon_mla_cost_model(d, b.COST_TYPHOON, B, 1, Ls, Ln)
    k = 1024
    assert mn == g["mac_per_token_x1024"]["naive"] * k * B * (Ls + Ln)
    assert ma == g["mac_per_token_x1024"]["absorb"] * k * B * (Ls + Ln)
    assert mt == 40 * k * B * Ls + 136 * k * B * Ln
    assert wn == 40 * k * (Ls + B * Ln)
    assert wa == int(g["hbm_per_token_x1024"]["absorb_exact"] * k) * (Ls + B * Ln)
    assert wt == 40 * k * Ls + 576 * B * Ln
    m3, _ = b.typhoon_mla_cost_model(d, b.COST_TYPHOON, B, 3, Ls, Ln)
    assert m3 == 3 * mt


def test_cost_model_matches_checker(b):
    """Same Table 1 terms as the CPU checker's independent helper."""
    from oracle import mla_oracle as O
    for H in (64, 128):
        d = b.make_dims(H)
        kw = dict(H=H, D_qk=192, D_v=128, D_l=512, D_r=64)
        for kind, name in ((b.COST_NAIVE, "naive"), (b.COST_ABSORB, "absorb"), (b.COST_TYPHOON, "typhoon")):
            m, w = b.typhoon_mla_cost_model(d, kind, 33, 2, 4096, 512)
            assert m == O.macs(name, 33, 2, 4096, 512, **kw)
            assert w == O.hbm_words(name, 33, 4096, 512, **kw)


def test_crossover_rule(b):
    d = b.make_dims(128)
    # zero fixed cost and the paper's NPU numbers: the switch happens where Eq. 1 says, up to the
    # rope keys being read once per token instead of once per head (256.5 vs 320 words per head-token)
    b.typhoon_mla_set_hw_model(376e12, 1.8e12, 0.0)
    b.typhoon_mla_set_absorb_efficiency(1.0)
    modes = [b.typhoon_mla_choose_mode_for(d, 4096, B) for B in range(1, 200)]
    first_hybrid = modes.index(b.MODE_HYBRID) + 1
    assert all(m == b.MODE_ABSORB for m in modes[: first_hybrid - 1])
    assert all(m == b.MODE_HYBRID for m in modes[first_hybrid - 1:])
    bt = b.typhoon_mla_batch_threshold(d, 1, 376e12, 1.8e12)
    assert bt * 256.5 / 320 - 1 <= first_hybrid <= bt + 1
    # a fixed cost pushes short prefixes to absorb, leaves long ones alone
    b.typhoon_mla_set_hw_model(376e12, 1.8e12, 50e-6)
    assert b.typhoon_mla_choose_mode_for(d, 64, 100) == b.MODE_ABSORB
    assert b.typhoon_mla_choose_mode_for(d, 65536, 100) == b.MODE_HYBRID
    # empty suffixes -> naive only; no prefix -> absorb
    assert b.typhoon_mla_choose_mode_for(d, 4096, 8, 0) == b.MODE_NAIVE
    assert b.typhoon_mla_choose_mode_for(d, 0, 512) == b.MODE_ABSORB
    # a less efficient absorb kernel lowers the threshold in proportion
    b.typhoon_mla_set_hw_model(376e12, 1.8e12, 0.0)
    b.typhoon_mla_set_absorb_efficiency(0.5)
    modes = [b.typhoon_mla_choose_mode_for(d, 4096, B) for B in range(1, 200)]
    assert abs((modes.index(b.MODE_HYBRID) + 1) - first_hybrid / 2) <= 1
    b.typhoon_mla_set_hw_model(0, 0, -1)   # restore defaults
    b.typhoon_mla_set_absorb_efficiency(0)
    # defaults (B200): tiny batches fall back, large batches go hybrid
    assert b.typhoon_mla_choose_mode_for(d, 16384, 1) == b.MODE_ABSORB
    assert b.typhoon_mla_choose_mode_for(d, 16384, 8) == b.MODE_ABSORB
    assert b.typhoon_mla_choose_mode_for(d, 16384, 32) == b.MODE_HYBRID
    assert b.typhoon_mla_choose_mode_for(d, 16384, 512) == b.MODE_HYBRID
    # The absorb kernel takes 64-row groups of the stacked [B * H] query matrix over the shared prefix, so with 16
    # heads per device four requests share a group.  Measured on B200 at L_s = 16384, H = 16: absorb-only 42 / 50 /
    # 56 / 77 us at B = 16 / 24 / 32 / 48 against 56 / 58 / 58 / 59 us hybrid; H = 32: 54 / 68 us at B = 16 / 24
    # against 60 / 63; H = 48: 66 / 112 us at B = 16 / 32 against 93 / 96.  The rule has to reproduce the sides.
    for H, B, want in ((16, 2, b.MODE_ABSORB), (16, 16, b.MODE_ABSORB), (16, 24, b.MODE_ABSORB), (16, 48, b.MODE_HYBRID),
                       (32, 16, b.MODE_ABSORB), (32, 24, b.MODE_HYBRID), (48, 16, b.MODE_ABSORB), (48, 32, b.MODE_HYBRID),
                       (128, 20, b.MODE_ABSORB), (128, 24, b.MODE_HYBRID)):
        assert b.typhoon_mla_choose_mode_for(b.make_dims(H), 16384, B) == want, (H, B)


def test_pure_entry_points_reject_bad_arguments(b):
    assert b._lib.typhoon_mla_workspace_bytes(None, 4, 4, 64, 0) == 0
    assert b._lib.typhoon_mla_free(None) == 0
    assert b.typhoon_mla_batch_threshold(b.make_dims(128), 0, 1.0, 1.0) < 0
    with pytest.raises(b.TyphoonMLAError):
        b.typhoon_mla_cost_model(b.make_dims(128), 9, 1, 1, 1, 1)


def test_naive_plan_invariants(b):
    """Work decomposition of the shared-prefix kernel: every schedule covers all tiles with at most
    `n_slots` segments per head; the benchmark sizes get the decompositions the design states."""
    import random
    rnd = random.Random(5)
    for _ in range(400):
        H = rnd.choice([16, 32, 48, 64, 128])
        B = rnd.choice([1, 7, 64, 65, 128, 129, 256, 300, 512, 1024])
        Ls = rnd.randint(1, 40000)
        for schedule in (0, 1, 2):
            tok, R, groups, slots = b.typhoon_mla_naive_plan(H, B, Ls, schedule)
            assert tok == (64 if B <= 128 else 128)
            assert groups == (1 if B <= 128 else (B + 255) // 256)
            n_tiles = (Ls + tok - 1) // tok
            T = H * n_tiles
            assert 1 <= R <= T
            # same partition as the kernel: ranges [0, rem) hold per + 1 tiles
            per, rem = divmod(T, R)
            big = rem * (per + 1)
            rng = lambda t: t // (per + 1) if t < big else rem + (t - big) // per
            seg_max = max(rng(h * n_tiles + n_tiles - 1) - rng(h * n_tiles) + 1 for h in range(H))
            assert slots == seg_max
            if schedule == 1:
                assert R % H == 0 and n_tiles % (R // H) == 0 and seg_max == R // H
            if schedule == 2:
                assert R == min(max(1, (148 if B <= 128 else 74) // groups), T)   # one range per SM, or per pair of SMs
            if schedule == 0 and B > 128:
                assert R % H == 0 or H % R == 0 or R == min(max(1, 74 // groups), T)
    # benchmark configs: config 1 one range per head; config 2 one CTA per SM; config 4 at B = 512 four heads per range
    assert b.typhoon_mla_naive_plan(128, 64, 4096)[1:] == (128, 1, 1)
    assert b.typhoon_mla_naive_plan(128, 128, 26624)[1] == 148
    assert b.typhoon_mla_naive_plan(128, 512, 16384)[1:3] == (32, 2)
    # what a step launches and sizes its partials for
    for H, B, Ls in ((128, 512, 16384), (64, 256, 8192), (16, 166, 7069), (32, 700, 2048), (128, 64, 4096), (16, 129, 1)):
        assert b.typhoon_mla_naive_plan(H, B, Ls)[3] == b.typhoon_mla_workspace_plan(H, Ls, B, 4, mode=b.MODE_HYBRID)[3]
    # every further partial slot is charged with 64-token tiles: shapes where equal ranges over all heads would
    # need three or more slots per head keep one or two ranges per head (measured to be the faster choice)
    assert b.typhoon_mla_naive_plan(128, 128, 16384)[1:] == (128, 1, 1)
    assert b.typhoon_mla_naive_plan(64, 128, 8192)[1:] == (128, 1, 2)
    assert b.typhoon_mla_naive_plan(16, 128, 8192)[1:] == (64, 1, 4)
    assert b.typhoon_mla_naive_plan(64, 70, 20000)[1] == 148        # ... unless the column split wastes too much
    for bad in ((8, 1, 10, 0), (128, 0, 10, 0), (128, 1, 0, 0), (128, 1, 10, 3)):
        with pytest.raises(Exception):
            b.typhoon_mla_naive_plan(*bad)


@pytest.mark.parametrize("H,B,L_s,suffix,beside,alone", [
    # ranges that were measured (B200) to be the fastest cut beside the absorb branch, or within 2 % of it, and by themselves: a
    # part of the places beside the branch, one wave of them alone; but all of them where the branch is short
    (128, 198, 244, 192, 32, 64), (128, 258, 194, 256, 16, 32), (128, 212, 660, 64, 32, 64), (64, 256, 8192, 4096, 64, 64), (16, 166, 7069, 1664, 16, 64), (48, 310, 2108, 576, 16, 37),
    (16, 134, 26345, 64, 74, 74), (48, 243, 17898, 128, 74, 74), (128, 1024, 16384, 256, 16, 18)])
def test_more_than_128_rows_leave_places_to_the_absorb_branch(b, H, B, L_s, suffix, beside, alone):
    assert b.typhoon_mla_naive_plan(H, B, L_s, suffix_tokens=suffix)[1] == beside
    assert b.typhoon_mla_naive_plan(H, B, L_s, suffix_tokens=0)[1] == alone


@pytest.mark.parametrize("H,B,slots,early", [(128, 64, 1, 1), (128, 128, 2, 1), (128, 129, 2, 0), (128, 198, 1, 0), (128, 1024, 1, 0),
                                             (64, 64, 2, 1), (64, 256, 1, 1), (64, 257, 2, 0), (16, 166, 8, 1), (16, 1024, 3, 1), (16, 2048, 1, 0)])
def test_projection_lets_the_next_kernel_start_early_up_to_one_head_and_row_tile_per_sm(b, H, B, slots, early):
    columns, items, ctas, got = b.typhoon_mla_project_plan(H, B, slots)
    assert items * columns == H * ((B + 127) // 128) * 128
    assert ctas == items or ctas == 148
    assert got == early == int(H * ((B + 127) // 128) <= 148)
    assert b.typhoon_mla_project_plan(H, B, slots, prefix_8bit=True) == (columns, items, ctas, 0)


def _slots(H, tiles, n_ranges):
    """From the definition: range of every tile, then the ranges each (head, prefix) meets."""
    T = H * sum(tiles)
    per, rem = divmod(T, n_ranges)
    owner = [r for r in range(n_ranges) for _ in range(per + (r < rem))]
    out, t = [0] * len(tiles), 0
    for _ in range(H):
        for i, n in enumerate(tiles):
            out[i] = max(out[i], owner[t + n - 1] - owner[t] + 1)
            t += n
    return out


@pytest.mark.parametrize("schedule", [0, 1, 2])
@pytest.mark.parametrize("H,rows,L_s", [(16, 1, [1]), (128, 64, [4096]), (128, 65, [129]), (16, 128, [64, 1]), (48, 7, [1, 1, 5000]),
                                        (128, 30, [1000, 900, 1500, 64]), (16, 20, [1 + 97 * i for i in range(16)])])
def test_partial_slots_of_every_prefix_of_a_launch(b, H, rows, L_s, schedule):
    tiles = [(n + 63) // 64 for n in L_s]
    for sms in (1, 20, 148):
        n_ranges, slots = b.typhoon_mla_naive_plan_multi(H, rows, L_s, schedule, sms)
        assert 1 <= n_ranges <= H * sum(tiles)
        assert slots == _slots(H, tiles, n_ranges)
        if len(L_s) == 1:
            assert b.typhoon_mla_naive_plan(H, rows, L_s[0], schedule, sms) == (64, n_ranges, 1, slots[0])


def test_planning_a_launch_of_many_prefixes_costs_no_more_than_planning_each(b):
    import time
    lib = b._lib

    def best(L_s):   # (the call alone: marshalling is done)
        n = len(L_s)
        args = (128, 8, (ctypes.c_int64 * n)(*L_s), n, 2, 148, ctypes.byref(ctypes.c_int32()), (ctypes.c_int32 * n)())
        times = []
        for _ in range(40):
            t = time.perf_counter()
            for _ in range(20):
                lib.typhoon_mla_naive_plan_multi(*args)
            times.append((time.perf_counter() - t) / 20)
        return min(times)

    assert best([256 + 64 * i for i in range(16)]) < 16 * best([736])


@pytest.mark.parametrize("H,L_s,pages,fp8,batches", [
    (16, 4096, 16, False, (8, 130)), (16, 8192, 4, False, (8, 32)), (16, 1000, 4, False, (32,)), (64, 256, 4, False, (32, 256)),
    (128, 1000, 4, False, (8, 130)), (128, 100, 200, False, (128,)), (48, 20000, 33, False, (300, 1024)), (32, 0, 16, False, (64,)),
    (16, 30, 0, False, (200,)), (96, 65536, 1, False, (900,)), (128, 4096, 8, True, (130, 400)), (16, 16384, 24, True, (130,))])
def test_workspace_serves_smaller_batches_and_page_tables(b, H, L_s, pages, fp8, batches):
    """Batches on both sides of 128 query rows and of 128 (request, head) rows, page tables on both sides of the prefix's length."""
    for batch in batches:
        for m in (b.MODE_AUTO, b.MODE_ABSORB, b.MODE_HYBRID, b.MODE_NAIVE):
            size = b.typhoon_mla_workspace_plan(H, L_s, batch, pages, mode=m, prefix_8bit=fp8)[0]
            for B in sorted({*range(1, min(batch, 33)), *range(1, batch + 1, max(1, batch // 29)), 127, 128, 129, batch - 1, batch}):
                if not 1 <= B <= batch:
                    continue
                for p in sorted({pages, pages * 3 // 4, pages // 2, min(pages, max(L_s // 64 - 1, 0)), min(pages, 1), 0}):
                    for path, schedule, stacked in ((0, 0, True), (0, 1, True), (0, 2, False), (1, 0, True)):
                        for mode in ((b.MODE_AUTO, b.MODE_ABSORB, b.MODE_HYBRID, b.MODE_NAIVE) if m == b.MODE_AUTO else (m,)):
                            args = dict(mode=mode, prefix_8bit=fp8, path=path, schedule=schedule, stacked=stacked)
                            _, step, chunks, slots, _ = b.typhoon_mla_workspace_plan(H, L_s, B, p, workspace_bytes=size, **args)
                            assert step <= size
                            _, own, own_chunks, own_slots, _ = b.typhoon_mla_workspace_plan(H, L_s, B, p, **args)
                            assert (chunks, slots) == (own_chunks, own_slots) if own <= size else (chunks < own_chunks or slots < own_slots)


def test_workspace_that_is_too_small_is_refused(b):
    for H, L_s, B, pages in ((16, 4096, 8, 16), (128, 16384, 64, 4), (64, 300, 256, 64), (96, 65536, 900, 1)):
        for mode in (b.MODE_ABSORB, b.MODE_HYBRID, b.MODE_NAIVE):
            _, step, chunks, slots, _ = b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=mode)
            assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=mode, workspace_bytes=step)[1:4] == (step, chunks, slots)
            # with a byte less the step takes fewer partials or is refused; without room for one of each kind it is refused
            try:
                assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=mode, workspace_bytes=step - 1)[1] < step
            except b.TyphoonMLAError as e:
                assert "workspace" in str(e)
            least = B * H * (512 * (2 + 2) + 128 * 4) + B * H * 4 * (512 if mode != b.MODE_NAIVE else 128)
            with pytest.raises(b.TyphoonMLAError, match="workspace"):
                b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=mode, workspace_bytes=least)


@pytest.mark.parametrize("H,B,L_s,pages,pairs", [
    # measured on B200 in both kernels, us per absorb-only step (64 rows per CTA, 128 per pair)
    (64, 12, 22865, 9, 1), (64, 44, 23213, 21, 1), (32, 31, 4399, 7, 1), (64, 2, 23872, 1, 1), (48, 73, 1816, 1, 1),   # 71.9 / 51.5 .. 56.3 / 44.4
    (16, 60, 1426, 1, 0), (48, 67, 131, 1, 0), (16, 187, 193, 1, 0), (16, 214, 199, 1, 0), (48, 465, 343, 1, 0), (32, 185, 3378, 1, 0),   # 28.0 / 33.8 .. 127 / 157
    (16, 7, 4096, 1, 0), (64, 16, 256, 8, 0)])   # fewer than 128 rows; a table wider than the prefix
def test_absorb_only_steps_take_the_kernel_that_is_faster_for_them(b, H, B, L_s, pages, pairs):
    assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=b.MODE_ABSORB)[4] == pairs
    assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=b.MODE_ABSORB, stacked=False)[4] == 0


@pytest.mark.parametrize("H,B,L_s,pages,pairs", [
    (96, 24, 2301, 1, 0), (128, 100, 1277, 1, 0), (128, 100, 1280, 4, 0), (96, 128, 508, 1, 0),   # 36.5 / 40.6, 63.7 / 66.4, 63.3 / 66.1, 48.9 / 51.5
    (128, 8, 809, 4, 1), (96, 24, 544, 4, 1), (128, 64, 4096, 8, 1), (128, 128, 26624, 32, 1), (128, 129, 1000, 1, 1)])   # 43.8 / 39.4, 40.3 / 37.4
def test_many_heads_beside_a_prefix_of_few_rows_take_the_kernel_that_is_faster_for_them(b, H, B, L_s, pages, pairs):
    assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=b.MODE_HYBRID)[4] == pairs
    assert b.typhoon_mla_workspace_plan(H, L_s, B, pages, mode=b.MODE_ABSORB)[4] == 1    # nothing runs beside
