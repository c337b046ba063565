"""Prefixes whose buffers lie in the caller's device memory: same results as the library's own allocation, storage that
is reused at once, refusals.  (Sizes: a prefix of one token, one below, at and above the 128-row padding.)"""
import ctypes as C

import pytest
import torch

from paper_2509_21081_b200 import inputs as I


@pytest.mark.parametrize("Ls", [0, 1, 127, 128, 129, 1000])
@pytest.mark.parametrize("fp8", [False, True])
def test_storage_bytes_cover_the_parts(Ls, fp8):
    from paper_2509_21081_b200 import binding as b
    H, Lp = 48, (Ls + 127) // 128 * 128
    scratch = C.c_size_t()
    n = b._lib.typhoon_mla_shared_storage_bytes(C.byref(b.make_dims(H)), Ls, int(fp8), C.byref(scratch))
    expanded = 2 * H * Lp * 128
    parts = Lp * (512 + 64) * 2 + H * 512 * 128 * 2 + 256 + (expanded if fp8 else 2 * expanded)
    assert parts <= n <= parts + (12 * H if fp8 else 0) + 8 * 256
    assert scratch.value == (expanded if fp8 else 0)
    assert b._lib.typhoon_mla_shared_storage_bytes(C.byref(b.make_dims(17)), Ls, int(fp8), None) == 0


def _step(b, prepare, dims, inp, dev, H, B):
    sh = prepare(dims, dev["ckv"], dev["kpe"], dev["w_uk"], dev["w_uv"])
    ws = torch.empty(b.typhoon_mla_workspace_bytes(sh, B, 0, 64), dtype=torch.uint8, device="cuda")
    out = torch.empty(B, H, 128, dtype=torch.bfloat16, device="cuda")
    lse = torch.empty(B, H, dtype=torch.float32, device="cuda")
    b.typhoon_mla_decode(sh, dev["qn"], dev["qp"], None, None, 64, None, None, inp.scale, out, ws, mode=b.MODE_NAIVE, lse_out=lse)
    b.typhoon_mla_check_status(sh)
    sh.free()
    return out, lse


@pytest.mark.gpu
@pytest.mark.parametrize("fp8", [False, True])
def test_storage_of_the_caller_gives_the_same_bits(fp8):
    from paper_2509_21081_b200 import binding as b
    H, B, dims = 16, 5, b.make_dims(16)
    prepare = b.typhoon_mla_prepare_shared_fp8 if fp8 else b.typhoon_mla_prepare_shared
    own = getattr(b._lib, "typhoon_mla_prepare_shared_fp8" if fp8 else "typhoon_mla_prepare_shared")

    def library_allocates(dims, ckv, kpe, w_uk, w_uv):
        h = C.c_void_p()
        assert own(C.byref(dims), b._ptr(ckv), b._ptr(kpe), ckv.shape[0], 512, 64, b._ptr(w_uk), b._ptr(w_uv), b._stream(),
                   C.byref(h)) == 0
        return b.SharedPrefix(h, dims, (w_uk, w_uv))

    for Ls in (1, 127, 129, 700):    # the later ones reuse the earlier ones' memory from the allocator
        inp = I.make_inputs(I.MLAConfig("storage", B=B, H=H, Ls=Ls, suffix_lo=0, suffix_hi=0, seed=Ls))
        dev = dict(ckv=inp.ckv_shared.cuda(), kpe=inp.kpe_shared.cuda(), w_uk=inp.w_uk.cuda(), w_uv=inp.w_uv.cuda(),
                   qn=inp.q_nope.cuda(), qp=inp.q_pe.cuda())
        ref = _step(b, library_allocates, dims, inp, dev, H, B)
        for _ in range(2):
            got = _step(b, prepare, dims, inp, dev, H, B)
            assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    assert b._lib.typhoon_mla_release_cached() == 0


@pytest.mark.gpu
def test_too_little_or_misaligned_storage_is_refused():
    from paper_2509_21081_b200 import binding as b
    dims, Ls = b.make_dims(16), 100
    inp = I.make_inputs(I.MLAConfig("storage", B=1, H=16, Ls=Ls, suffix_lo=0, suffix_hi=0, seed=1))
    t = [x.cuda() for x in (inp.ckv_shared, inp.kpe_shared, inp.w_uk, inp.w_uv)]
    scratch = C.c_size_t()
    n = b._lib.typhoon_mla_shared_storage_bytes(C.byref(dims), Ls, 1, C.byref(scratch))
    mem = torch.empty(n + 512, dtype=torch.uint8, device="cuda")
    tmp = torch.empty(scratch.value, dtype=torch.uint8, device="cuda")

    def prepare(storage, nbytes, scr, scr_bytes):
        h = C.c_void_p()
        st = b._lib.typhoon_mla_prepare_shared_in(C.byref(dims), b._ptr(t[0]), b._ptr(t[1]), Ls, 512, 64, b._ptr(t[2]),
                                                  b._ptr(t[3]), 1, storage, nbytes, scr, scr_bytes, b._stream(), C.byref(h))
        assert st != 0 and not h.value
        return st

    ok = C.c_void_p(mem.data_ptr())
    assert prepare(ok, n - 1, b._ptr(tmp), scratch.value) == 3
    assert prepare(ok, n, b._ptr(tmp), scratch.value - 1) == 3
    assert prepare(ok, n, None, 0) == 3
    assert prepare(C.c_void_p(mem.data_ptr() + 16), n, b._ptr(tmp), scratch.value) == 1
    assert prepare(None, 0, b._ptr(tmp), scratch.value) == 1
