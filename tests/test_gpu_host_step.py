"""Steps whose tensors live in host memory: the bits of the device call for pinned, pageable and oddly placed buffers, on
both sides of the size where the copy engines take over (512 KB in: 10 and 11 requests x 128 heads)."""
import pytest
import torch

from paper_2509_21081_b200 import inputs as I
from tests.gpu_harness import captured_step

pytestmark = pytest.mark.gpu


def _place(t, kind):
    """A host copy of `t`: pinned, pageable, or pinned and starting 2, 4 or 16 bytes behind a 256-byte boundary."""
    if kind == "pageable":
        return t.clone()
    shift = {"pinned": 0, "pinned+2": 2, "pinned+4": 4, "pinned+16": 16}[kind]
    if shift % t.element_size():
        shift = 0
    raw = torch.empty(t.numel() * t.element_size() + 256, dtype=torch.uint8).pin_memory()
    at = (-raw.data_ptr()) % 256 + shift
    view = raw[at:at + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
    return view.copy_(t)


@pytest.mark.parametrize("kind", ["pinned", "pageable", "pinned+2", "pinned+4", "pinned+16"])
@pytest.mark.parametrize("H,B,hi", [(16, 1, 64), (16, 3, 0), (48, 17, 130), (128, 10, 64), (128, 11, 64), (128, 33, 64), (128, 200, 64)])
def test_host_step(kind, H, B, hi):
    from paper_2509_21081_b200.decoder import TyphoonMLADecoder
    inp = I.make_inputs(I.MLAConfig("host", B=B, H=H, Ls=300, suffix_lo=min(hi, 1), suffix_hi=hi, seed=B))
    pc = I.build_pages(inp)
    dec = TyphoonMLADecoder(H, inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), inp.w_uk.cuda(), inp.w_uv.cuda(), inp.scale, B,
                            pc.block_table.shape[1])
    pages = pc.ckv_pages.cuda(), pc.kpe_pages.cuda()
    ref = dec.decode(inp.q_nope.cuda(), inp.q_pe.cuda(), *pages, pc.block_table.cuda(), pc.seq_lens.cuda()).cpu()
    args = [_place(t, kind) for t in (inp.q_nope, inp.q_pe, pc.block_table, pc.seq_lens)]
    out = _place(torch.zeros(B, H, 128, dtype=torch.bfloat16), kind)
    for _ in range(2):
        out.zero_()
        dec.decode_host(args[0], args[1], *pages, args[2], args[3], out)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
    dec.close()


def test_only_one_pinned_block_is_accessed_in_place():
    """A range that leaves its pinned block is left to the copy engines, also where its last byte lies in another pinned
    block.  Only the library's check is asked: nothing is copied or launched."""
    from paper_2509_21081_b200 import binding as b
    torch.cuda.init()
    rt = torch.cuda.cudart()
    raw = torch.zeros(12 * 4096, dtype=torch.uint8)
    base = (raw.data_ptr() + 4095) // 4096 * 4096
    blocks = [(base, 8192), (base + 12288, 8192), (base + 20480, 4096)]      # 4096 pageable bytes between the first two
    mapped = b._lib.typhoon_mla_host_range_mapped
    assert not mapped(base, 64)
    for at, size in blocks:
        assert int(rt.cudaHostRegister(at, size, 0)) == 0
    try:
        assert mapped(base, 8192) and mapped(base + 4, 8188) and mapped(base + 12288, 8192)
        assert not mapped(base, 8196) and not mapped(base + 4096, 4100)      # runs out of its block
        assert not mapped(base, 20480) and not mapped(base + 8188, 4104)     # both ends pinned, the middle not
        assert not mapped(base + 8192, 64) and not mapped(base + 4096, 12288)
        assert not mapped(base + 2, 64) and not mapped(base, 0) and not mapped(None, 64)
        assert not mapped(base + 12288, 12288)                               # two neighbouring blocks
    finally:
        for at, _ in blocks:
            assert int(rt.cudaHostUnregister(at)) == 0
    assert not mapped(base, 64)
    pinned = torch.empty(1 << 20, dtype=torch.uint8).pin_memory()
    assert mapped(pinned.data_ptr(), 1 << 20) and mapped(pinned.data_ptr() + 1000, 4096)
    assert not mapped(raw.data_ptr(), 64)
    assert not mapped(torch.empty(64, dtype=torch.uint8, device="cuda").data_ptr(), 64)


@pytest.mark.parametrize("B,engines", [(8, False), (10, False), (11, True), (64, True)])
def test_copies_leave_room_for_other_streams(B, engines):
    """What keeps several host-fed steps in flight from slowing each other down: engines above 512 KB of inputs, for both
    directions; below it copying blocks that fit on an SM beside an attention kernel (384 threads with 128 of the 65536
    registers each) and do not queue behind other streams' CTAs."""
    from paper_2509_21081_b200 import binding as b
    from paper_2509_21081_b200.decoder import TyphoonMLADecoder
    H = 128
    inp = I.make_inputs(I.MLAConfig("host", B=B, H=H, Ls=200, suffix_lo=64, suffix_hi=64, seed=B))
    pc = I.build_pages(inp)
    dec = TyphoonMLADecoder(H, inp.ckv_shared.cuda(), inp.kpe_shared.cuda(), inp.w_uk.cuda(), inp.w_uv.cuda(), inp.scale, B,
                            pc.block_table.shape[1])
    pages = pc.ckv_pages.cuda(), pc.kpe_pages.cuda()
    args = [t.pin_memory() for t in (inp.q_nope, inp.q_pe, pc.block_table, pc.seq_lens)]
    out = torch.empty(B, H, 128, dtype=torch.bfloat16).pin_memory()
    n_memcpy, kernels = captured_step(lambda: dec.decode_host(args[0], args[1], *pages, args[2], args[3], out, mode=b.MODE_ABSORB))
    copies = [k for k in kernels if "host_copy" in k["name"]]
    assert n_memcpy == (5 if engines else 0) and len(copies) == (0 if engines else 2)
    for k in copies:
        assert k["priority"] == k["highest_priority"] and k["threads"] * k["registers"] + 384 * 128 <= 65536
    dec.close()
