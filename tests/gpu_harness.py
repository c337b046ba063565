"""Helpers of the GPU parity tests: upload a seeded problem, run the library, run the CPU checker."""
import math

import numpy as np
import torch

from oracle import mla_oracle as O
from paper_2509_21081_b200 import inputs as I

MAX_ABS_TOL = 2e-2      # bar on max |gpu - oracle| over the output tensor
REL_FRO_TOL = 5e-3      # bar on ||gpu - oracle||_F / ||oracle||_F
LSE_TOL = 2e-2          # natural-log LSE; bf16 inputs, fp32 statistics


def run_gpu(inp, mode, page_size=None, pages=None, want_lse=True, poison=True, min_max_pages=0,
            force_max_pages=None, fp8_shared=False):
    from paper_2509_21081_b200 import binding as b
    from paper_2509_21081_b200.decoder import TyphoonMLADecoder
    cfg = inp.cfg
    ps = page_size or cfg.page_size
    pc = pages or I.build_pages(inp, page_size=ps, poison=poison, min_max_pages=min_max_pages)
    dev = "cuda"
    max_pages = pc.block_table.shape[1] if force_max_pages is None else force_max_pages
    dec = TyphoonMLADecoder(cfg.H, inp.ckv_shared.to(dev), inp.kpe_shared.to(dev), inp.w_uk.to(dev),
                            inp.w_uv.to(dev), inp.scale, cfg.B, max_pages, ps, fp8_shared=fp8_shared)
    lse = torch.empty(cfg.B, cfg.H, dtype=torch.float32, device=dev) if want_lse else None
    if force_max_pages == 0:
        out = dec.decode(inp.q_nope.to(dev), inp.q_pe.to(dev), None, None, None, None, mode=mode, lse_out=lse)
    else:
        out = dec.decode(inp.q_nope.to(dev), inp.q_pe.to(dev), pc.ckv_pages.to(dev), pc.kpe_pages.to(dev),
                         pc.block_table.to(dev), pc.seq_lens.to(dev), mode=mode, lse_out=lse)
    launches = b.typhoon_mla_last_launch_count()
    assert b.typhoon_mla_check_status(dec.shared) == 0   # synchronises; raises if an in-kernel wait expired
    res = out.float().cpu().double().numpy(), (lse.cpu().double().numpy() if want_lse else None), launches
    dec.close()
    return res


def run_oracle(inp, pairs=None, drop_suffix=False):
    f = I.to_f64
    ckv_suf = [f(x[:0] if drop_suffix else x) for x in inp.ckv_suffix]
    kpe_suf = [f(x[:0] if drop_suffix else x) for x in inp.kpe_suffix]
    return O.mla_decode(f(inp.q_nope), f(inp.q_pe), f(inp.ckv_shared), f(inp.kpe_shared), ckv_suf, kpe_suf,
                        f(inp.w_uk), f(inp.w_uv), inp.scale, pairs=pairs)


def run_oracle_fp8(inp, pairs=None, drop_suffix=False):
    """The checker for a prefix whose expanded K_nope / V are stored as E4M3 codes."""
    from oracle import fp8_oracle as F
    f = I.to_f64
    ckv_suf = [f(x[:0] if drop_suffix else x) for x in inp.ckv_suffix]
    kpe_suf = [f(x[:0] if drop_suffix else x) for x in inp.kpe_suffix]
    return F.mla_decode_fp8_shared(f(inp.q_nope), f(inp.q_pe), f(inp.ckv_shared), f(inp.kpe_shared), ckv_suf, kpe_suf,
                                   f(inp.w_uk), f(inp.w_uv), inp.scale, pairs=pairs)


def reference64(inp):
    """The step from its definition in 64 bits on the GPU (one softmax over shared prefix and own tokens): numpy (out, lse)."""
    B, H = inp.cfg.B, inp.cfg.H
    qn, qp, w_uk, w_uv, ckv, kpe = (x.cuda().double() for x in (inp.q_nope, inp.q_pe, inp.w_uk, inp.w_uv, inp.ckv_shared,
                                                                inp.kpe_shared))
    lse = torch.full((B, H), -math.inf, dtype=torch.float64, device="cuda")
    out = torch.zeros(B, H, 128, dtype=torch.float64, device="cuda")

    def merge(where, l, o):
        old = lse[where]
        new = torch.logaddexp(old, l)
        out[where] = out[where] * torch.exp(old - new)[..., None] + o * torch.exp(l - new)[..., None]
        lse[where] = new

    if ckv.shape[0]:
        for h in range(H):
            logits = (qn[:, h] @ (ckv @ w_uk[h].T).T + qp[:, h] @ kpe.T) * inp.scale
            merge((slice(None), h), torch.logsumexp(logits, -1), torch.softmax(logits, -1) @ (ckv @ w_uv[h].T))
    q_lat = torch.einsum("bhd,hdc->bhc", qn, w_uk)
    for r in range(B):
        c, k = inp.ckv_suffix[r].cuda().double(), inp.kpe_suffix[r].cuda().double()
        if c.shape[0]:
            logits = (q_lat[r] @ c.T + qp[r] @ k.T) * inp.scale
            merge(r, torch.logsumexp(logits, -1), torch.einsum("hc,hdc->hd", torch.softmax(logits, -1) @ c, w_uv))
    return out.cpu().numpy(), lse.cpu().numpy()


def worst_row(got, ref):
    """Largest relative error (2-norm) of a (request, head) row: an error in one row cannot hide in the whole tensor's norm
    (385 x 128 rows, one of them wrong: 4.5e-3)."""
    got, ref = got.reshape(-1, got.shape[-1]).double(), ref.reshape(-1, ref.shape[-1]).double()
    return (torch.linalg.norm(got - ref, dim=1) / torch.linalg.norm(ref, dim=1)).max().item()


def errors(gpu, ref, mask=None):
    if mask is not None:
        gpu, ref = gpu[mask], ref[mask]
    d = gpu - ref
    max_abs = float(np.max(np.abs(d))) if d.size else 0.0
    denom = float(np.linalg.norm(ref))
    rel = float(np.linalg.norm(d)) / denom if denom > 0 else float(np.linalg.norm(d))
    return max_abs, rel


def assert_parity(gpu_out, ref_out, gpu_lse=None, ref_lse=None, mask=None, what=""):
    assert np.isfinite(gpu_out if mask is None else gpu_out[mask]).all(), f"{what}: non-finite output"
    max_abs, rel = errors(gpu_out, ref_out, mask)
    # The 2e-2 bar is stated for outputs of the benchmark distributions (|out| < 1).  Stress inputs
    # (peaked softmax) produce outputs of magnitude several units, whose final bf16 rounding alone is
    # 2^-9 relative, so the absolute bar scales with the largest expected magnitude once that exceeds 1.
    ref_sel = ref_out if mask is None else ref_out[mask]
    abs_tol = MAX_ABS_TOL * max(1.0, float(np.max(np.abs(ref_sel))) if ref_sel.size else 1.0)
    assert max_abs <= abs_tol, f"{what}: max-abs {max_abs:.3e} > {abs_tol:.3e}"
    assert rel <= REL_FRO_TOL, f"{what}: rel-Frobenius {rel:.3e} > {REL_FRO_TOL}"
    # no single (b, h) row may hide behind the aggregate: per-row relative error bar (looser)
    if mask is None:
        rows_g = gpu_out.reshape(-1, gpu_out.shape[-1]); rows_r = ref_out.reshape(-1, ref_out.shape[-1])
    else:
        rows_g, rows_r = gpu_out[mask], ref_out[mask]
    rn = np.linalg.norm(rows_r, axis=1)
    re = np.linalg.norm(rows_g - rows_r, axis=1)
    ok = rn > 0
    if ok.any():
        worst = float(np.max(re[ok] / rn[ok]))
        assert worst <= 4 * REL_FRO_TOL, f"{what}: worst row rel error {worst:.3e}"
    if gpu_lse is not None:
        gl = gpu_lse if mask is None else gpu_lse[mask]
        rl = ref_lse if mask is None else ref_lse[mask]
        inf = np.isinf(rl)
        assert np.array_equal(np.isinf(gl), inf), f"{what}: -inf pattern of lse differs"
        if (~inf).any():
            e = float(np.max(np.abs(gl[~inf] - rl[~inf])))
            # logits carry bf16-level relative error (stored K, absorbed q), so the LSE bar scales with
            # the LSE magnitude once that exceeds the benchmark distributions' (about 9)
            tol = LSE_TOL * max(1.0, float(np.max(np.abs(rl[~inf]))) / 10.0)
            assert e <= tol, f"{what}: lse error {e:.3e} > {tol:.3e}"
    return max_abs, rel


def captured_step(step):
    """Captures `step()` as a CUDA graph: (number of copy nodes, its kernels' launch properties); nothing runs."""
    import pytest
    driver = pytest.importorskip("cuda.bindings.driver")

    def call(fn, *a):
        err, *res = fn(*a)
        assert int(err) == 0, (fn, err)
        return res[0] if len(res) == 1 else res

    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph, stream=torch.cuda.Stream()):
        step()
    g = driver.CUgraph(graph.raw_cuda_graph())
    _, n = call(driver.cuGraphGetNodes, g, 0)
    nodes, n = call(driver.cuGraphGetNodes, g, n)
    kind, of_func = driver.CUgraphNodeType, driver.CUfunction_attribute
    copies, kernels = 0, []
    for node in nodes[:n]:
        t = call(driver.cuGraphNodeGetType, node)
        copies += t == kind.CU_GRAPH_NODE_TYPE_MEMCPY
        if t != kind.CU_GRAPH_NODE_TYPE_KERNEL:
            continue
        prm = call(driver.cuGraphKernelNodeGetParams, node)
        func = prm.func if int(prm.func) else call(driver.cuKernelGetFunction, prm.kern)
        attr = call(driver.cuGraphKernelNodeGetAttribute, node, driver.CUlaunchAttributeID.CU_LAUNCH_ATTRIBUTE_PRIORITY)
        kernels.append(dict(name=call(driver.cuFuncGetName, func).decode(), priority=attr.priority,
                            highest_priority=call(driver.cuCtxGetStreamPriorityRange)[1], threads=prm.blockDimX, grid=(prm.gridDimX, prm.gridDimY),
                            registers=call(driver.cuFuncGetAttribute, of_func.CU_FUNC_ATTRIBUTE_NUM_REGS, func),
                            local_bytes=call(driver.cuFuncGetAttribute, of_func.CU_FUNC_ATTRIBUTE_LOCAL_SIZE_BYTES, func)))
    return copies, kernels
