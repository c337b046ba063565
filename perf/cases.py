"""The decode-attention work that a serving program has this library do, as a list of measurable cases.

All calls go through the package's public entry points: ``TyphoonMLADecoder`` (a prepared prefix, a workspace and one
call per decode step, with the step's tensors on the device or in pinned host memory), ``typhoon_mla_decode_tree``
(several shared prefixes per step), ``typhoon_mla_expand_query_rows`` (several query tokens per request) and the 8-bit
storage option of the expanded prefix.  The step's mode is left to the library's own rule everywhere.

Shapes follow ``paper_2509_21081_b200/inputs.py``: d_nope = 128, d_rope = 64, d_v = 128, latent width 512, activations
N(0, 1), projection weights N(0, 1/512), suffix lengths uniform in a range, physical pages in random order.
"""
import math

import torch

from paper_2509_21081_b200 import binding as b
from paper_2509_21081_b200.decoder import TyphoonMLADecoder

SCALE = (128 + 64) ** -0.5


def _case(name, kind, heads, batch, prefix, lo, hi, page=64, queries=1, branches=0, branch=0):
    case = {"kind": kind, "heads": heads, "batch": batch, "prefix": prefix, "suffix_lo": lo, "suffix_hi": hi, "page": page,
            "queries": queries, "branches": branches, "branch": branch}
    return dict(case, name=name) if name else case


def listed():
    return [
        # a few requests on one of eight devices that share the heads: nothing but launches and latency
        _case("tiny", "decode", 16, 4, 256, 64, 64),
        # one conversation over a long prompt
        _case("one_request", "decode", 128, 1, 16384, 256, 256),
        # a small fan-out (sampled answers to one question), still in the fall-back formulation
        _case("fanout_8", "decode", 128, 8, 16384, 256, 256),
        # a medium fan-out whose per-step tensors live in the serving process's pinned host memory
        _case("fanout_32_host", "host", 128, 32, 16384, 256, 256),
        # the ordinary step: a system prompt, a batch of chats of equal length
        _case("system_prompt_64", "decode", 128, 64, 4096, 512, 512),
        # a very long system prompt, ragged chats
        _case("long_prompt_128", "decode", 128, 128, 26624, 256, 2048),
        # half the heads, long ragged suffixes: most of the bytes are the requests' own
        _case("ragged_256", "decode", 64, 256, 8192, 128, 4096),
        # the largest fan-out (parallel reasoning)
        _case("fanout_1024", "decode", 128, 1024, 16384, 256, 256),
        # speculative verification, two query tokens per request, on one of eight devices that share the heads; odd sizes
        _case("verify_shard", "decode", 16, 83, 7069, 3, 1537, page=128, queries=2),
        # a system prompt and one more prompt per group of requests
        _case("prompt_tree", "tree", 128, 72, 4096, 100, 700, branches=4, branch=1111),
        # the expanded prefix stored in 8 bits
        _case("prefix_8bit", "fp8", 128, 64, 4096, 512, 512),
        # a new system prompt arrives: expand it, answer the first step of the waiting requests, drop it
        _case("new_prompt", "prepare", 128, 24, 4759, 1, 64),
    ]


def _seconds(case):
    w = work(case)
    return max(w["bytes"] / 5.0e12, w["flops"] / 1.0e15)


def draw(rng):
    def log_int(lo, hi):
        return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    kind = rng.choice(["decode"] * 6 + ["host", "tree", "fp8", "prepare"])
    heads = rng.choice([128, 128, 128, 64, 64, 32, 16])
    batch = log_int(1, 1024)
    prefix = log_int(256, 26624)
    hi = log_int(16, 4096)
    lo = rng.randint(1, hi)
    page = rng.choice([64, 64, 64, 128])
    queries = rng.choice([1, 1, 1, 2, 3]) if kind == "decode" else 1
    branches = branch = 0
    if kind == "tree":
        batch = max(batch, 8)
        branches, branch = rng.randint(2, 6), log_int(128, 4096)
    if kind == "prepare":
        batch, prefix, hi = min(batch, 64), min(prefix, 8192), min(hi, 256)
        lo = min(lo, hi)
    largest = max(_seconds(c) for c in listed())
    while True:
        case = _case("", kind, heads, batch, prefix, lo, hi, page, queries, branches, branch)
        if (_seconds(case) <= largest and batch * queries <= 1024 and batch * hi <= 1 << 20) or batch <= 8:
            return case
        batch = batch * 3 // 4


# ---------------------------------------------------------------- inputs
def _normal(gen, *shape, mul=1.0):
    x = torch.randn(*shape, generator=gen, dtype=torch.float32, device="cuda")
    return x.mul_(mul).to(torch.bfloat16)


def _groups(case):
    """First request of every branch (and the end): groups of different sizes."""
    n, total = case["branches"], case["branch"]
    weights = [2 + (i * 3 + total) % 4 for i in range(n)]
    begin, acc = [0], 0
    for w in weights:
        acc += w
        begin.append(case["batch"] * acc // sum(weights))
    return begin


def _branch_lengths(case):
    return [max(1, case["branch"] * (4 + i % 3) // 5) for i in range(case["branches"])]


class State:
    pass


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed * 7919 + 17)
    cpu = torch.Generator()
    cpu.manual_seed(seed * 104729 + 5)
    H, B, page, S = case["heads"], case["batch"], case["page"], case["queries"]
    st = State()
    st.case = case
    st.ckv = _normal(gen, case["prefix"], 512)
    st.kpe = _normal(gen, case["prefix"], 64)
    st.w_uk = _normal(gen, H, 128, 512, mul=512 ** -0.5)
    st.w_uv = _normal(gen, H, 128, 512, mul=512 ** -0.5)
    st.q_nope = _normal(gen, B * S, H, 128)
    st.q_pe = _normal(gen, B * S, H, 64)

    # the paged cache of the requests' own tokens
    lens = torch.randint(case["suffix_lo"], case["suffix_hi"] + 1, (B,), generator=cpu)
    need = (lens + page - 1) // page
    st.max_pages = (case["suffix_hi"] + page - 1) // page
    total = int(need.sum())
    n_pages = total + 2
    ids = torch.randperm(n_pages, generator=cpu)[:total].to(torch.int32)
    table = torch.full((B, st.max_pages), -1, dtype=torch.int32)
    table[torch.arange(st.max_pages)[None, :] < need[:, None]] = ids
    st.ckv_pages = torch.empty(n_pages, page, 512, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    st.kpe_pages = torch.empty(n_pages, page, 64, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)
    lens = lens.to(torch.int32)

    st.table, st.lens = table, lens
    # the prompts of a tree's branches
    st.parts = [(_normal(gen, n, 512), _normal(gen, n, 64)) for n in _branch_lengths(case)]
    return st


def prepare(case, seed):
    st = _inputs(case, seed)
    H, B, page, kind = case["heads"], case["batch"], case["page"], case["kind"]
    st.parts, parts_in = [], st.parts
    if kind == "host":
        st.q_nope, st.q_pe = st.q_nope.cpu().pin_memory(), st.q_pe.cpu().pin_memory()
        st.table, st.lens = st.table.pin_memory(), st.lens.pin_memory()
        st.out = torch.empty(B, H, 128, dtype=torch.bfloat16).pin_memory()
    else:
        st.table, st.lens = st.table.cuda(), st.lens.cuda()
    if kind == "tree":
        dims = b.make_dims(H)
        root = b.typhoon_mla_prepare_shared(dims, st.ckv, st.kpe, st.w_uk, st.w_uv)
        parts = [b.typhoon_mla_prepare_shared(dims, ckv, kpe, st.w_uk, st.w_uv) for ckv, kpe in parts_in]
        st.levels = [([root], [0, B]), (parts, _groups(case))]
        size = b.typhoon_mla_tree_workspace_bytes(st.levels, B, st.max_pages, page)
        st.workspace = torch.empty(size, dtype=torch.uint8, device="cuda")
    elif kind != "prepare":
        st.decoder = _decoder(st)
    torch.cuda.synchronize()
    return st


def _decoder(st):
    c = st.case
    return TyphoonMLADecoder(c["heads"], st.ckv, st.kpe, st.w_uk, st.w_uv, SCALE, c["batch"] * c["queries"], st.max_pages,
                             c["page"], fp8_shared=c["kind"] == "fp8")


# ---------------------------------------------------------------- one pass
def run(st):
    c = st.case
    if c["kind"] == "host":
        st.decoder.decode_host(st.q_nope, st.q_pe, st.ckv_pages, st.kpe_pages, st.table, st.lens, st.out)
        return st.out
    if c["kind"] == "tree":
        out = torch.empty(c["batch"], c["heads"], 128, dtype=torch.bfloat16, device="cuda")
        b.typhoon_mla_decode_tree(st.levels, st.q_nope, st.q_pe, st.ckv_pages, st.kpe_pages, c["page"], st.table, st.lens,
                                  SCALE, out, st.workspace)
        return out
    if c["kind"] == "prepare":
        decoder = _decoder(st)
        out = decoder.decode(st.q_nope, st.q_pe, st.ckv_pages, st.kpe_pages, st.table, st.lens)
        decoder.close()
        return out
    table, lens = st.table, st.lens
    if c["queries"] > 1:
        table, lens = b.typhoon_mla_expand_query_rows(table, lens, c["queries"])
    lse = torch.empty(c["batch"] * c["queries"], c["heads"], dtype=torch.float32, device="cuda")
    out = st.decoder.decode(st.q_nope, st.q_pe, st.ckv_pages, st.kpe_pages, table, lens, lse_out=lse)
    return out, lse


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    """The cheaper of the two formulations of the shared part (expanded per-head keys and values, or the latent cache
    itself); every input is read once and every output written once, at 2 operations per multiply-add."""
    H, B, rows = case["heads"], case["batch"], case["batch"] * case["queries"]
    shared = [(rows, case["prefix"])]
    if case["kind"] == "tree":
        begin = _groups(case)
        shared += [(e - a, n) for a, e, n in zip(begin, begin[1:], _branch_lengths(case)) if e > a]
    suffix = B * (case["suffix_lo"] + case["suffix_hi"]) / 2
    # projections in and out of the latent space, queries and output, weights, the requests' own tokens
    flops = 262144.0 * H * rows + 2176.0 * H * case["queries"] * suffix
    bytes_ = 640.0 * H * rows + 262144.0 * H + 1152.0 * suffix
    for r, n in shared:
        token = 256 if case["kind"] == "fp8" else 512
        expanded = {"flops": 640.0 * H * r * n, "bytes": (token * H + 128.0) * n}
        latent = {"flops": 2176.0 * H * r * n, "bytes": 1152.0 * n}
        best = min((expanded, latent), key=lambda w: max(w["bytes"] / 6.5e12, w["flops"] / 1.6e15))
        flops += best["flops"]
        bytes_ += best["bytes"]
    if case["kind"] == "prepare":
        flops += 262144.0 * H * case["prefix"]
        bytes_ += (512.0 * H + 2 * 1152.0) * case["prefix"] + 262144.0 * H
    return {"bytes": bytes_, "flops": flops}


def _e4m3(x):
    """The values that the 8-bit option keeps: bf16, then E4M3 codes under one power-of-two scale per head."""
    x = x.to(torch.bfloat16).double()
    mant, ex = torch.frexp(x.abs().amax() / 448.0)
    scale = 2.0 ** float(ex - 1 if float(mant) == 0.5 else ex)
    return (x / scale).float().to(torch.float8_e4m3fn).double() * scale


def exact(case, seed):
    """Attention over prefix, branch and own tokens with one softmax, from the definition, in 64 bits."""
    st = _inputs(case, seed)
    H, B, S = case["heads"], case["batch"], case["queries"]
    qn, qp, w_uk, w_uv = (x.double() for x in (st.q_nope, st.q_pe, st.w_uk, st.w_uv))

    def add(logits, value):
        """logits [.., rows, tokens], value [.., tokens, d] -> (lse [.., rows], o [.., rows, d])"""
        lse = torch.logsumexp(logits, -1)
        return lse, torch.exp(logits - lse[..., None]) @ value

    shared = [(0, B, st.ckv, st.kpe)]
    if case["kind"] == "tree":
        begin = _groups(case)
        shared += [(a, e, ckv, kpe) for a, e, (ckv, kpe) in zip(begin, begin[1:], st.parts) if e > a]
    rows = B * S
    total_lse = torch.full((rows, H), -math.inf, dtype=torch.float64, device="cuda")
    total = torch.zeros(rows, H, 128, dtype=torch.float64, device="cuda")

    def merge(where, lse, o):
        old = total_lse[where]
        new = torch.logaddexp(old, lse)
        total[where] = total[where] * torch.exp(old - new)[..., None] + o * torch.exp(lse - new)[..., None]
        total_lse[where] = new

    for a, e, ckv, kpe in shared:
        ckv, kpe = ckv.double(), kpe.double()
        for h in range(H):
            k, v = ckv @ w_uk[h].T, ckv @ w_uv[h].T
            if case["kind"] == "fp8":
                k, v = _e4m3(k), _e4m3(v)
            where = (slice(a * S, e * S), h)
            merge(where, *add((qn[where] @ k.T + qp[where] @ kpe.T) * SCALE, v))
    q_lat = torch.einsum("rhd,hdc->rhc", qn, w_uk)   # the same logits, from the latent form
    for r in range(B):
        ids = st.table[r][st.table[r] >= 0].long().cuda()
        ckv = st.ckv_pages[ids].reshape(-1, 512).double()
        kpe = st.kpe_pages[ids].reshape(-1, 64).double()
        for j in range(S):
            n = max(int(st.lens[r]) - (S - 1 - j), 0)
            if n > 0:
                row = r * S + j
                lse, o = add((q_lat[row] @ ckv[:n].T + qp[row] @ kpe[:n].T) * SCALE, ckv[:n])
                merge(row, lse, torch.einsum("hc,hdc->hd", o, w_uv))
    if case["kind"] in ("host", "tree", "prepare"):
        return total
    return total, total_lse


def tolerance(case):
    # 16-bit operands and results, 32-bit accumulation.  Against the same operation in 64 bits the listed cases differ by
    # 1.8e-3 to 3.0e-3 (2-norm) and at most 1.5e-2 of the root mean square (log-sum-exps: 3e-5); this is about four times
    # that.  (With the 8-bit prefix the encoding itself is part of the operation.)
    return {"rel": 1e-2, "max": 0.06}
