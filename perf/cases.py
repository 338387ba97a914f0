"""The calls a decode server makes into this library, as cases that can be timed.

A case is one call (or one pair of calls) on one attention layer: the decode step, sparse decode over given lists,
the threshold gate followed by sparse decode, the multi-token step, dense decode, and the bulk build of the
compressed-key cache after prefill.  Head counts, lengths, budgets and block sizes are those of the workloads in
``paper_2506_08889_b200/synth.py``, of the paper's 64/8-head kernel grid, and of the tests.

``listed()`` names a dozen of them, ``draw(rng)`` gives further ones of the same ranges.
"""
from __future__ import annotations

import math

import torch

from paper_2506_08889_b200 import binding, synth

D = 128                          # head_dim, the library's only one
THETA = 1.0e6
SCALE = 1.0 / math.sqrt(D)
GATE_STD = 0.02                  # random-init gate projections
PEAKED_GATE_STD = 0.045          # the threshold method only makes sense with scores that differ
MAX_CACHE_BYTES = 4.4e9          # K and V of one state

_ctx = None


def _context():
    """A server has one context per stream; it serves every layer."""
    global _ctx
    if _ctx is None:
        _ctx = binding.Context(torch.cuda.current_device())
    return _ctx


def _case(kind, batch, hq, hkv, block, len_max, len_min=0, budget=0, page=0, token_major=False, q_len=1, d_gate=128,
          threshold=0.0, sparsity=0.0, name=None):
    c = dict(kind=kind, batch=batch, hq=hq, hkv=hkv, block=block, len_max=len_max, len_min=len_min or len_max,
             budget=budget, page=page, token_major=token_major, q_len=q_len, d_gate=d_gate, threshold=threshold,
             sparsity=sparsity)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest step: one tensor-parallel slice (one KV head) of a short chat, 8 of 64 blocks; pure latency
        _case("step", 1, 4, 1, 64, 4096, budget=512, name="step_b1_h4_l4k"),
        # one user, long reasoning trace, 4096-token budget; the length is not a multiple of the block, as in 63 of 64 steps
        _case("step", 1, 32, 8, 64, 32741, budget=4096, name="step_b1_l32k"),
        # the same at 40/8 heads and 64k in the step in which a block fills (the append has work to do)
        _case("step", 1, 40, 8, 64, 65536, budget=4096, name="step_b1_l64k"),
        # continuous batching on a paged cache: four users of very different lengths
        _case("step", 4, 32, 8, 64, 32000, len_min=2500, budget=4096, page=128, name="step_b4_ragged_paged"),
        # the benchmark's own workload: batch 8 at 128k, 90 % of the blocks skipped
        _case("step", 8, 40, 8, 64, 131072, budget=205 * 64, name="step_b8_l128k_s90"),
        # a million-token context: more compressed keys per head than the one-kernel gate holds
        _case("step", 1, 32, 8, 64, 1000003, budget=8192, name="step_b1_l1m"),
        # lists chosen by the caller (another gate), blocks of 128, large ragged batch
        _case("sparse", 16, 32, 8, 128, 65536, len_min=8192, sparsity=0.9, name="sparse_b16_ragged_b128"),
        # the paper's second sparsify method at the paper's kernel-grid head counts, small blocks
        _case("threshold", 4, 64, 8, 32, 49152, len_min=40000, threshold=2.0e-3, name="threshold_b4_l48k_b32"),
        # speculative decoding: four query tokens per sequence verified in one step
        _case("multi", 4, 40, 8, 64, 65536, len_min=60000, budget=4096, q_len=4, name="multi_b4_l64k_q4"),
        # dense layers of the same model (or a request without sparsity), ragged and long
        _case("dense", 8, 40, 8, 64, 131072, len_min=16000, name="dense_b8_ragged_l128k"),
        # after prefill: the compressed keys of two 128k prompts, head-major pre-RoPE keys
        _case("build", 2, 40, 8, 64, 131072, name="build_b2_l128k"),
        # the same for a batch of shorter prompts with blocks of 128 and token-major keys (as a projection writes them)
        _case("build", 6, 32, 8, 128, 32768, len_min=5000, token_major=True, name="build_b6_ragged_b128"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    limit = max(work(c)["bytes"] for c in listed())
    while True:
        kind = rng.choice(["step", "step", "step", "sparse", "threshold", "multi", "dense", "build"])
        hq, hkv = rng.choice([(32, 8), (40, 8), (64, 8), (32, 8), (40, 8), (8, 2), (4, 1)])
        block = rng.choice([64, 64, 64, 128, 32, 16])
        batch = _log_int(rng, 1, 16)
        len_max = _log_int(rng, 1500, 262144 if kind != "build" else 131072)
        if rng.random() < 0.3:
            len_max = -(-len_max // 128) * 128
        len_min = len_max if batch == 1 or rng.random() < 0.4 else max(1000, int(len_max * rng.uniform(0.1, 0.9)))
        c = _case(kind, batch, hq, hkv, block, len_max, len_min=min(len_min, len_max),
                  token_major=rng.random() < 0.3)
        if kind in ("step", "multi"):
            c["budget"] = min(_log_int(rng, 1024, 16384), max(256, len_max // 2))
        if kind in ("step", "multi", "threshold"):
            c["d_gate"] = rng.choice([128, 128, 128, 64, 256])
        if kind == "multi":
            c["q_len"] = rng.randint(2, 8)
        if kind == "sparse":
            c["sparsity"] = rng.choice([0.5, 0.7, 0.8, 0.9, 0.95])
        if kind == "threshold":
            c["threshold"] = round(rng.uniform(1.5, 5.0) / _blocks(c, len_max), 6)
        if kind in ("step", "multi", "sparse", "dense") and rng.random() < 0.4:
            c["page"], c["token_major"] = rng.choice([64, 128, 256]), False
            c["page"] = max(c["page"], block)
        cache = 2 * batch * hkv * _capacity(c) * D * 2
        if cache <= MAX_CACHE_BYTES and work(c)["bytes"] <= limit:
            return c


def _blocks(c, length):
    return -(-length // c["block"])


def _capacity(c):
    unit = max(c["block"], c["page"], 64)
    return -(-c["len_max"] // unit) * unit


def _lengths(c):
    """Spread evenly over [len_min, len_max] in no particular order; the same for every seed."""
    if c["len_min"] == c["len_max"]:
        return [c["len_max"]] * c["batch"]
    span = c["len_max"] - c["len_min"]
    return [c["len_min"] + int(span * ((i + 1) * 0.6180339887498949 % 1.0)) for i in range(c["batch"])]


def _keep(c, n):
    """Blocks of a list of a sequence of n blocks."""
    if c["kind"] == "sparse":
        return synth.keep_count(n, c["sparsity"])
    if c["kind"] == "threshold":
        return _threshold_keep(c, n)
    if c["kind"] == "dense":
        return n
    return min(max(1, c["budget"] // c["block"]), n)


def _threshold_keep(c, n):
    """Expected list length: that of scores normal with standard deviation 1.1, i.e. the probability that a normal
    variable exceeds (log(n tau) + s^2 / 2) / s.  The scores that ``prepare`` leads to have heavier tails (the rotary
    embedding makes them wander along the sequence), but the measured lists are within 20 % of it (103 blocks on
    average for 90 expected, 52 for 55, 7.8 for 6, 9.8 for 9)."""
    s = 1.1
    z = (math.log(max(n, 1) * c["threshold"]) + s * s / 2) / s
    return min(n, 1 + int(n * 0.5 * math.erfc(z / math.sqrt(2))))


def work(case):
    """What the call cannot do without: selected K and V once, compressed keys and gate weights once, pre-RoPE keys of a
    build once, queries, lists and results."""
    c = case
    B, hq, hkv, b, dg, ql = c["batch"], c["hq"], c["hkv"], c["block"], c["d_gate"], c["q_len"]
    g = hq // hkv
    byts = flops = 0
    lens = _lengths(c)
    if c["kind"] == "build":
        for L in lens:
            n = L // b
            byts += hkv * n * (b * D * 2 + dg * 2)
            flops += hkv * n * (3 * b * D + 2 * dg * 3 * D)
        return {"bytes": byts + hkv * dg * 3 * D * 2, "flops": flops}
    for L in lens:
        n = _blocks(c, L)
        k = _keep(c, n)
        tokens = min(L, k * b)
        byts += hkv * tokens * D * 2 * 2 + 2 * ql * hq * D * 2 + ql * hq * 4
        flops += 4 * ql * hq * tokens * D
        if c["kind"] != "dense":
            byts += hkv * k * 4
        if c["kind"] in ("step", "multi", "threshold"):
            byts += hkv * (L // b) * dg * 2 + ql * hq * D * 2
            flops += 2 * ql * hkv * (L // b) * dg + 2 * ql * hq * D * dg
            if c["kind"] != "threshold" and L % b < ql:
                byts += hkv * (b * D * 2 + dg * 2)
    if c["kind"] in ("step", "multi", "threshold"):
        byts += hkv * dg * g * D * 2
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    """bf16 inputs and outputs, fp32 accumulation.  Against the same sums in 64 bits the attention output is off by
    2.0e-3 to 2.3e-3 in the 2-norm and by 6e-3 to 1e-2 of the larger of value and root mean square at most (bf16
    output, bf16 probabilities), compressed keys by 4e-5 to 8e-5 and 8e-3 (single bf16 steps); the log-sum-exp by
    5e-8.  Four times that is stated.  Lists are whole numbers: a block whose score equals the last one taken to within
    fp32 rounding can change places with it, which moves the entries between the two by one place."""
    if case["kind"] == "build":
        return {"rel": 4e-4, "max": 0.032}
    if case["kind"] in ("step", "multi", "threshold"):
        return {"rel": 8e-3, "max": 0.04, "differ": 0.005}
    return {"rel": 8e-3, "max": 0.04}


def _rand(shape, g, std=1.0):
    t = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    return t if std == 1.0 else t.mul_(std)


def _cache(c, g):
    """One of K or V: [B, Hkv, S, d] (head- or token-major in memory) or a page pool [pages, Hkv, P, d]."""
    B, hkv, S = c["batch"], c["hkv"], _capacity(c)
    if c["page"]:
        return _rand((B * S // c["page"], hkv, c["page"], D), g)
    if c["token_major"]:
        return _rand((B, S, hkv, D), g).permute(0, 2, 1, 3)
    return _rand((B, hkv, S, D), g)


def _compress(c, k, table, w_k):
    """The compressed-key cache that decoding starts from: pooled keys, projected and rotated (plain torch)."""
    B, hkv, b, dg = c["batch"], c["hkv"], c["block"], c["d_gate"]
    outer, _, rows, _ = k.shape
    n = _capacity(c) // b
    kb = k.unflatten(2, (rows // b, b))
    feat = torch.cat([kb.amax(3).float(), kb.amin(3).float(), kb.mean(3, dtype=torch.float32)], -1)
    if table is not None:
        feat = feat[table.long()].transpose(1, 2)                            # [B, Hkv, pages, P/b, 3d]
    feat = feat.reshape(B, hkv, n, 3 * D)
    y = torch.einsum("bhnf,hcf->bhnc", feat, w_k.float())
    pos = torch.arange(n, device="cuda", dtype=torch.float64) * b
    freq = THETA ** (-2.0 * torch.arange(dg // 2, device="cuda", dtype=torch.float64) / dg)
    ang = pos[:, None] * freq[None, :]
    cs, sn = ang.cos().float(), ang.sin().float()
    a, d = y[..., : dg // 2], y[..., dg // 2:]
    return torch.cat([a * cs - d * sn, d * cs + a * sn], -1).to(torch.bfloat16).contiguous()


class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + 17)
    B, hq, hkv, b, dg, ql = c["batch"], c["hq"], c["hkv"], c["block"], c["d_gate"], c["q_len"]
    lens = _lengths(c)
    s.kind, s.q_len, s.budget, s.threshold = c["kind"], ql, c["budget"], c["threshold"]
    s.ctx = _context()
    s.shape = binding.make_shape(B, hq, hkv, D, b, SCALE)
    s.lens = torch.tensor(lens, dtype=torch.int32, device="cuda")
    S = _capacity(c)
    n_max = S // b
    if s.kind == "build":
        # pre-RoPE keys as prefill leaves them
        s.k_nope = _cache(c, g)
        s.w_k = _rand((hkv, dg, 3 * D), g, GATE_STD)
        s.kcomp = torch.zeros((B, hkv, n_max, dg), dtype=torch.bfloat16, device="cuda")
        s.gate = binding.make_gate(dg, THETA, None, s.w_k, s.kcomp, n_max)
        s.n = max(L // b for L in lens)
        return s
    s.k, s.v = _cache(c, g), _cache(c, g)
    table = None
    if c["page"]:
        table = torch.randperm(B * S // c["page"], generator=g, device="cuda").to(torch.int32).view(B, -1)
    s.table = table
    s.kv = binding.make_kv(s.k, s.v, s.lens, S, table, c["page"])
    q_shape = (B, ql, hq, D) if s.kind == "multi" else (B, hq, D)
    s.q = _rand(q_shape, g)
    s.out = torch.empty_like(s.q)
    s.lse = torch.empty(q_shape[:-1], dtype=torch.float32, device="cuda")
    if s.kind == "dense":
        return s
    n_seq = [_blocks(c, L) for L in lens]
    if s.kind == "sparse":
        s.max_sel = max(_keep(c, n) for n in n_seq)
        idx, cnt = synth.random_block_lists(lens, hkv, b, [_keep(c, n) for n in n_seq], s.max_sel, int(seed))
        s.idx, s.cnt = torch.from_numpy(idx).cuda(), torch.from_numpy(cnt).cuda()
        return s
    s.max_sel = max(1, n_max // 4) if s.kind == "threshold" else max(1, min(s.budget // b, n_max))
    s.idx = torch.empty((B, hkv, s.max_sel), dtype=torch.int32, device="cuda")
    s.cnt = torch.empty((B, hkv), dtype=torch.int32, device="cuda")
    std = PEAKED_GATE_STD if s.kind == "threshold" else GATE_STD
    s.w_q = _rand((hkv, dg, hq // hkv * D), g, std)
    s.w_k = _rand((hkv, dg, 3 * D), g, std)
    s.q_nope = _rand(q_shape, g)
    s.kcomp = _compress(c, s.k, table, s.w_k)
    s.gate = binding.make_gate(dg, THETA, s.w_q, s.w_k, s.kcomp, n_max)
    # the rolling window of the newest block's pre-RoPE keys that a decode loop keeps
    s.window = _rand((B, hkv, b, D), g)
    return s


def run(s):
    """One call; the results are the state's own output buffers, as in a decode loop."""
    if s.kind == "step":
        s.ctx.seer_decode_step(s.shape, s.kv, s.gate, s.q, s.q_nope, s.window, s.budget, s.idx, s.cnt, s.max_sel, s.out,
                               s.lse, rows_block_local=True)
        return {"out": s.out, "lse": s.lse, "idx": s.idx, "cnt": s.cnt, "kcomp": s.kcomp}
    if s.kind == "multi":
        s.ctx.seer_decode_step_multi(s.shape, s.kv, s.gate, s.q, s.q_nope, s.q_len, s.window, s.budget, s.idx, s.cnt,
                                     s.max_sel, s.out, s.lse, rows_block_local=True)
        return {"out": s.out, "lse": s.lse, "idx": s.idx, "cnt": s.cnt, "kcomp": s.kcomp}
    if s.kind == "threshold":
        s.ctx.seer_gate_select_threshold(s.shape, s.gate, s.lens, s.q_nope, None, s.threshold, s.idx, s.cnt, s.max_sel)
        s.ctx.seer_sparse_decode(s.shape, s.kv, s.q, s.idx, s.cnt, s.max_sel, s.out, s.lse)
        return {"out": s.out, "lse": s.lse, "idx": s.idx, "cnt": s.cnt}
    if s.kind == "sparse":
        s.ctx.seer_sparse_decode(s.shape, s.kv, s.q, s.idx, s.cnt, s.max_sel, s.out, s.lse)
        return {"out": s.out, "lse": s.lse}
    if s.kind == "dense":
        s.ctx.seer_dense_decode(s.shape, s.kv, s.q, s.out, s.lse)
        return {"out": s.out, "lse": s.lse}
    s.ctx.seer_kcomp_append(s.shape, s.gate, s.lens, s.k_nope, first_block=0, num_blocks=s.n)
    return {"kcomp": s.kcomp}


# ---- the same results in 64 bits, in plain torch ------------------------------------------------------------------

def _rope(y, pos):
    """Rotate-half pairing (c, c + d_gate/2); y [..., d_gate] float64, pos: one position per row of y's last but one axis."""
    half = y.shape[-1] // 2
    freq = THETA ** (-2.0 * torch.arange(half, device="cuda", dtype=torch.float64) / y.shape[-1])
    ang = pos.to(torch.float64)[:, None] * freq
    a, d = y[..., :half], y[..., half:]
    return torch.cat([a * ang.cos() - d * ang.sin(), d * ang.cos() + a * ang.sin()], -1)


def _pooled(rows, w, first, b):
    """Compressed keys of the complete blocks of `rows` [n * b, d], the first of which is block `first`."""
    x = rows.double().view(-1, b, D)
    feat = torch.cat([x.amax(1), x.amin(1), x.mean(1)], -1)
    return _rope(feat @ w.double().T, (first + torch.arange(len(x), device="cuda")) * b)


def _list64(c, s, i, h, L, max_sel):
    """The blocks that the gate selects for sequence i, KV head h, in ascending order."""
    b, ql, g = c["block"], c["q_len"], c["hq"] // c["hkv"]
    n, j_f = _blocks(c, L), max(0, L - ql) // b
    n_forced = min(n - j_f, max_sel)
    x = s.q_nope.view(c["batch"], ql, c["hq"], D)[i, :, h * g:(h + 1) * g].reshape(ql, g * D).double()
    qg = _rope(x @ s.w_q[h].double().T, (L - ql + torch.arange(ql, device="cuda")).clamp(min=0))
    score = (s.kcomp[i, h, :j_f].double() @ qg.T).amax(1) / math.sqrt(c["d_gate"])
    if c["kind"] == "threshold":
        need = int((score.softmax(0) > c["threshold"]).sum()) if j_f else 0
        need = min(need, max_sel - n_forced)
    else:
        need = min(max(1, c["budget"] // b), n, max_sel) - n_forced
    best = score.sort(descending=True, stable=True).indices[:max(0, min(need, j_f))]
    return torch.cat([best.sort().values, torch.arange(n - n_forced, n, device="cuda")])


def exact(case, seed):
    """What ``run`` returns for these inputs, in 64 bits; no value is given for the lists."""
    c, s = case, prepare(case, seed)
    hkv, b, ql, g, lens = c["hkv"], c["block"], c["q_len"], c["hq"] // c["hkv"], _lengths(c)
    if c["kind"] == "build":
        kcomp = torch.zeros(s.kcomp.shape, dtype=torch.float64, device="cuda")
        for i, L in enumerate(lens):
            for h in range(hkv):
                n = L // b
                kcomp[i, h, :n] = _pooled(s.k_nope[i, h, :n * b], s.w_k[h], 0, b)
        return {"kcomp": kcomp}
    out = torch.zeros((c["batch"], ql, c["hq"], D), dtype=torch.float64, device="cuda")
    lse = torch.full(out.shape[:-1], -math.inf, dtype=torch.float64, device="cuda")
    q = s.q.view(out.shape)
    for i, L in enumerate(lens):
        for h in range(hkv):
            if c["kind"] == "dense":
                blocks = torch.arange(_blocks(c, L), device="cuda")
            elif c["kind"] == "sparse":
                blocks = s.idx[i, h, :int(s.cnt[i, h])].long()
            else:
                blocks = _list64(c, s, i, h, L, s.max_sel)
            t = (blocks[:, None] * b + torch.arange(b, device="cuda")).view(-1)
            t = t[t < L]
            if s.table is None:
                k, v = s.k[i, h, t].double(), s.v[i, h, t].double()
            else:
                page, row = s.table[i].long()[t // c["page"]], t % c["page"]
                k, v = s.k[page, h, row].double(), s.v[page, h, row].double()
            for x in range(ql):
                z = q[i, x, h * g:(h + 1) * g].double() @ k.T * SCALE
                z = z.masked_fill(t > L - ql + x, -math.inf)
                lse[i, x, h * g:(h + 1) * g] = z.logsumexp(1)
                out[i, x, h * g:(h + 1) * g] = z.softmax(1) @ v
    res = {"out": out.view(s.q.shape), "lse": lse.view(s.lse.shape)}
    if c["kind"] not in ("dense", "sparse"):
        res["idx"] = res["cnt"] = None
    if c["kind"] in ("step", "multi"):
        kcomp = s.kcomp.double()
        for i, L in enumerate(lens):
            if L >= b and L % b < ql:
                for h in range(hkv):
                    kcomp[i, h, L // b - 1] = _pooled(s.window[i, h], s.w_k[h], L // b - 1, b)[0]
        res["kcomp"] = kcomp
    return res
