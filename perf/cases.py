"""What the speed of this package is measured on: one pass of each case below is work that a serving
program has the package do, through its public entry points.

Three kinds of case ("path"):

attention   one transformer layer's attention over a mixed batch: the fused QKV of the new tokens goes
            into the paged cache (`append_kv`) and the meta-kernel runs (`run`).  One plan serves all
            layers of a step, so the plan is made in `prepare`, except where "steps" is above zero:
            then a pass is that many consecutive steps of the same requests, each of them planned and
            then run for "layers" layers with caches of their own.  Shared-prefix groups ("groups") run
            on a cache that already holds the new tokens.
fp8         the same over an e4m3 cache (`run_fp8kv`; that cache is filled elsewhere, nothing is appended)
linear      the four Linear operators of one layer (QKV, output, gate + up, down projections) on a chunk
            of tokens (`xy_gemm_run` with its scratch memory)

The lengths of a batch are drawn from "layout", so that a case is the same work for every seed; the
values and the page permutation come from the seed.
"""
import math

import numpy as np
import torch

from paper_2412_18106_b200 import binding as xb
from paper_2412_18106_b200 import gemm as xg
from paper_2412_18106_b200 import workloads as W

D = W.HEAD_DIM
SCALE = 1.0 / math.sqrt(D)


def _attention(name=None, **kw):
    c = dict(path="attention", hq=32, hkv=8, page=128, layout=0, steps=0, layers=1, log=False,
             prefill=0, new_lo=0, new_hi=0, cached_lo=0, cached_hi=0,
             decode=0, kv_lo=0, kv_hi=0, verify=0, nodes_lo=0, nodes_hi=0, vkv_lo=0, vkv_hi=0,
             groups=0, members=0, prefix=0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def _linear(name=None, **kw):
    c = dict(path="linear", tokens=1, hidden=4096, hq=32, hkv=8, inter=14336)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest batch of the test suite (8/2 heads, 16-token pages: two prefill chunks, a decode
        # token, a four-token verify chain), planned and run for two steps: host work and launches.
        _attention("tiny_steps", hq=8, hkv=2, page=16, steps=2, prefill=2, new_lo=64, new_hi=64, cached_lo=0,
                   cached_hi=128, decode=1, kv_lo=300, kv_hi=300, verify=1, nodes_lo=4, nodes_hi=4, vkv_lo=200,
                   vkv_hi=200),
        # A lightly loaded server: two decode steps of 13 sessions with short histories, eight layers each.
        _attention("decode_steps", steps=2, layers=8, decode=13, kv_lo=300, kv_hi=2500),
        # Decode-only batch of the benchmark: 64 requests, 28/4 heads.
        _attention("decode_batch", hq=28, hkv=4, decode=64, kv_lo=512, kv_hi=8192),
        # The same batch over an fp8 cache.
        _attention("decode_fp8", path="fp8", hq=28, hkv=4, decode=64, kv_lo=512, kv_hi=8192),
        # Prompts of 4096 new tokens on reused prefixes.
        _attention("prefill_prefix", prefill=4, new_lo=4096, new_hi=4096, cached_lo=0, cached_hi=4096),
        # Decode requests that share long prompts (4 groups of 32 on 8192 common tokens).
        _attention("decode_shared", groups=4, members=32, prefix=8192, kv_lo=0, kv_hi=1024),
        # Speculative verification: 32 trees of 8 .. 64 nodes, 64/8 heads.
        _attention("verify_trees", hq=64, hkv=8, verify=32, nodes_lo=8, nodes_hi=64, vkv_lo=1024, vkv_hi=32768),
        # Chunked prefill beside decode: a 2048-token chunk on 6144 cached tokens and 48 decode requests.
        _attention("splitfuse", prefill=1, new_lo=2048, new_hi=2048, cached_lo=6144, cached_hi=6144, decode=48,
                   kv_lo=1024, kv_hi=16384),
        # Full serving mix of the benchmark: 96 requests, prompts of 128 .. 4096 new tokens on reused
        # prefixes, decode and verify on 256 .. 64k cached tokens.  The largest case.
        _attention("full_mix", hq=64, hkv=8, log=True, prefill=19, new_lo=128, new_hi=4096, cached_lo=64,
                   cached_hi=16384, decode=58, kv_lo=256, kv_hi=65536, verify=19, nodes_lo=4, nodes_hi=32,
                   vkv_lo=256, vkv_hi=65536),
        # Linear operators of a decode batch, of a ragged mixed chunk and of a full prefill chunk.
        _linear("linear_decode", tokens=16),
        _linear("linear_chunk", tokens=333),
        _linear("linear_prefill", tokens=4096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: batches from one request to a hundred, contexts from a few
    tokens to half a million, chunks from one token to 4096; the cost stays below full_mix."""
    kind = rng.choice(["decode", "decode", "steps", "fp8", "long", "shared", "verify", "prefill", "mix", "mix",
                       "linear", "linear", "linear"])
    if kind == "linear":
        hq, hkv, hidden, inter = rng.choice([(32, 8, 4096, 14336), (28, 4, 3584, 18944), (64, 8, 8192, 28672)])
        return _linear(tokens=_log_int(rng, 1, 4096 if hidden < 8192 else 2048), hidden=hidden, hq=hq, hkv=hkv, inter=inter)
    hq, hkv = rng.choice([(8, 2), (28, 4), (32, 8), (64, 8)])
    c = _attention(hq=hq, hkv=hkv, page=rng.choice([16, 32, 64, 128, 128, 128]), layout=rng.randrange(1 << 20),
                   log=rng.random() < 0.5)
    hi = _log_int(rng, 1000, 65536)
    kv = dict(kv_lo=rng.randrange(1, 1 + hi // 4), kv_hi=hi)
    verify = dict(nodes_lo=rng.randrange(2, 9), nodes_hi=rng.randrange(9, 65), vkv_lo=kv["kv_lo"], vkv_hi=hi)
    chunk = _log_int(rng, 64, 4096)
    prefill = dict(new_lo=rng.randrange(1 + chunk // 8, chunk + 1), new_hi=chunk, cached_lo=1,
                   cached_hi=_log_int(rng, 2, 16384))
    if kind == "steps":
        c.update(steps=2, layers=rng.randrange(1, 9), decode=_log_int(rng, 1, 48), kv_lo=rng.randrange(1, 300),
                 kv_hi=rng.randrange(301, 4000), verify=rng.randrange(0, 3), nodes_lo=2, nodes_hi=9, vkv_lo=50,
                 vkv_hi=2000)
    elif kind in ("decode", "fp8"):
        c.update(kv, path="fp8" if kind == "fp8" else "attention", decode=_log_int(rng, 4, 128))
    elif kind == "long":
        c.update(log=True, decode=rng.randrange(1, 7), kv_lo=_log_int(rng, 50000, 131072), kv_hi=_log_int(rng, 131073, 524288))
    elif kind == "shared":
        c.update(groups=rng.randrange(1, 6), members=rng.randrange(6, 49), prefix=128 * rng.randrange(8, 129), kv_lo=0,
                 kv_hi=rng.randrange(1, 2048))
    elif kind == "verify":
        c.update(verify, verify=_log_int(rng, 2, 48))
    elif kind == "prefill":
        c.update(prefill, prefill=_log_int(rng, 1, 8))
    else:
        c.update(kv)
        c.update(verify)
        c.update(prefill, prefill=rng.randrange(1, 20), decode=rng.randrange(8, 64), verify=rng.randrange(0, 20))
    # not dearer than the largest listed case: fewer requests until the estimate fits
    while True:
        w = work(c)
        if max(w["bytes"] / 4.5e12, w["flops"] / 7e14) < 5e-3:
            return c
        for k in ("prefill", "decode", "verify", "members"):
            c[k] = (c[k] + 1) // 2 if c[k] > 1 else c[k]
        c["new_hi"], c["new_lo"] = max(c["new_lo"], c["new_hi"] * 2 // 3), c["new_lo"]
        c["kv_hi"], c["vkv_hi"] = max(c["kv_lo"], c["kv_hi"] * 2 // 3), max(c["vkv_lo"], c["vkv_hi"] * 2 // 3)


def _requests(case):
    """Lengths and trees of the batch at its first step, in a shuffled order (groups stay together)."""
    rng = np.random.default_rng(case["layout"])

    def length(lo, hi):
        if hi <= lo:
            return int(lo)
        return W._log_uniform_int(rng, max(lo, 1), hi) if case["log"] else int(rng.integers(lo, hi + 1))

    reqs = [(1, case["prefix"] + length(case["kv_lo"], case["kv_hi"]), None)
            for _ in range(case["groups"] * case["members"])]
    if not reqs:
        for _ in range(case["prefill"]):
            reqs.append((length(case["new_lo"], case["new_hi"]), length(case["cached_lo"], case["cached_hi"]), None))
        for _ in range(case["decode"]):
            reqs.append((1, length(case["kv_lo"], case["kv_hi"]), None))
        for _ in range(case["verify"]):
            n = int(rng.integers(case["nodes_lo"], case["nodes_hi"] + 1))
            reqs.append((n, length(case["vkv_lo"], case["vkv_hi"]), W.random_tree(rng, n, 8)))
        reqs = [reqs[i] for i in rng.permutation(len(reqs))]
    return reqs


def _batch(case, seed):
    """The batch as it stands after its last step (so that the pages suffice for all steps)."""
    reqs = _requests(case)
    more = max(case["steps"], 1) - 1
    kinds = [W.MASK_CAUSAL if t is None else W.MASK_TREE for _, _, t in reqs]
    b = W.assemble("case", case["hq"], case["hkv"], case["page"], [r[0] for r in reqs],
                   [r[1] + more * r[0] for r in reqs], kinds, [r[2] for r in reqs], np.random.default_rng(seed), seed)
    if case["groups"]:  # the members of a group hold the same pages for the common prefix
        pages = case["prefix"] // case["page"]
        for g in range(case["groups"]):
            first = g * case["members"]
            b.block_table[first:first + case["members"], :pages] = b.block_table[first, :pages]
    return b


def _randn(shape, gen, std=1.0):
    return torch.empty(shape, dtype=torch.bfloat16, device="cuda").normal_(0.0, std, generator=gen)


def _e4m3(pool):
    """e4m3 bytes of a bf16 pool and one scale per (page, kv head)."""
    scale = (pool.abs().amax(dim=(2, 3)).float() / 448.0).clamp_min(2.0 ** -20)
    out = torch.empty(pool.shape, dtype=torch.uint8, device="cuda")
    for p in range(0, pool.shape[0], 512):
        q = (pool[p:p + 512].float() / scale[p:p + 512, :, None, None]).to(torch.float8_e4m3fn)
        out[p:p + 512] = q.view(torch.uint8)
    return out, scale.contiguous()


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if case["path"] == "linear":
        M, hid, att = case["tokens"], case["hidden"], case["hq"] * D
        ops = []
        for N, K in (((case["hq"] + 2 * case["hkv"]) * D, hid), (hid, att), (2 * case["inter"], hid), (hid, case["inter"])):
            ops.append((_randn((M, K), gen), _randn((N, K), gen, K ** -0.5),
                        torch.empty((M, N), dtype=torch.bfloat16, device="cuda")))
        return dict(case=case, ops=ops, scratch=xg.xy_gemm_workspace("cuda"))
    b = _batch(case, seed)
    fp8 = case["path"] == "fp8"
    steps, layers = max(case["steps"], 1), case["layers"]
    ctx = xb.XYAttn(case["hq"], case["hkv"], case["page"], max_requests=max(256, b.num_requests + case["groups"]),
                    max_q_tokens=max(1 << 15, b.total_q), max_pages_per_req=max(1024, b.block_table.shape[1]),
                    kv_dtype=xb.XY_KV_FP8_E4M3 if fp8 else xb.XY_KV_BF16)
    s = dict(case=case, ctx=ctx, batch=b)
    s["table"] = torch.from_numpy(np.where(b.block_table < 0, 0, b.block_table).astype(np.int32)).cuda()
    s["kv"] = [b.kv_len - (steps - 1 - k) * b.q_len for k in range(steps)]
    pool = (b.num_pages, case["hkv"], case["page"], D)
    s["pools"] = [(_randn(pool, gen), _randn(pool, gen)) for _ in range(layers)]
    s["qkv"] = [[_randn((b.total_q, case["hq"] + 2 * case["hkv"], D), gen) for _ in range(layers)] for _ in range(steps)]
    if fp8:
        (k, ks), (v, vs) = _e4m3(s["pools"][0][0]), _e4m3(s["pools"][0][1])
        s["pools"], s["scales"] = [(k, v)], (ks, vs)
    s["out"] = [[(torch.empty((b.total_q, case["hq"], D), dtype=torch.bfloat16, device="cuda"),
                  torch.empty((b.total_q, case["hq"]), dtype=torch.float32, device="cuda"))
                 for _ in range(layers)] for _ in range(steps)]
    if case["steps"]:
        # The chunks of a serving stream do not come twice; here they do, so their plans are not cached.
        ctx.plan_cache(0)
    else:
        ctx.plan_batch(b, groups="auto" if case["groups"] else None)
    return s


def run(state):
    case = state["case"]
    if case["path"] == "linear":
        for a, w, c in state["ops"]:
            xg.xy_gemm_run(a, w, c, workspace=state["scratch"])
        return [c for _, _, c in state["ops"]]
    ctx, b, table, hq = state["ctx"], state["batch"], state["table"], case["hq"]
    if case["path"] == "fp8":
        (k, v), (o, lse) = state["pools"][0], state["out"][0][0]
        ctx.run_fp8kv(state["qkv"][0][0][:, :hq], k, v, *state["scales"], table, SCALE, o, lse)
        return [o, lse]
    for step, kv_len in enumerate(state["kv"]):
        if case["steps"]:
            ctx.plan(b.q_len, kv_len, b.mask_kind, b.parent_off, b.parents)
        for layer, (k, v) in enumerate(state["pools"]):
            qkv, (o, lse) = state["qkv"][step][layer], state["out"][step][layer]
            if not case["groups"]:
                ctx.append_kv(qkv, k, v, table)
            ctx.run(qkv[:, :hq], k, v, table, SCALE, o, lse)
    return [state["out"], state["pools"]]


def work(case):
    if case["path"] == "linear":
        M, hid, att, inter = case["tokens"], case["hidden"], case["hq"] * D, case["inter"]
        n = [((case["hq"] + 2 * case["hkv"]) * D, hid), (hid, att), (2 * inter, hid), (hid, inter)]
        return dict(bytes=2 * sum(M * K + N * K + M * N for N, K in n), flops=2 * M * sum(N * K for N, K in n))
    reqs = _requests(case)
    hq, hkv, fp8 = case["hq"], case["hkv"], case["path"] == "fp8"
    nbytes = flops = 0
    for step in range(max(case["steps"], 1)):
        tokens = keys = pairs = 0
        for n, kv, tree in reqs:
            h = kv + step * n
            tokens += n
            keys += n + h - case["prefix"]
            if tree is None:
                pairs += n * h + n * (n + 1) // 2
            else:
                depth = np.zeros(n, dtype=np.int64)
                for i in range(n):
                    depth[i] = 1 if tree[i] < 0 else depth[tree[i]] + 1
                pairs += n * h + int(depth.sum())
        keys += case["groups"] * case["prefix"]  # a common prefix is read once
        kv_row = 2 * hkv * (D * (1 if fp8 else 2) + (8.0 / case["page"] / 2 if fp8 else 0))
        nbytes += keys * kv_row + tokens * hq * (4 * D + 4) + 4 * keys // case["page"]
        if not fp8 and not case["groups"]:
            nbytes += tokens * 2 * hkv * D * 4  # the new tokens' K and V rows, read and written into the cache
        flops += 4 * D * hq * pairs
    return dict(bytes=case["layers"] * nbytes, flops=case["layers"] * flops)


def tolerance(case):
    # Outputs are rounded once to bf16 (2^-9 at most), the probabilities of attention once more before
    # P V.  Measured against fp64: attention rel 2.2e-3 .. 2.4e-3, max 0.8e-2 .. 1.0e-2; linear 1.7e-3, 3.9e-3.
    if case["path"] == "linear":
        return {"rel": 6.6e-3, "max": 0.016}
    return {"rel": 9e-3, "max": 0.04}
