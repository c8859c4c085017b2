"""The work this library is used for, as cases that can be timed and whose outputs can be compared.

Every pass goes through the public entry points of ``paper_2510_19875_b200.stream`` the way a
program that estimates masks and runs the sparse attention on them does. Sizes are those of the
workloads in ``paper_2510_19875_b200/workloads.py`` and of the tests, or plain numbers around
them; inputs follow the same recipe (normal Q, K, V with an attention sink, local windows, anchors
or a needle block), drawn on the GPU.
"""
import math

import numpy as np
import torch

from paper_2510_19875_b200 import stream as S


def _case(name, kind, H, G, T, d, block, k, *, dtype="bf16", batch=1, causal=True, plant="sink", sparsity=0.0, ks=""):
    """kind: what a pass does (see run()). plant: structure in the inputs. sparsity > 0: one k per
    query block from the library's schedule, k the row width. ks: the list of a several-k build."""
    c = dict(kind=kind, batch=batch, H=H, G=G, T=T, d=d, block=block, k=k, dtype=dtype, causal=causal, plant=plant,
             sparsity=sparsity, ks=ks)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest call: one fp32 head in blocks of 32, the setting of a first look at one head
        # (64 rows; launches and latency count)
        _case("head_fp32_2k", "layer", 1, 1, 2048, 64, 32, 8, dtype="f32", plant=""),
        # a small model's layer kept in fp32, length not a multiple of the block
        _case("layer_fp32_5003", "layer", 8, 2, 5003, 64, 32, 8, dtype="f32"),
        # one GQA layer at a short, an ordinary and the longest context: mask, then attention on it
        _case("layer_4k", "layer", 32, 8, 4096, 128, 64, 32),
        _case("layer_16k", "layer", 32, 8, 16384, 128, 64, 16, plant="sink,local"),
        _case("layer_128k", "layer", 32, 8, 131072, 128, 64, 32, plant="sink,anchors"),
        # several layers in one call (batch), seven query heads per kv head, a needle, ragged length
        _case("stack_9999", "layer", 28, 4, 9999, 128, 64, 16, batch=4, plant="needle"),
        # one k per query block, so that late rows are not pruned harder; ragged length
        _case("layer_60001_var_k", "layer", 32, 8, 60001, 128, 64, 32, plant="sink,anchors", sparsity=1 / 64),
        # looking for the smallest sufficient k: several masks at once, what the larger budget keeps
        # beyond the smaller one, and which key blocks attract the later queries (the outputs hold
        # block scores in ascending block order; with a needle only the last rows' scores differ much
        # in size, so that a near tie that falls the other way does not move a huge score by a place)
        _case("search_k_32k", "search", 32, 8, 32768, 128, 64, 32, plant="needle", ks="8,16,32"),
        # a mask row for every query token, and the attention on it
        _case("tokens_4k", "tokens", 32, 8, 4096, 128, 64, 16),
        # tensors that live in pinned host memory: copies, mask, attention and copies back
        _case("host_32k", "host", 32, 8, 32768, 128, 64, 16),
        # a small model in blocks of 32 (the block size the method was published with)
        _case("layer_10k_block_32", "layer", 12, 2, 10007, 128, 32, 8),
        # not causal, a head dimension of 64, every head its own keys, more than 32 blocks per row
        _case("encoder_8k_d64", "layer", 16, 16, 8192, 64, 64, 40, causal=False, plant="local"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: lengths log-uniform and mostly not multiples of a block."""
    what = rng.choice(["layer", "layer", "layer", "fp32", "other", "other", "search", "tokens", "host"])
    H, G = rng.choice([(32, 8), (28, 4), (8, 2), (12, 2), (16, 16), (6, 2)])
    plant = rng.choice(["", "sink", "sink,local", "sink,anchors", "needle"])
    if what == "layer":
        causal = rng.random() < 0.85
        T = _log(rng, 300, 131072 if causal else 49152)
        batch = rng.randint(1, max(1, min(4, 32 * 65536 // (H * T))))
        return _case("", what, H, G, T, 128, 64, rng.randint(4, 32), batch=batch, causal=causal, plant=plant,
                     sparsity=rng.choice([0.0, 0.0, 1 / 32, 1 / 128]))
    if what == "fp32":
        H, G = rng.choice([(1, 1), (4, 1), (8, 2), (6, 2)])
        return _case("", "layer", H, G, _log(rng, 300, 5500), rng.choice([32, 64, 128]), rng.choice([16, 32, 64]),
                     rng.randint(4, 16), dtype="f32", plant=plant)
    if what == "other":  # bf16 in block sizes, head dimensions and widths other than the common ones
        d, block = rng.choice([(64, 64), (64, 32), (128, 32), (128, 64), (256, 64), (128, 16)])
        T = _log(rng, 500, 131072 // H)
        wide = (d, block) == (128, 64) or rng.random() < 0.4
        return _case("", "layer", H, G, T, d, block, rng.randint(33, 64) if wide else rng.randint(4, 32),
                     causal=rng.random() < 0.6, plant=plant)
    if what == "search":
        k = rng.randint(12, 32)
        return _case("", what, H, G, _log(rng, 2000, 32768), 128, 64, k, plant=rng.choice(["", "needle"]), ks="%d,%d,%d" % (k // 4, k // 2, k))
    if what == "tokens":
        return _case("", what, H, G, _log(rng, 300, 131072 // H), 128, 64, rng.randint(6, 16), plant=plant)
    return _case("", "host", H, G, _log(rng, 1000, 32768), 128, 64, rng.randint(8, 32), plant=plant)


# ------------------------------------------------------------------------------------------------
def _inputs(c, seed):
    """Q [B, H, T, d], K and V [B, G, T, d] on the GPU, in the recipe of workloads.py."""
    gen = torch.Generator("cuda").manual_seed(1000003 * seed + 17)
    B, H, G, T, d = c["batch"], c["H"], c["G"], c["T"], c["d"]
    hpg, plant = H // G, c["plant"].split(",")
    dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda")

    def unit(x):
        return x / x.norm(dim=-1, keepdim=True)

    def turned(x, target, cos):  # rows of x at the given cosine with the unit vectors `target`, norms kept
        perp = unit(x - (x * target).sum(-1, keepdim=True) * target)
        return x.norm(dim=-1, keepdim=True) * (cos * target + math.sqrt(1 - cos * cos) * perp)

    q = torch.empty(B, H, T, d, dtype=dt, device="cuda")
    k = torch.empty(B, G, T, d, dtype=dt, device="cuda")
    v = torch.empty(B, G, T, d, dtype=dt, device="cuda")
    for b in range(B):
        for g in range(G):
            kg, qg = normal(T, d), normal(hpg, T, d)
            v[b, g] = normal(T, d)
            if "local" in plant:
                win = normal(-(-T // 256), d).repeat_interleave(256, 0)[:T]
                kg += 0.5 * win
                qg += win
            if "sink" in plant:
                u = unit(normal(d))
                kg[0] = 4 * math.sqrt(d) * u
                qg += 2 * u
            if "anchors" in plant:
                pos = torch.randperm(T - 1, generator=gen, device="cuda")[:64].sort().values + 1
                tok = torch.arange(T, device="cuda").expand(hpg, T)
                before = torch.searchsorted(pos, tok.contiguous())
                chosen = (torch.rand(hpg, T, generator=gen, device="cuda") < 0.1) & (before > 0)
                pick = (torch.rand(hpg, T, generator=gen, device="cuda") * before).long().clamp_(max=pos.numel() - 1)
                qg[chosen] = turned(qg[chosen], unit(kg[pos[pick[chosen]]]), 0.8)
            if "needle" in plant:
                blk = 1 + seed * 7919 % max(1, T // c["block"] // 2 - 1)
                n = unit(normal(d))
                rows = kg[blk * c["block"]:(blk + 1) * c["block"]]
                rows[:] = rows.norm(dim=-1, keepdim=True) * n
                qg[:, -128:] = turned(qg[:, -128:], n, 0.9)
            k[b, g] = kg
            q[b, g * hpg:(g + 1) * hpg] = qg
    return q, k, v


def prepare(case, seed):
    q, k, v = _inputs(case, seed)
    st = dict(case=case, q=q, k=k, v=v, k_row=None)
    blocks = dict(block_q=1 if case["kind"] == "tokens" else case["block"], block_k=case["block"])
    st["blocks"] = blocks
    p = S.make_problem(q, k, k_top=case["k"], causal=case["causal"], **blocks)
    if case["sparsity"] > 0:
        st["k_row"] = S.k_schedule(p, case["sparsity"]).cuda()
    if case["kind"] == "search":
        st["problem"] = p
        st["k_list"] = [int(x) for x in case["ks"].split(",")]
    if case["kind"] == "host":
        for n in ("q", "k", "v"):
            st[n] = st[n].cpu().pin_memory()
        st["mask"] = torch.empty(1, case["H"], S.n_query_blocks(p), case["k"], dtype=torch.int32, pin_memory=True)
        st["out"] = torch.empty(st["q"].shape, dtype=st["q"].dtype, pin_memory=True)
        st["staging"] = torch.empty(S.stream_host_staging_bytes(p), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    c = st["case"]
    if c["kind"] == "host":
        S.run_host(st["q"], st["k"], st["v"], st["mask"], st["out"], st["staging"], k_top=c["k"], causal=c["causal"], **st["blocks"])
        return st["mask"], st["out"]
    if c["kind"] == "search":
        res = S.build_masks(st["q"], st["k"], st["k_list"], causal=c["causal"], want_scores=True, **st["blocks"])
        more, weight = S.mask_difference(res.mask[-1], res.mask[-2], res.scores[-1])
        vertical, kurtosis = S.vertical_scores(st["problem"], res.mask[-1], res.scores[-1])
        return res.mask, res.scores, more, weight, vertical, kurtosis
    res = S.build_mask(st["q"], st["k"], k_top=c["k"], causal=c["causal"], k_row=st["k_row"], **st["blocks"])
    return res.mask, S.sparse_attention(st["q"], st["k"], st["v"], res.mask, causal=c["causal"], **st["blocks"])


# ------------------------------------------------------------------------------------------------
def _counts(c):
    """(block tiles scored, blocks kept) over all rows: a row with n allowed of N key blocks starts
    with its share of the k nodes, scores both halves of each, then one new half of every surviving
    node per level, and keeps min(k, n) blocks."""
    T, block = c["T"], c["block"]
    N = -(-T // block)
    n_row = T if c["kind"] == "tokens" else N
    tok = np.arange(n_row, dtype=np.int64) if c["kind"] == "tokens" else np.minimum((np.arange(n_row) + 1) * block, T) - 1
    n = (tok // block + 1) if c["causal"] else np.full(n_row, N)
    k = np.full(n_row, c["k"])
    if c["sparsity"] > 0:
        k = np.clip(np.floor(1 + (n - 1) * c["sparsity"]), 1, c["k"])
    nodes = np.ceil(np.minimum(k, N) * n / N)
    size = np.ceil(N / k)
    tiles = np.minimum(2 * nodes, n)
    for _ in range(int(math.ceil(math.log2(max(2, size.max()))))):
        nodes = np.minimum(np.minimum(2 * nodes, k), n)
        size = np.ceil(size / 2)
        tiles = tiles + np.where(size > 1, np.minimum(nodes, n), 0)
    heads = c["batch"] * c["H"]
    return heads * float(np.minimum(tiles, n).sum()), heads * float(np.minimum(k, n).sum())


def work(case):
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    B, H, G, T, d = c["batch"], c["H"], c["G"], c["T"], c["d"]
    bq = 1 if c["kind"] == "tokens" else c["block"]
    rows = B * H * -(-T // bq)
    tiles, kept = _counts(c)
    tile_flops = 2.0 * bq * c["block"] * d
    if c["kind"] == "search":  # the masks, their scores, the difference with its weights, the column sums
        n_k = len(c["ks"].split(","))
        return {"bytes": e * B * (H + G) * T * d + 8.0 * rows * c["k"] * (n_k + 1) + 4.0 * B * H * -(-T // c["block"]),
                "flops": tiles * tile_flops}
    return {"bytes": e * B * (2 * H + 2 * G) * T * d + 4.0 * rows * c["k"], "flops": (tiles + 2 * kept) * tile_flops}


def tolerance(case):
    """Measured by running the listed cases and ten drawn ones again with the channels of Q and K in
    another order (same products, sums in another order) and by comparing with the attention in
    64 bits on the same mask; about four times what was seen.

    fp32: rel up to 5e-7, max up to 6e-6. bf16: rel up to 2.4e-3 (the rounding of the output, and of
    the weights P where a kernel keeps them in bf16), max up to 0.09: a row whose k-th and next score
    are a near tie may keep the other block, which changes its output visibly. At most 1e-5 of the
    mask entries did so; where a case has few rows the bound is two rows."""
    rows = case["batch"] * case["H"] * -(-case["T"] // (1 if case["kind"] == "tokens" else case["block"]))
    differ = min(0.01, max(1e-4, 2 / rows))
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4, "differ": differ}
    return {"rel": 1e-2, "max": 0.4, "differ": differ}
