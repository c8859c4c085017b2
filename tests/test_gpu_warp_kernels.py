"""The kernels behind the shapes other than 64 x 64 blocks at d = 128 (mma.sync, fp32 FMA, per-token
attention on tcgen05) against the CPU oracle, at the sizes where their tiles,
remainders and launch shapes change: masks bit for bit outside near-ties, attention within
tolerance, also on arbitrary masks (holes, empty rows, a block twice in a row)."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

from helpers import compare_masks, oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S, assert_mask_parity  # noqa: F401  (S: fixture)

pytestmark = pytest.mark.gpu

# fp32: the products' and sums' rounding. bf16: half a unit in the last place of an output of size up
# to 4 is 2^-7 = 7.8e-3 (8 bits), the fp32 sums add less than 1e-4.
TOL = {"f32": 1e-4, "bf16": 8e-3}

CASES = [  # spec changes, block_q, block_k (None: the spec's block), causal
    (dict(), None, None, True),                                        # bf16, d = 64, blocks of 32, few rows: wide CTAs
    (dict(d=128, T=1003), None, None, True),
    (dict(d=128, T=1003, n_q_heads=16), None, None, True),             # more rows than SMs: the four-warp form
    (dict(d=256, T=600, block=64), None, None, False),
    (dict(block=16, k_top=40, T=2001), None, None, True),              # more candidates than two words of slots
    (dict(block=64, k_top=100, T=5000), None, None, True),             # k covers every block
    (dict(d=128, T=515), 1, 16, True),                                 # per-token rows, merged walk
    (dict(T=515), 1, 64, True),
    (dict(d=128, T=515, k_top=7), 5, 24, True),                        # a row's tokens straddle warps; odd key block
    (dict(d=128, T=515, k_top=7), 24, 16, True),
    (dict(d=128, T=700, k_top=7), 48, 64, False),
    (dict(d=128, T=9000, k_top=6, block=64, n_q_heads=2, n_kv_heads=1), 8, 64, True),  # two windows of key blocks
    (dict(d=128, block=64, k_top=1, T=64), None, None, True),          # a single key block
    (dict(d=128, T=1, k_top=3), None, None, True),                     # a single token
    (dict(d=128, T=515, k_top=7), 1, 64, True),                        # per-token attention on tcgen05: tokens beyond T
    (dict(d=128, T=128, k_top=2), 1, 64, False),
    (dict(d=128, T=9000, k_top=1, n_q_heads=2, n_kv_heads=1), 1, 64, True),  # (arbitrary masks) whole groups of tokens that keep nothing
    (dict(d=128, T=700, k_top=7, n_q_heads=3, n_kv_heads=1), 5, 64, False),  # rows that straddle 128 tokens
    (dict(d=128, T=33000, k_top=4, n_q_heads=1, n_kv_heads=1), 1, 64, True),  # two windows of 512 key blocks
    (dict(block=64, T=1003, n_q_heads=3, n_kv_heads=1, k_top=7), None, None, True),   # attention on tcgen05, d = 64: a row alone in its pair
    (dict(d=128, T=515, n_q_heads=7, n_kv_heads=1), None, None, True),                # blocks of 32: four rows across query blocks, three left over
    (dict(d=128, T=515, n_q_heads=5, n_kv_heads=1, k_top=512), None, None, False),    # mask rows as long as they go with four to a unit
    (dict(d=128, T=515, k_top=7), 16, 64, True),                       # 16 tokens a row, 64 keys a tile: groups as shared memory allows
    (dict(d=256, T=515, k_top=7), 16, 32, True),
    (dict(d=256, T=515, k_top=7), 16, 64, False),
    (dict(d=256, T=515, k_top=7), 32, 64, True),
    (dict(d=256, T=2003, k_top=4, n_q_heads=8), 16, 64, True),         # the same with more rows than three an SM
    (dict(dtype="f32", T=1003, n_q_heads=8), None, None, True),
    (dict(dtype="f32", T=515, d=128, k_top=40, block=16), None, None, True),
    (dict(dtype="f32", T=300, block=64, n_q_heads=1, n_kv_heads=1, k_top=8), None, None, True),    # a row over eight CTAs
    (dict(dtype="f32", T=2047, n_q_heads=1, n_kv_heads=1, k_top=7), None, None, False),            # over two
    (dict(dtype="f32", T=300, d=256, block=64, k_top=3), None, None, False),
    (dict(dtype="f32", T=300, d=16, k_top=3), 1, 24, True),
    (dict(dtype="f32", T=300, d=256, block=64, n_q_heads=1, n_kv_heads=1, k_top=1024), None, None, True),  # sixteen warps a row do not fit
    (dict(d=16, T=1003, block=24), None, None, True),                  # bf16 on the fp32-FMA kernels
    (dict(d=32, T=515, n_q_heads=16), 8, 64, False),
]


@pytest.mark.parametrize("kw,bq,bk,causal", CASES)
def test_masks_and_attention_at_tile_edges(S, kw, bq, bk, causal):
    base = dict(name="w", seed=5, batch=1, n_q_heads=4, n_kv_heads=2, T=700, d=64, block=32, k_top=5, dtype="bf16")
    spec = wl.WorkloadSpec(**{**base, **kw})
    w = wl.generate(spec)
    q, k, v = w.torch_tensors("cuda")
    BQ, BK = bq or spec.block, bk or spec.block
    p = oracle_problem(spec, block_q=bq, block_k=bk, causal=causal)
    nqb = so.num_query_blocks(p)
    n_rows = spec.n_q_heads * nqb
    rows = np.arange(n_rows) if n_rows <= 3000 else np.unique(np.random.default_rng(1).choice(n_rows, 1500, replace=False))
    res = S.build_mask(q, k, block_q=BQ, block_k=BK, k_top=spec.k_top, causal=causal, want_scores=True, row_tiles=True)
    ora = so.build_mask_rows(p, w.q, w.k, rows, want_scores=True)
    got = res.mask.cpu().numpy().reshape(-1, spec.k_top)[rows]
    assert res.stats().error == 0 and compare_masks(got, ora)["bad"] == 0
    same = (got == ora["mask"]).all(1)
    scores = res.scores.cpu().numpy().reshape(-1, spec.k_top)[rows]
    np.testing.assert_allclose(scores[same], ora["scores"][same], rtol=2e-5, atol=2e-5)
    sure = same & (ora["min_gap"] >= 1e-5)
    tiles = res.row_tiles().cpu().numpy().reshape(-1)[rows].astype(np.int64)
    assert (tiles[sure] == ora["tiles"][sure]).all()

    rng = np.random.default_rng(3)
    arbitrary = rng.integers(0, -(-spec.T // BK), size=(n_rows, spec.k_top)).astype(np.int32)
    arbitrary[rng.random(arbitrary.shape) < 0.3] = -1
    arbitrary[rng.random(n_rows) < 0.1] = -1
    for mask in (res.mask.cpu().numpy().reshape(n_rows, -1), arbitrary):
        out = S.sparse_attention(q, k, v, torch.from_numpy(mask.reshape(res.mask.shape)).cuda(), block_q=BQ, block_k=BK, causal=causal)
        out = out.float().cpu().numpy().reshape(-1, spec.T, spec.d)
        ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask[rows], rows)
        for i, rid in enumerate(rows):
            bh, qb = divmod(int(rid), nqb)
            lo, hi = qb * BQ, min(spec.T, qb * BQ + BQ)
            assert np.abs(out[bh, lo:hi] - ref[i, : hi - lo]).max() <= TOL[spec.dtype], rid


@pytest.mark.parametrize("k_top", [624, 1024])  # the largest k at which sixteen warps a row fit, the largest there is
@pytest.mark.parametrize("dtype,impl", [("f32", "auto"), ("bf16", "generic")])
def test_masks_of_few_rows_at_the_largest_k(S, dtype, impl, k_top):
    """d = 256 in blocks of 64 on the fp32-FMA form, 76 rows: one k, and two k in one call."""
    spec = wl.WorkloadSpec("k", 12, 1, 1, 1, 4801, 256, 64, k_top, dtype)
    w = wl.generate(spec)
    assert_mask_parity(S, w, None, impl=impl)
    q, k, _ = w.torch_tensors("cuda")
    both = S.build_masks(q, k, [3, k_top], block_q=64, block_k=64, impl=impl).mask
    for got, kq in zip(both, (3, k_top)):
        assert torch.equal(got[..., :kq], S.build_mask(q, k, block_q=64, block_k=64, k_top=kq, impl=impl).mask)


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d,bq,bk", [(16, 48, 24), (64, 20, 64), (128, 16, 48), (256, 64, 16)])
@pytest.mark.parametrize("pitch,start", [(1, 0), (2, 2), (4, 4), (8, 1)])  # elements between rows, in front of the first
def test_rows_off_the_vector_loads_give_the_same_bits(S, dtype, d, bq, bk, pitch, start):
    """The fp32-FMA kernels read keys and values 16, 8 or 4 bytes at a time, or one by one, as the rows lie; the sums are the
    same, and nothing beside the rows is used (NaN there)."""
    torch.manual_seed(d + pitch)

    def rows(heads):
        room = torch.full((start + heads * 403 * (d + pitch),), float("nan"), device="cuda", dtype=dtype)
        x = room[start:].view(1, heads, 403, d + pitch)[..., :d]
        x.copy_(torch.randn(1, heads, 403, d, device="cuda"))
        return x

    q, k, v = rows(4), rows(2), rows(2)
    kw = dict(block_q=bq, block_k=bk, impl="generic")
    plain = [x.contiguous() for x in (q, k, v)]
    got, ref = (S.build_mask(x, y, k_top=7, want_scores=True, **kw) for x, y in ((q, k), plain[:2]))
    assert torch.equal(got.mask, ref.mask) and torch.equal(got.scores, ref.scores)
    assert torch.equal(S.sparse_attention(q, k, v, ref.mask, **kw), S.sparse_attention(*plain, ref.mask, **kw))


@pytest.mark.parametrize("bq", [64, 1])
@pytest.mark.parametrize("shift,scale", [(0.0, 8.0), (-40.0, 1.0), (40.0, 1.0), (-40.0, 6.0)])
def test_attention_with_logits_far_from_the_reference(S, bq, shift, scale):
    """Logits of several hundred in size, all far below zero, or growing along the row: the tcgen05
    attention kernels keep a reference per token instead of a running maximum, and move it."""
    spec = wl.WorkloadSpec("far", 9, 1, 3, 1, 900, 128, 64, 6, "bf16")
    w = wl.generate(spec)
    q, k, v = w.torch_tensors("cpu")
    u = torch.ones(128) / 128 ** 0.5
    ramp = torch.linspace(0.2, 1.0, spec.T)[:, None]  # later keys lie further out
    qf = q.float() * scale + 25 * u
    kf = k.float() * ramp + shift * ramp * u
    w.q = wl.to_bf16_bits(qf.numpy())
    w.k = wl.to_bf16_bits(kf.numpy())
    q, k, v = w.torch_tensors("cuda")
    p = oracle_problem(spec, block_q=bq)
    n_rows = spec.n_q_heads * so.num_query_blocks(p)
    mask = np.random.default_rng(2).integers(0, spec.n_blocks, size=(n_rows, spec.k_top)).astype(np.int32)
    mask[np.random.default_rng(4).random(mask.shape) < 0.2] = -1
    out = S.sparse_attention(q, k, v, torch.from_numpy(mask.reshape(1, spec.n_q_heads, -1, spec.k_top)).cuda(), block_q=bq, block_k=64)
    S.stream_check_device_status()
    out = out.float().cpu().numpy().reshape(-1, spec.T, spec.d)
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask, None)
    nqb = so.num_query_blocks(p)
    # The output's rounding to bf16 is up to 2^-8 of its size. The logits reach 500: 2^-22 of that each for
    # their fp32 sums, their scaling and the exponential's argument make the weights, and with them an
    # output of size up to 5, uncertain by 2e-3. Weights in bf16 (block_q = 64) add 2^-8 of a value's size.
    few = 2e-3 if bq == 1 else 2e-3 + 5 / 256
    for rid in range(n_rows):
        bh, qb = divmod(rid, nqb)
        lo, hi = qb * bq, min(spec.T, qb * bq + bq)
        want = ref[rid, : hi - lo]
        assert (np.abs(out[bh, lo:hi] - want) <= few + np.abs(want) / 256).all(), rid


@pytest.mark.parametrize("d,bq,bk", [(128, 64, 64), (64, 64, 64), (128, 32, 32), (64, 32, 32), (128, 1, 64)])
def test_attention_with_references_that_move_at_many_entries(S, d, bq, bk):
    """The logits of a token grow, fall or stay from block to block, each lane of a warp in its own way: the
    tcgen05 attention kernels hand the references that move on between two groups of warps, lane by
    lane. One stale reference and a weight is off by 2^30 or more; and every launch gives the same bits."""
    spec = wl.WorkloadSpec("moves", 10, 1, 3, 1, 900, d, bk, 6, "bf16")
    w = wl.generate(spec)
    q, k, v = w.torch_tensors("cpu")
    u = torch.ones(d) / d ** 0.5
    slope = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, size=(1, 3, spec.T, 1)).astype(np.float32))
    level = torch.arange(spec.T)[:, None] // bk * (bk / 64)  # a slope of 1: 30 a block of 64, 43 in the exponents of two
    w.q = wl.to_bf16_bits((q.float() + d ** 0.5 * slope * u).numpy())
    w.k = wl.to_bf16_bits((k.float() * 0.5 + 30 * level * u).numpy())
    q, k, v = w.torch_tensors("cuda")
    p = oracle_problem(spec, block_q=bq, block_k=bk)
    nqb = so.num_query_blocks(p)
    mask = np.random.default_rng(6).integers(0, spec.n_blocks, size=(spec.n_q_heads * nqb, spec.k_top)).astype(np.int32)
    blocks = torch.from_numpy(mask.reshape(1, spec.n_q_heads, nqb, spec.k_top)).cuda()
    outs = [S.sparse_attention(q, k, v, blocks, block_q=bq, block_k=bk) for _ in range(20)]
    S.stream_check_device_status()
    assert all(torch.equal(outs[0], o) for o in outs[1:])
    out = outs[0].float().cpu().numpy().reshape(-1, spec.T, d)
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask, None)
    few = 2e-3 + (5 / 256 if (d, bq) == (128, 64) else 0)  # as above: logits of up to 450
    for rid in range(len(mask)):
        bh, qb = divmod(rid, nqb)
        lo, hi = qb * bq, min(spec.T, qb * bq + bq)
        want = ref[rid, : hi - lo]
        assert (np.abs(out[bh, lo:hi] - want) <= few + np.abs(want) / 256).all(), rid

@pytest.mark.parametrize("kw,causal", [
    (dict(d=64, T=2100, block=64, k_top=33), True),                                       # two nodes a lane, one more than one would hold
    (dict(T=4500, k_top=64, n_q_heads=7, n_kv_heads=1), False),                           # the most; N_k just above k; 4 + 3 heads or fewer
    (dict(d=64, T=9000, block=32, k_top=64, n_q_heads=2, n_kv_heads=1), True),            # four tiles a stage, lists of up to 128
    (dict(block=32, T=6001, k_top=9, n_q_heads=3, n_kv_heads=3, batch=2), True),          # query blocks as rows, their number no multiple
    (dict(d=64, block=64, T=40000, k_top=3, n_q_heads=4, n_kv_heads=2), True),            # two heads at two query blocks, many levels
    (dict(T=40001, k_top=32, n_q_heads=3, n_kv_heads=3, local=True), False),
    (dict(d=64, block=32, T=97, k_top=64), True),                                         # k beyond the number of blocks
])
def test_masks_on_tcgen05_beyond_four_heads_and_32_blocks(S, kw, causal):
    base = dict(name="w", seed=6, batch=1, n_q_heads=4, n_kv_heads=1, T=700, d=128, block=64, k_top=5, dtype="bf16")
    spec = wl.WorkloadSpec(**{**base, **kw})
    w = wl.generate(spec)
    rows = None if spec.n_rows <= 600 else np.unique(np.random.default_rng(1).choice(spec.n_rows, 500, replace=False))
    assert_mask_parity(S, w, rows, score_cache=False, causal=causal)


@pytest.mark.parametrize("kw", [dict(n_q_heads=8, n_kv_heads=8, batch=2, T=300),      # three kv heads to a chunk, across the batch; the last one alone
                                dict(n_q_heads=11, n_kv_heads=11, T=2001, dtype="f32", d=64, block=32)])
def test_run_host_with_several_kv_heads_to_a_chunk(S, kw):
    spec = wl.WorkloadSpec(**{**dict(name="w", seed=8, batch=1, T=700, d=128, block=64, k_top=5, dtype="bf16"), **kw})
    q, k, v = wl.generate(spec).torch_tensors("cpu")
    qh, kh, vh = (x.contiguous().pin_memory() for x in (q, k, v))
    mask = torch.empty(spec.batch, spec.n_q_heads, spec.n_blocks, spec.k_top, dtype=torch.int32, pin_memory=True)
    out = torch.empty_like(qh).pin_memory()
    blocks = dict(block_q=spec.block, block_k=spec.block)
    p = S.make_problem(qh, kh, k_top=spec.k_top, **blocks)
    staging = torch.empty(S.stream_host_staging_bytes(p), dtype=torch.uint8, device="cuda")
    S.run_host(qh, kh, vh, mask, out, staging, k_top=spec.k_top, **blocks)
    torch.cuda.synchronize()
    q, k, v = q.cuda(), k.cuda(), v.cuda()
    ref = S.build_mask(q, k, k_top=spec.k_top, **blocks).mask
    assert torch.equal(mask, ref.cpu())
    assert (out.float() - S.sparse_attention(q, k, v, ref, **blocks).float().cpu()).abs().max().item() <= TOL[spec.dtype]


@pytest.mark.parametrize("dtype,d,bq", [(torch.float32, 64, 64), (torch.bfloat16, 256, 64)])  # fp32 FMA, mma.sync
def test_threads_with_different_sizes_on_one_kernel(S, dtype, d, bq):
    """Threads with streams and outputs of their own launch the same kernels, some with rows of 2 blocks, some of 1024:
    no thread's launch may take from another the shared memory that it needs."""
    torch.manual_seed(3)
    q, k, v = (torch.randn(1, 80, 64, d, device="cuda", dtype=dtype) for _ in range(3))

    class Thread:
        def __init__(self, k_top):
            self.p = S.make_problem(q, k, block_q=bq, block_k=64, k_top=k_top)
            self.stream = torch.cuda.Stream()
            self.mask = torch.empty(1, 80, 64 // bq, k_top, dtype=torch.int32, device="cuda")
            self.out, self.ws = torch.empty_like(q), torch.empty(256, dtype=torch.uint8, device="cuda")
            self.vertical = torch.empty(1, 80, 1, device="cuda")

        def once(self):
            S.stream_build_mask(self.p, q, k, self.mask, None, self.ws, 256, self.stream)
            S.stream_sparse_attention(self.p, q, k, v, self.mask, 0.0, self.out, self.stream)
            S.stream_vertical_scores(self.p, self.mask, None, self.vertical, None, self.ws, 256, self.stream)

        def run(self, n=2000):
            for i in range(n):
                self.once()
                if i % 100 == 0:
                    self.stream.synchronize()

    threads = [Thread(k_top) for k_top in (2, 1024, 2, 1024)]
    torch.cuda.synchronize()
    for t in threads:
        t.once()
    torch.cuda.synchronize()
    want = [(t.mask.clone(), t.out.clone(), t.vertical.clone()) for t in threads]
    for t in threads:
        t.mask.fill_(-7), t.out.zero_(), t.vertical.zero_()
    torch.cuda.synchronize()
    with ThreadPoolExecutor(len(threads)) as pool:
        for done in [pool.submit(t.run) for t in threads]:
            done.result()
    torch.cuda.synchronize()
    for t, ref in zip(threads, want):
        assert all(torch.equal(a, b) for a, b in zip((t.mask, t.out, t.vertical), ref))


def test_a_list_of_k_beyond_32_bits_is_refused(S):
    q = torch.zeros(1, 1, 256, 64, device="cuda")
    for bad in ([2**32 + 4, 2], [2, 2**31]):
        with pytest.raises(OverflowError):
            S.build_masks(q, q, bad, block_q=32, block_k=32)


def test_a_mask_build_with_a_workspace_says_why_it_is_refused(S):
    q = torch.zeros(1, 1, 256, 64, device="cuda")
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    for kw, status in ((dict(k_top=2000), S.STREAM_ERR_UNSUPPORTED), (dict(k_top=2, block_k=65), S.STREAM_ERR_UNSUPPORTED),
                       (dict(k_top=0), S.STREAM_ERR_INVALID_ARG)):
        with pytest.raises(S.StreamError) as e:
            S.build_mask(q, q, workspace=ws, **{**dict(block_q=32, block_k=32), **kw})
        assert e.value.status == status
