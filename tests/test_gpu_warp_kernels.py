"""The warp-level kernels (mma.sync and fp32 FMA) against the CPU oracle, at the sizes where their tiles,
remainders and launch shapes change: masks bit for bit outside near-ties, attention within
tolerance, also on arbitrary masks (holes, empty rows, a block twice in a row)."""
import numpy as np
import pytest
import torch

from helpers import compare_masks, oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)

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
    (dict(dtype="f32", T=1003, n_q_heads=8), None, None, True),
    (dict(dtype="f32", T=515, d=128, k_top=40, block=16), None, None, True),
    (dict(dtype="f32", T=300, d=256, block=64, k_top=3), None, None, False),
    (dict(dtype="f32", T=300, d=16, k_top=3), 1, 24, True),
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
