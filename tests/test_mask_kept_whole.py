"""Mask levels that cannot drop anything, because no more candidates are allowed than k: their scores are not waited for, and a row
that keeps all its allowed blocks has none computed unless they are asked for. Masks and tile counts are the oracle's."""
import numpy as np
import pytest
import torch

from helpers import check_mask_invariants, compare_masks, oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S, run_mask  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# k around the number of key blocks and around halves and quarters of it, where a level begins to rank; one to seven heads per kv head
# (rows of several query blocks in a group), ragged lengths, both block sizes and head dimensions
CASES = [dict(T=T, k_top=k, n_q_heads=H, n_kv_heads=G, d=d, block=blk, causal=causal)
         for T, k, H, G, d, blk, causal in [
             (1000, 15, 4, 1, 128, 64, True), (1000, 16, 4, 1, 128, 64, True), (1000, 16, 2, 2, 128, 64, False), (1025, 16, 7, 1, 128, 64, True),
             (2100, 31, 3, 3, 64, 64, True), (2100, 33, 8, 2, 64, 64, True), (2100, 34, 2, 2, 64, 64, False), (64 * 33, 32, 4, 1, 128, 64, True),
             (1000, 31, 6, 2, 128, 32, True), (1000, 40, 6, 2, 128, 32, True), (3001, 23, 1, 1, 64, 32, True), (70, 1, 4, 2, 128, 64, True),
             (6000, 7, 14, 2, 128, 64, True), (9000, 64, 4, 2, 128, 64, True), (9000, 9, 3, 3, 128, 64, True), (60, 3, 4, 2, 128, 64, True)]]


def check(S, kw, impl="auto", dtype="bf16", **blocks):
    kw = dict(kw)
    causal = kw.pop("causal")
    w = wl.generate(wl.WorkloadSpec(name="t", seed=6, batch=2, dtype=dtype, **kw))
    res = run_mask(S, w, impl=impl, causal=causal, **blocks)
    mask = res.mask.cpu().numpy()
    check_mask_invariants(mask, w.spec, causal=causal, **blocks)
    ora = so.build_mask_rows(oracle_problem(w.spec, causal=causal, **blocks), w.q, w.k, None, score_cache=True)
    flat = mask.reshape(-1, kw["k_top"])
    assert compare_masks(flat, ora)["bad"] == 0
    st, tiles = res.stats(), res.row_tiles().cpu().numpy().reshape(-1).astype(np.int64)
    assert st.error == 0 and st.rows == flat.shape[0] and st.tiles_scored == int(tiles.sum())
    clear = (flat == ora["mask"]).all(axis=1) & (ora["min_gap"] >= 1e-5)
    assert (tiles[clear] == ora["tiles"][clear]).all()


@pytest.mark.parametrize("kw", CASES, ids=str)
def test_masks_without_scores(S, kw):
    check(S, kw)


# A row per token, 128 tokens a group: some groups, half of one, all of them kept whole; up to 16 nodes and more
@pytest.mark.parametrize("T,k,H,G,causal", [(2100, 16, 2, 1, True), (2100, 17, 2, 1, True), (1500, 5, 2, 2, True), (1500, 23, 1, 1, True), (1500, 23, 1, 1, False),
                                            (1500, 24, 1, 1, True), (3000, 11, 2, 1, True), (4200, 32, 1, 1, True), (4200, 1, 1, 1, True), (130, 1, 2, 1, True), (2000, 9, 1, 1, False)])
def test_masks_of_tokens_without_scores(S, T, k, H, G, causal):
    check(S, dict(T=T, k_top=k, n_q_heads=H, n_kv_heads=G, d=128, block=64, causal=causal), impl="tensor", block_q=1, block_k=64)


# The kernels of all other shapes: fp32 and mma.sync, a row over a cluster, sixteen warps, four; one key block; block_q != block_k
@pytest.mark.parametrize("T,k,H,G,d,bq,bk,dtype,causal", [
    (900, 7, 1, 1, 64, 32, 32, "f32", True), (2048, 8, 1, 1, 64, 32, 32, "f32", True), (1500, 12, 2, 1, 32, 32, 32, "f32", True), (3000, 9, 4, 2, 64, 32, 32, "f32", True),
    (3000, 24, 4, 1, 128, 16, 16, "f32", True), (1000, 40, 2, 2, 128, 16, 32, "f32", False), (1000, 20, 3, 1, 64, 24, 48, "f32", True), (500, 6, 2, 1, 64, 64, 16, "f32", True),
    (30, 3, 2, 1, 64, 32, 32, "f32", True), (2500, 11, 4, 2, 256, 64, 64, "bf16", True), (2500, 70, 4, 2, 128, 16, 16, "bf16", True), (2500, 160, 4, 2, 128, 16, 16, "bf16", True),
    (5000, 50, 8, 2, 256, 64, 64, "bf16", True), (3000, 24, 16, 4, 64, 32, 32, "f32", True)])
def test_masks_of_other_shapes_without_scores(S, T, k, H, G, d, bq, bk, dtype, causal):
    check(S, dict(T=T, k_top=k, n_q_heads=H, n_kv_heads=G, d=d, block=bk, causal=causal), dtype=dtype, block_q=bq, block_k=bk)


@pytest.mark.parametrize("causal", [True, False])
def test_rows_kept_whole_do_not_depend_on_the_numbers(S, causal):
    """Queries and keys of infinities and NaN: a row that keeps all it may keeps them whatever their scores."""
    q = torch.randn(1, 4, 1500, 128, device="cuda").bfloat16()
    k = torch.randn(1, 1, 1500, 128, device="cuda").bfloat16()
    q[:, 1], q[:, 2], k[..., 700, :], k[..., 900:, :] = float("nan"), float("inf"), float("nan"), -float("inf")
    for k_top in (10, 24, 40):
        kw = dict(block_q=64, block_k=64, k_top=k_top, causal=causal)
        masks = [S.build_mask(q, k, want_scores=scores, **kw).mask[0].cpu() for scores in (True, False)]
        rows = torch.arange(24) if causal else torch.full((24,), 23)
        want = torch.arange(k_top).expand(24, -1).clone()
        want[want > rows[:, None]] = -1
        whole = rows < k_top
        for m in masks:
            assert (m[:, whole] == want[whole]).all()
