"""The tcgen05 mask kernels where an SM holds two CTAs, where groups have four, two or one rows, and where the last heads that are walked
together are fewer than the ones before: launches repeated with several groups a CTA, and masks against the oracle and against builds of one head."""
import numpy as np
import pytest
import torch

from helpers import TIE_GAP, check_mask_invariants, oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def workload(H, G, T, d=128, block=64, k=8, seed=9):
    return wl.generate(wl.WorkloadSpec("t", seed, 1, H, G, T, d, block, k, "bf16", local=True), with_v=False)


def against_oracle(w, mask, causal, n, **kw):
    """Rows of one mask [H, n_qb, k] against the oracle, n of them and the last of every head."""
    H, n_qb, k = mask.shape
    rows = np.unique(np.concatenate([np.random.default_rng(1).choice(H * n_qb, min(n, H * n_qb), replace=False), np.arange(1, H + 1) * n_qb - 1]))
    ora = so.build_mask_rows(oracle_problem(w.spec, causal=causal, **kw), w.q, w.k, rows, score_cache=True)
    clear = ora["min_gap"] >= TIE_GAP
    assert (mask.reshape(-1, k)[rows][clear] == ora["mask"][clear]).all()


# Rows an SM enough for several groups a CTA, without scores, so that rows kept whole are written beside the last ones: two CTAs of two
# rows (d = 128, blocks of 64, k up to 8), two of four rows, one CTA; one query head per kv head (rows of several query blocks), three, seven
@pytest.mark.parametrize("H,G,T,d,block,k,causal", [
    (8, 8, 30000, 128, 64, 8, True), (14, 2, 16800, 128, 64, 8, True), (6, 2, 9000, 128, 64, 5, False),
    (8, 8, 25000, 64, 64, 16, True), (14, 2, 20000, 64, 64, 20, True), (6, 2, 14000, 64, 64, 40, False), (8, 8, 9000, 64, 64, 50, True),
    (8, 8, 13000, 128, 32, 8, True), (14, 2, 10000, 128, 32, 16, True), (8, 8, 14000, 64, 32, 40, False), (14, 2, 9000, 64, 32, 9, True),
    (14, 2, 4000, 128, 32, 40, True), (12, 2, 12000, 128, 32, 40, False), (3, 3, 60000, 128, 64, 12, True), (14, 2, 20000, 128, 64, 40, True)])
def test_repeated_launches_without_scores(S, H, G, T, d, block, k, causal):
    w = workload(H, G, T, d, block, k)
    q, key = (x.cuda() for x in w.torch_tensors("cpu")[:2])
    kw = dict(block_q=block, block_k=block, k_top=k, causal=causal)
    first = S.build_mask(q, key, **kw)
    torch.cuda.synchronize()
    st = first.stats()
    assert st.error == 0 and st.rows == first.mask[..., 0].numel()
    for it in range(20):
        res = S.build_mask(q, key, **kw)
        torch.cuda.synchronize()
        assert res.stats().error == 0 and res.stats().tiles_scored == st.tiles_scored, it
        assert torch.equal(res.mask, first.mask), it
    mask = first.mask.cpu().numpy()
    check_mask_invariants(mask, w.spec, causal=causal)
    against_oracle(w, mask[0], causal, 60)


# Two heads' keys of 11 MB are walked together and the third alone; at 5000 tokens all are
@pytest.mark.parametrize("H,G,T", [(3, 3, 44000), (6, 3, 44000), (12, 3, 44100), (3, 3, 5000), (21, 3, 5000)])
def test_heads_walked_together_and_a_rest(S, H, G, T):
    w = workload(H, G, T, k=9)
    q, key = (x.cuda() for x in w.torch_tensors("cpu")[:2])
    kw, ks, hpg = dict(block_q=64, block_k=64), [9, 3, 5], H // G
    mask = S.build_mask(q, key, k_top=9, **kw).mask
    many = S.build_masks(q, key, ks, **kw).mask
    for g in range(G):
        heads = slice(g * hpg, (g + 1) * hpg)
        one_q, one_k = q[:, heads].contiguous(), key[:, g:g + 1].contiguous()
        assert torch.equal(mask[:, heads], S.build_mask(one_q, one_k, k_top=9, **kw).mask)
        assert torch.equal(many[:, :, heads], S.build_masks(one_q, one_k, ks, **kw).mask)
    for i, k in enumerate(ks):
        assert torch.equal(many[i, ..., :k], S.build_mask(q, key, k_top=k, **kw).mask) and bool((many[i, ..., k:] == -1).all())
    against_oracle(w, mask[0].cpu().numpy(), True, 40)


@pytest.mark.parametrize("H,G,T", [(3, 3, 44000), (4, 2, 1453), (12, 2, 1000), (6, 2, 5000)])
def test_tokens_of_heads_walked_together_and_a_rest(S, H, G, T):
    """Rows kept whole are written by CTAs without a group, or by all behind their last."""
    w = workload(H, G, T, k=17)
    q, key = (x.cuda() for x in w.torch_tensors("cpu")[:2])
    kw, hpg = dict(block_q=1, block_k=64, k_top=17, impl="tensor"), H // G
    res = S.build_mask(q, key, **kw)
    torch.cuda.synchronize()
    assert res.stats().error == 0 and res.stats().rows == H * T
    for g in range(G):
        heads = slice(g * hpg, (g + 1) * hpg)
        assert torch.equal(res.mask[:, heads], S.build_mask(q[:, heads].contiguous(), key[:, g:g + 1].contiguous(), **kw).mask)
    against_oracle(w, res.mask[0].cpu().numpy(), True, 60, block_q=1, block_k=64)


# A ragged end, and k whose first ranking levels differ: levels are passed over in one pass of a group and not in the next
@pytest.mark.parametrize("causal", [True, False])
@pytest.mark.parametrize("T,H,G,ks", [(2047, 4, 1, [32, 8, 3]), (2100, 3, 3, [31, 16, 15]), (2100, 7, 1, [5, 32]), (4100, 6, 2, [7, 14, 28]), (9001, 2, 2, [32, 1, 17]),
                                      (10311, 8, 2, [5, 10, 21]), (65, 4, 2, [1, 2]), (1000, 5, 1, [16, 15, 8])])
def test_several_k_are_the_builds_of_one(S, T, H, G, ks, causal):
    w = workload(H, G, T, k=max(ks))
    q, key = (x.cuda() for x in w.torch_tensors("cpu")[:2])
    kw = dict(block_q=64, block_k=64, causal=causal, want_scores=True)
    many = S.build_masks(q, key, ks, **kw)
    torch.cuda.synchronize()
    assert many.stats().error == 0
    for i, k in enumerate(ks):
        one = S.build_mask(q, key, k_top=k, **kw)
        assert torch.equal(many.mask[i, ..., :k], one.mask) and bool((many.mask[i, ..., k:] == -1).all())
        assert torch.equal(many.scores[i, ..., :k], one.scores)
    against_oracle(w, many.mask[0, 0].cpu().numpy()[..., :ks[0]], causal, 60, k_top=ks[0])
