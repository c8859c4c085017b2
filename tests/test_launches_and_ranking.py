"""Ranking with many equal scores in the tcgen05 mask kernel, a chain of launches that share buffers, and the fp32 attention
where its weights lie over the key tile, against the CPU oracle."""
import gc

import numpy as np
import pytest
import torch

from helpers import oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def leave_no_garbage():  # (what follows counts the allocator's bytes around a call: no collection may fall there)
    yield
    gc.collect()


@pytest.mark.parametrize("block,T,k_top", [(64, 4000, 32), (64, 4000, 31), (64, 3000, 1), (32, 3001, 8), (32, 5000, 17), (64, 9000, 16)])
def test_equal_scores_keep_the_first(S, block, T, k_top):
    """Queries and keys of 0 and 1 with few ones: scores are small whole numbers, exact whatever the order of the sums, and most
    rows have more candidates at the k-th score than places left. Every row has to be the oracle's, none is exempt."""
    spec = wl.WorkloadSpec("ties", 3, 1, 6, 2, T, 128, block, k_top, "bf16")
    w = wl.generate(spec)
    rng = np.random.default_rng(k_top)
    w.q = wl.to_bf16_bits((rng.random((1, 6, T, 128)) < 0.05).astype(np.float32))
    w.k = wl.to_bf16_bits((rng.random((1, 2, T, 128)) < 0.05).astype(np.float32))
    q, k, _ = w.torch_tensors("cuda")
    res = S.build_mask(q, k, block_q=block, block_k=block, k_top=k_top, want_scores=True)
    p = oracle_problem(spec)
    n_rows = 6 * so.num_query_blocks(p)
    rows = np.unique(np.random.default_rng(1).choice(n_rows, min(n_rows, 400), replace=False))
    ora = so.build_mask_rows(p, w.q, w.k, rows, want_scores=True)
    assert res.stats().error == 0
    assert np.array_equal(res.mask.cpu().numpy().reshape(-1, k_top)[rows], ora["mask"])
    assert np.array_equal(res.scores.cpu().numpy().reshape(-1, k_top)[rows], ora["scores"])


@pytest.mark.parametrize("dtype,d,block_q,block_k", [(torch.bfloat16, 128, 64, 64), (torch.bfloat16, 64, 32, 32), (torch.float32, 64, 32, 32),
                                                     (torch.bfloat16, 256, 64, 64), (torch.bfloat16, 128, 1, 64)])
def test_launches_that_share_buffers_wait_for_each_other(S, dtype, d, block_q, block_k):
    """Two inputs in turn through one mask, one output and one workspace, without a synchronisation in between. The attention begins
    while the mask build still runs and has to see its result; copies and memsets stand between all others (chains of
    kernels alone: test_dependent_launches.py)."""
    torch.manual_seed(d)
    kw = dict(block_q=block_q, block_k=block_k)
    inputs = [tuple(torch.randn(1, h, 1100, d, device="cuda").to(dtype) for h in (8, 2, 2)) for _ in range(2)]
    want = []
    for q, k, v in inputs:
        m = S.build_mask(q, k, k_top=4, **kw).mask
        torch.cuda.synchronize()
        want.append((m, S.sparse_attention(q, k, v, m, **kw)))
        torch.cuda.synchronize()
    q, k, v = (x.clone() for x in inputs[0])
    mask, out, ws = want[0][0].clone(), torch.empty_like(q), torch.empty(256, dtype=torch.uint8, device="cuda")
    got = []
    for i in range(60):
        for dst, src in zip((q, k, v), inputs[i % 2]):
            dst.copy_(src)
        S.build_mask(q, k, k_top=4, mask_out=mask, workspace=ws, **kw)
        S.sparse_attention(q, k, v, mask, out=out, **kw)
        got.append((mask.clone(), out.clone()))
        S.sparse_attention(q, k, v, mask, out=out, **kw)  # (behind the copies: what it writes again, the next round's kernels find)
    torch.cuda.synchronize()
    for i, pair in enumerate(got):
        assert all(torch.equal(a, b) for a, b in zip(pair, want[i % 2])), i


@pytest.mark.parametrize("heads,T,d,block_q,block_k,k", [(8, 1500, 64, 32, 32, 1), (8, 1503, 64, 32, 32, 9), (12, 1001, 64, 16, 16, 5),
                                                        (12, 1001, 64, 24, 48, 3), (8, 1481, 64, 32, 64, 4), (8, 1500, 32, 32, 32, 7)])
def test_fp32_attention_with_rows_for_three_ctas_an_sm(S, heads, T, d, block_q, block_k, k):
    """More rows than two and a half an SM: a warp's weights lie over its key tile, fetched anew behind the second product. Holes,
    empty rows, a block twice. fp32: the products' and sums' rounding."""
    spec = wl.WorkloadSpec("w", 7, 1, heads, 2, T, d, block_k, k, "f32")
    w = wl.generate(spec)
    q, k_, v = w.torch_tensors("cuda")
    p = oracle_problem(spec, block_q=block_q, block_k=block_k)
    n_rows = heads * so.num_query_blocks(p)
    assert 2 * n_rows > 5 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(3)
    mask = rng.integers(0, -(-T // block_k), size=(n_rows, k)).astype(np.int32)
    mask[rng.random(mask.shape) < 0.2] = -1
    mask[rng.random(n_rows) < 0.1] = -1
    out = S.sparse_attention(q, k_, v, torch.from_numpy(mask.reshape(1, heads, -1, k)).cuda(), block_q=block_q, block_k=block_k)
    out = out.cpu().numpy().reshape(-1, T, d)
    rows = np.unique(rng.choice(n_rows, 300, replace=False))
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask[rows], rows)
    nqb = so.num_query_blocks(p)
    for i, rid in enumerate(rows):
        bh, qb = divmod(int(rid), nqb)
        lo, hi = qb * block_q, min(T, qb * block_q + block_q)
        assert np.abs(out[bh, lo:hi] - ref[i, : hi - lo]).max() <= 1e-4, rid
