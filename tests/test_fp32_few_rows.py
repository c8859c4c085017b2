"""The fp32-FMA attention with fewer rows than half of the SMs, on both sides of the line between a row over a cluster and a row in one CTA:
eight tiles of 32 queries, keys and 64 channels. Against the CPU oracle."""
import numpy as np
import pytest
import torch

from helpers import oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)
from test_gpu_warp_kernels import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d,block_q,block_k,k_top", [
    (64, 64, 64, 2), (64, 64, 64, 3), (64, 64, 64, 4), (32, 64, 64, 4), (16, 64, 64, 3), (16, 64, 64, 2), (64, 33, 32, 4), (64, 33, 32, 5),
    (64, 32, 32, 8), (64, 32, 32, 9), (32, 16, 16, 8), (32, 16, 16, 9), (64, 16, 64, 4), (64, 16, 64, 5), (64, 48, 24, 700)])
@pytest.mark.parametrize("heads,n_qb", [(1, 1), (1, 10), (2, 20), (2, 36)])
def test_few_rows_against_the_oracle(S, heads, n_qb, d, block_q, block_k, k_top, dtype):
    T = max(1, n_qb * block_q - 3)
    spec = wl.WorkloadSpec("w", 7, 1, heads, 1, T, d, block_k, k_top, dtype)
    w = wl.generate(spec)
    q, k, v = w.torch_tensors("cuda")
    p = oracle_problem(spec, block_q=block_q, block_k=block_k)
    rng = np.random.default_rng(n_qb)
    mask = rng.integers(0, -(-T // block_k), size=(heads * n_qb, k_top)).astype(np.int32)
    mask[rng.random(mask.shape) < max(0.1, 1 - 12 / k_top)] = -1
    out = S.sparse_attention(q, k, v, torch.from_numpy(mask.reshape(1, heads, n_qb, k_top)).cuda(), block_q=block_q, block_k=block_k, impl="generic")
    out = out.float().cpu().numpy().reshape(-1, T, d)
    rows = np.arange(heads * n_qb)
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask, rows)
    for i, rid in enumerate(rows):
        bh, qb = divmod(int(rid), n_qb)
        lo, hi = qb * block_q, min(T, qb * block_q + block_q)
        assert np.abs(out[bh, lo:hi] - ref[i, : hi - lo]).max() <= TOL[dtype], rid
