"""tcgen05 attention where two rows of a unit name the same key blocks: one fetch serves both. Ascending rows that share some,
all or none of their blocks, of unequal length, empty, and rows that are not ascending (which share nothing), against the oracle."""
import numpy as np
import pytest
import torch

from helpers import oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def rows(rng, n_rows, n_blocks, k, common, kind):
    """Rows of up to k blocks, most of each out of `common` * k blocks that all rows have in common."""
    base = rng.permutation(n_blocks)[: int(round(common * k))]
    mask = np.full((n_rows, k), -1, np.int32)
    for m in mask:
        n = 0 if rng.random() < 0.05 else int(rng.integers(max(1, k - 3), k + 1)) if rng.random() < 0.7 else int(rng.integers(1, k + 1))
        rest = rng.permutation(np.setdiff1d(np.arange(n_blocks), base))
        blocks = np.concatenate([base, rest])[:n]
        m[: len(blocks)] = np.sort(blocks) if kind == "ascending" or rng.random() < 0.5 else rng.permutation(blocks)
        if kind == "any":
            m[rng.random(k) < 0.2] = -1                 # holes
            if rng.random() < 0.3:
                m[rng.integers(0, k)] = m[0]            # a block twice
    return mask


@pytest.mark.parametrize("kind", ["ascending", "any"])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("H,G,T,k,common,causal", [(2, 1, 3000, 1, 1.0, True), (2, 1, 3000, 2, 0.5, True), (4, 2, 2000, 5, 0.6, False), (7, 1, 2001, 16, 1.0, True),
                                                   (7, 1, 1300, 16, 0.0, False), (2, 2, 4130, 31, 0.5, True), (4, 1, 4096, 32, 0.8, False), (3, 1, 4500, 33, 0.5, False),
                                                   (2, 1, 6000, 63, 0.9, True), (2, 1, 6000, 64, 0.4, False), (2, 1, 6000, 65, 0.5, False), (1, 1, 64, 1, 1.0, True)])
def test_rows_that_share_blocks(S, kind, d, H, G, T, k, common, causal):
    """bf16: the rounding of the output and, at d = 128, of the weights (2e-2 as everywhere)."""
    spec = wl.WorkloadSpec("w", 8, 1, H, G, T, d, 64, k, "bf16")
    w = wl.generate(spec)
    q, k_, v = w.torch_tensors("cuda")
    p = oracle_problem(spec, causal=causal)
    n_qb = so.num_query_blocks(p)
    mask = rows(np.random.default_rng(k), H * n_qb, n_qb, k, common, kind)
    out = S.sparse_attention(q, k_, v, torch.from_numpy(mask.reshape(1, H, n_qb, k)).cuda(), block_q=64, block_k=64, causal=causal)
    out = out.float().cpu().numpy().reshape(H, T, d)
    some = np.unique(np.random.default_rng(1).choice(H * n_qb, min(H * n_qb, 120), replace=False))
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask[some], some)
    for i, row in enumerate(some):
        h, qb = divmod(int(row), n_qb)
        lo, hi = qb * 64, min(T, qb * 64 + 64)
        assert np.abs(out[h, lo:hi] - ref[i, : hi - lo]).max() <= 2e-2, row
    assert S.stream_check_device_status() is None
