"""The fp32-FMA attention on both sides of the lines between its builds (by rows an SM), with every way of loading keys and values,
against the CPU oracle."""
import gc

import numpy as np
import pytest
import torch

from helpers import oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl
from test_gpu_parity import S  # noqa: F401  (fixture)
from test_gpu_warp_kernels import TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def leave_no_garbage():  # (what follows counts the allocator's bytes around a call: no collection may fall there)
    yield
    gc.collect()


def off_boundary(x):
    """The same values in rows that begin on no 8-byte boundary."""
    y = torch.empty(*x.shape[:-1], x.shape[-1] + 1, dtype=x.dtype, device=x.device)[..., :x.shape[-1]]
    return y.copy_(x)


# d, block_q, block_k, k_top, rows an SM between
BUILDS = [
    (64, 32, 32, 9, 2.5, 3), (64, 16, 16, 5, 2.5, 3), (64, 24, 48, 3, 2.5, 3),        # three CTAs, P over the key tile
    (64, 32, 32, 4, 3, 4.25), (64, 16, 32, 6, 4.25, 6), (64, 32, 64, 5, 4.25, 6),     # two; three again
    (64, 32, 32, 700, 2.5, 3),                                                        # a list too long for a third CTA
    (64, 32, 32, 2, 4.25, 6),                                                         # two warps a CTA
    (32, 32, 32, 7, 2, 2.5), (32, 32, 32, 7, 2.5, 3), (32, 17, 32, 5, 3, 4.25), (32, 32, 16, 9, 6, 7),
    (32, 64, 32, 4, 2.5, 3), (32, 64, 64, 5, 3, 4.25), (32, 48, 32, 3, 4.25, 6), (32, 33, 64, 4, 6, 7),  # two warps a group: up to four
]


@pytest.mark.parametrize("off", [False, True])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d,block_q,block_k,k_top,low,high", BUILDS)
def test_builds_by_rows_against_the_oracle(S, d, block_q, block_k, k_top, low, high, dtype, off):
    heads, n_sm = 8, torch.cuda.get_device_properties(0).multi_processor_count
    n_qb = int((low + high) / 2 * n_sm / heads)
    T = n_qb * block_q - 3
    assert low * n_sm < heads * n_qb <= high * n_sm
    spec = wl.WorkloadSpec("w", 5, 1, heads, 2, T, d, block_k, k_top, dtype)
    w = wl.generate(spec)
    q, k, v = w.torch_tensors("cuda")
    if off:
        q, k, v = off_boundary(q), off_boundary(k), off_boundary(v)
    p = oracle_problem(spec, block_q=block_q, block_k=block_k)
    n_rows = heads * n_qb
    # holes, empty rows, a block twice; a row of 700 places has entries in a few of them only
    rng = np.random.default_rng(k_top)
    mask = rng.integers(0, -(-T // block_k), size=(n_rows, k_top)).astype(np.int32)
    mask[rng.random(mask.shape) < max(0.2, 1 - 12 / k_top)] = -1
    mask[rng.random(n_rows) < 0.1] = -1
    out = S.sparse_attention(q, k, v, torch.from_numpy(mask.reshape(1, heads, -1, k_top)).cuda(), block_q=block_q, block_k=block_k, impl="generic")
    out = out.float().cpu().numpy().reshape(-1, T, d)
    rows = np.unique(rng.choice(n_rows, 120, replace=False))
    ref = so.sparse_attention_rows(p, w.q, w.k, w.v, mask[rows], rows)
    for i, rid in enumerate(rows):
        bh, qb = divmod(int(rid), n_qb)
        lo, hi = qb * block_q, min(T, qb * block_q + block_q)
        assert np.abs(out[bh, lo:hi] - ref[i, : hi - lo]).max() <= TOL[dtype], rid
