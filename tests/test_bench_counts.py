"""What the benchmark line counts beside the library's own counters: tiles of rows that are kept whole, which nobody multiplies, and the
tiles that the attention copies."""
import numpy as np
import pytest
import torch

import bench
from helpers import oracle_problem
from oracle import stream_oracle as so
from paper_2510_19875_b200 import workloads as wl


@pytest.mark.parametrize("T,k,block_q", [(64, 1, 64), (1000, 15, 64), (1000, 16, 64), (1025, 16, 64), (4096, 32, 64), (9999, 16, 64), (1453, 17, 1), (1088, 17, 1), (300, 3, 1), (65, 1, 64)])
def test_tiles_of_rows_kept_whole(T, k, block_q):
    spec = wl.WorkloadSpec("w", 1, 2, 4, 2, T, 16, 64, k, "f32")
    tokens = [min((qb + 1) * block_q, T) - 1 for qb in range(-(-T // block_q))]
    allowed = [t // 64 + 1 for t in tokens]
    whole = [n <= k for n in allowed]
    if block_q == 1 and not all(whole):  # a group of 128 tokens has products as soon as one of them ranks
        whole = [all(whole[g - g % 128: g - g % 128 + 128]) for g in range(T)]
    want = 8 * sum(n for n, w in zip(allowed, whole) if w) if T > 64 else 0
    assert bench.tiles_kept_whole(spec, block_q if block_q == 1 else 0) == want
    if block_q == 64:  # what is left of the method's tiles is what a row that ranks scores
        w = wl.generate(spec, with_v=False)
        ora = so.build_mask_rows(oracle_problem(spec), w.q, w.k, None, score_cache=True)
        tiles = ora["tiles"].astype(np.int64)
        assert tiles.sum() - want == sum(int(x) for x, i in zip(tiles, range(len(tiles))) if not whole[i % len(whole)]) or T <= 64


@pytest.mark.parametrize("B,H,G,n_qb,k", [(1, 4, 2, 9, 5), (2, 3, 1, 7, 6), (1, 7, 1, 5, 70), (1, 2, 2, 4, 3)])
def test_tiles_the_attention_copies(B, H, G, n_qb, k):
    rng = np.random.default_rng(k)
    mask = np.full((B, H, n_qb, k), -1, np.int32)
    for row in mask.reshape(-1, k):
        n = int(rng.integers(0, k + 1))
        row[:n] = np.sort(rng.permutation(k + 2)[:n])
    want, hpg = 0, H // G
    for b in range(B):
        for g in range(G):
            rows = [mask[b, g * hpg + h, qb] for qb in range(n_qb) for h in range(hpg)][::-1]
            for i in range(0, len(rows), 2):
                pair = rows[i:i + 2] + [np.full(k, -1)] * (len(rows) - i == 1)
                for e in range(k):
                    if max(pair[0][e], pair[1][e]) >= 0:
                        want += 2 * (1 if pair[0][e] == pair[1][e] and e < 64 else 2)
    assert bench.attention_tiles_fetched(torch.from_numpy(mask), G) == want


@pytest.mark.gpu
@pytest.mark.parametrize("T,k,block_q", [(1000, 16, 64), (3000, 9, 64), (40, 2, 64), (1453, 17, 1), (900, 16, 1)])
def test_rows_kept_whole_have_no_products(T, k, block_q):
    from paper_2510_19875_b200 import stream as S

    spec = wl.WorkloadSpec("w", 1, 1, 4, 2, T, 128, 64, k, "bf16")
    q, key, _ = wl.generate(spec).torch_tensors("cuda")
    res = S.build_mask(q, key, block_q=block_q, block_k=64, k_top=k)
    torch.cuda.synchronize()
    st = res.stats()
    computed = st.tiles_scored - bench.tiles_kept_whole(spec, block_q if block_q == 1 else 0)
    assert st.error == 0 and st.rows == 4 * -(-T // block_q)
    if T <= 64 * k:
        assert computed == st.tile_products == st.tiles_fetched == 0
    elif block_q == 64:
        q_tiles = 4 * (st.rows // 4 - k)
        assert computed // 4 + q_tiles <= st.tiles_fetched <= computed + q_tiles
    else:
        assert 0 < computed / 64 <= st.tile_products
