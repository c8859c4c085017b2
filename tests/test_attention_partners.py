"""The tcgen05 attention takes two mask rows through a unit side by side. A row's output is its own: bit for bit the same whatever the row
beside it holds, alone or in a layer, and so however a call groups the query heads."""
import pytest
import torch

from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def ascending(gen, rows, k, out_of):
    """Rows of k or fewer ascending blocks, drawn from the list `out_of`; -1 behind them."""
    mask = torch.full((rows, k), -1, dtype=torch.int32)
    for m in mask:
        n = int(torch.randint(max(1, k - 4), k + 1, (1,), generator=gen))
        blocks = out_of[torch.randperm(len(out_of), generator=gen)[:n]].sort().values
        m[: len(blocks)] = blocks
    return mask


@pytest.mark.parametrize("T,k,causal", [(900, 5, True), (2000, 16, True), (4096, 32, False), (3001, 40, True), (5000, 64, False), (5000, 70, False)])
def test_a_head_does_not_depend_on_the_one_beside_it(S, T, k, causal):
    gen = torch.Generator().manual_seed(T)
    q, key, v = (torch.randn(1, h, T, 128, generator=gen).bfloat16().cuda() for h in (2, 1, 1))
    n = -(-T // 64)
    every = torch.arange(n, dtype=torch.int32)
    first = ascending(gen, n, k, every)
    if causal:  # what a mask build leaves: nothing behind the query block
        for qb, m in enumerate(first):
            m[m > qb] = -1
    kw = dict(block_q=64, block_k=64, causal=causal)
    alone = S.sparse_attention(q[:, :1].contiguous(), key, v, first.view(1, 1, n, k).cuda(), **kw)
    beside = [first.clone(), torch.full_like(first, -1), ascending(gen, n, k, every), ascending(gen, n, k, every[::2]), first.clone()]
    beside[-1][:, k // 2:] = -1  # the same blocks, but fewer
    for other in beside:
        pair = torch.stack([first, other]).view(1, 2, n, k).cuda()
        assert torch.equal(S.sparse_attention(q, key, v, pair, **kw)[:, :1], alone)
    assert S.stream_check_device_status() is None


@pytest.mark.parametrize("H,G", [(14, 2), (6, 1), (5, 1)])
def test_the_host_path_gives_the_bits_of_the_device_calls_however_it_splits_a_head(S, H, G):
    """The query heads of the last kv head go through in two halves, which are other pairs than in one device call."""
    gen = torch.Generator().manual_seed(H)
    T, kw = 3000, dict(block_q=64, block_k=64, k_top=16)
    qh, kh, vh = (torch.randn(1, h, T, 128, generator=gen).bfloat16().pin_memory() for h in (H, G, G))
    assert (H // G + 2) * T * 128 * 2 >= 3 << 20  # (below this size a head stays whole)
    q, k, v = qh.cuda(), kh.cuda(), vh.cuda()
    ref = S.build_mask(q, k, **kw)
    want = S.sparse_attention(q, k, v, ref.mask, block_q=64, block_k=64)
    p = S.make_problem(qh, kh, **kw)
    staging = torch.empty(S.stream_host_staging_bytes(p), dtype=torch.uint8, device="cuda")
    mask, out = torch.empty(ref.mask.shape, dtype=torch.int32).pin_memory(), torch.empty(want.shape, dtype=want.dtype).pin_memory()
    S.run_host(qh, kh, vh, mask, out, staging, **kw)
    torch.cuda.synchronize()
    assert torch.equal(mask, ref.mask.cpu())
    assert torch.equal(out, want.cpu())
