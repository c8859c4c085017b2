"""Threads that launch the row kernels of the mask build with rows of very different shared memory: no thread's launch may take from
another what it needs. Scores are asked for, or rows rank, so that the row kernels run and not the one that writes rows kept whole."""
from concurrent.futures import ThreadPoolExecutor

import pytest
import torch

from test_gpu_parity import S  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scores", [True, False])
@pytest.mark.parametrize("dtype,d,bq", [(torch.float32, 64, 64), (torch.bfloat16, 256, 64)])  # fp32 FMA, mma.sync
def test_threads_with_different_sizes_on_one_mask_kernel(S, dtype, d, bq, scores):
    torch.manual_seed(4)
    # Without scores: 75 key blocks, more than 2 and than 70. 70 blocks a row take 30 times the list and slots of 2.
    T, H, small, large = (64, 80, 2, 1024) if scores else (75 * 64, 2, 2, 70)
    q, k = (torch.randn(1, H, T, d, device="cuda", dtype=dtype) for _ in range(2))

    class Thread:
        def __init__(self, k_top):
            self.p = S.make_problem(q, k, block_q=bq, block_k=64, k_top=k_top, causal=False)
            self.stream = torch.cuda.Stream()
            self.mask = torch.empty(1, H, T // bq, k_top, dtype=torch.int32, device="cuda")
            self.scores = torch.empty(self.mask.shape, device="cuda") if scores else None
            self.ws = torch.empty(256, dtype=torch.uint8, device="cuda")

        def once(self):
            S.stream_build_mask(self.p, q, k, self.mask, self.scores, self.ws, 256, self.stream)

        def run(self, n=1000 if scores else 200):
            for i in range(n):
                self.once()
                if i % 100 == 0:
                    self.stream.synchronize()

    threads = [Thread(k_top) for k_top in (small, large, small, large)]
    torch.cuda.synchronize()
    for t in threads:
        t.once()
    torch.cuda.synchronize()
    want = [[x.clone() for x in (t.mask, t.scores) if x is not None] for t in threads]
    for t in threads:
        t.mask.fill_(-7)
        if scores:
            t.scores.zero_()
    torch.cuda.synchronize()
    with ThreadPoolExecutor(len(threads)) as pool:
        for done in [pool.submit(t.run) for t in threads]:
            done.result()
    torch.cuda.synchronize()
    for t, ref in zip(threads, want):
        assert all(torch.equal(a, b) for a, b in zip([x for x in (t.mask, t.scores) if x is not None], ref))
