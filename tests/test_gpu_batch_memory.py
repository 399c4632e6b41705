"""A batch plan leaves most of the free device memory to the caller: the
workspaces of its streams together take at most a quarter of what is free when
the plan lays out its buckets."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _haar_pair(n, g):
    X = torch.randn(2 * n, n, dtype=torch.float64, device="cuda:0", generator=g)
    Q = torch.linalg.qr(X)[0]
    return Q[:n].t().contiguous().t(), Q[n:].t().contiguous().t()


def test_workspace_is_a_fraction_of_the_free_memory():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding as B
    g = torch.Generator(device="cuda:0").manual_seed(3)
    sizes = [n for n in range(576, 1025, 64) for _ in range(3)]  # eight buckets of 2 to 7 GiB
    data = [_haar_pair(n, g) for n in sizes]
    ctx = B.Context(0)
    hold = None
    try:
        plan = B.Batch(ctx, sizes)
        plan.load([a for a, _ in data], [b for _, b in data])
        torch.cuda.synchronize()
        hold = torch.empty(3 * (torch.cuda.mem_get_info()[0] // 4), dtype=torch.uint8, device="cuda:0")
        free = torch.cuda.mem_get_info()[0]
        status = plan.run()
        used = free - torch.cuda.mem_get_info()[0]
        assert np.all(status == 0)
        assert used <= free // 4 + (2 << 30), (used >> 20, free >> 20)
        plan.close()
    finally:
        del hold
        torch.cuda.empty_cache()
        ctx.close()
