"""What the batch autotuner reports and compares is the whole batch, its
buckets side by side, and not the sum of the buckets alone."""
import numpy as np
import pytest

from paper_1804_09002_gb300 import inputs as I
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_tune_ms_is_the_time_of_a_run():
    """Sixteen buckets of one instance on eight streams: the reported time is
    that of the captured batch, and the same sizes as sixteen plans of one
    bucket add up to more (two buckets of similar size share a stream, so half
    the sum is what the largest pairs alone can take; 0.75 lies between)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding as B
    sizes = list(range(16, 257, 16))
    data = [I.haar_csd(n, seed=n) for n in sizes]
    ctx = B.Context(0)
    try:
        plan = B.Batch(ctx, sizes)
        plan.load([to_dev(d[0]) for d in data], [to_dev(d[1]) for d in data])
        assert np.all(plan.run() == 0)
        tuned = plan.stats()["tune_ms"][16]
        plan.close()
        alone = 0.0
        for n, d in zip(sizes, data):
            one = B.Batch(ctx, [n])
            one.load([to_dev(d[0])], [to_dev(d[1])])
            one.run()
            alone += min(one.stats()["tune_ms"].values())
            one.close()
        assert tuned <= 0.75 * alone, (tuned, alone)
    finally:
        ctx.close()
