"""A batch whose angles are graded over many orders of magnitude: its leaves need
several passes of the leaf eigensolver, which a captured batch runs from
conditional nodes of its graph."""
import numpy as np
import pytest

from paper_1804_09002_gb300 import inputs as I
from tests.gpu_util import U, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _replay_ms(plan):
    best = np.inf
    for _ in range(4):
        e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        e0.record()
        status = plan.run()
        e1.record()
        e1.synchronize()
        assert np.all(status == 0)
        best = min(best, e0.elapsed_time(e1))
    return best


@pytest.mark.parametrize("sizes", [[40], [250], [30, 97, 250, 260, 400]])
def test_small_angles(sizes):
    """The bars for every instance, the same bits from every replay, also with
    other data in the same buffers in between, and the time: at most eight
    passes where separated angles take one, so eight times their time bounds it."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding as B
    rng = np.random.default_rng(len(sizes))
    hard, even = [], []
    for n in sizes:
        th = np.pi / 2 * 10.0 ** (-12 * rng.random(n))
        hard.append((I.from_angles(th, rng, False), np.sort(th)))
        even.append(I.from_angles((np.arange(n) + 0.5) * (np.pi / 2 / n), rng, False))
    ctx = B.Context(0)
    try:
        plan = B.Batch(ctx, sizes)

        def load(pairs):
            plan.load([to_dev(a) for a, _ in pairs], [to_dev(b) for _, b in pairs])

        load(even)
        plan.run()
        ref = _replay_ms(plan)
        load([p for p, _ in hard])
        ms = _replay_ms(plan)
        first = [x.clone() for x in (plan.theta, plan.V1, plan.U1)]
        for i, (n, ((A1, A2), th)) in enumerate(zip(sizes, hard)):
            R = plan.result(i)
            U1, U2, V1, t = (to_host(R[k]) for k in ("U1", "U2", "V1", "theta"))
            assert np.max(np.abs(t - th)) <= 1e-12 * n
            be = np.hypot(np.linalg.norm(A1 - (U1 * np.cos(t)) @ V1.T), np.linalg.norm(A2 - (U2 * np.sin(t)) @ V1.T))
            assert be / np.sqrt(n) <= 50 * n * U
            for X in (U1, U2, V1):
                assert np.linalg.norm(X.T @ X - np.eye(n), 2) <= 50 * n * U
        load(even)
        plan.run()
        load([p for p, _ in hard])
        plan.run()
        assert all(torch.equal(x, y) for x, y in zip(first, (plan.theta, plan.V1, plan.U1)))
        assert ms <= 8 * ref, (ms, ref)
        plan.close()
    finally:
        ctx.close()
