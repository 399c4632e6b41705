"""Inputs that are no partial isometry: blocks of norm 1e5 with singular values
down to zero, whose X^* X + c I is not positive definite in FP64 at the small
shifts c of Zolo-pd.  The result is then finite or the call says that it is
not; NaN with CSD_OK is neither."""
import numpy as np
import pytest

from tests.gpu_util import to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    return binding


def _blocks(n, cplx, norm=1e5):
    rng = np.random.default_rng(n + cplx)

    def haar():
        X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
        return np.linalg.qr(X)[0]

    s = norm * np.concatenate([np.ones(n // 2), np.zeros(n - n // 2)])
    return (haar() * s) @ haar().conj().T, (haar() * s[::-1]) @ haar().conj().T


@pytest.mark.parametrize("n,cplx,tc", [(100, False, False), (100, True, False), (300, False, False),
                                       (400, False, True)])
def test_csd_is_finite_or_says_so(B, n, cplx, tc):
    A1, A2 = _blocks(n, cplx)
    ctx = B.Context(0)
    try:
        ctx.set_tensor_cores(tc)
        try:
            R = ctx.csd_polar(to_dev(A1), to_dev(A2))
        except B.CSDError:
            R = None
        if R is not None:
            for k in ("U1", "U2", "V1", "theta"):
                assert np.all(np.isfinite(to_host(R[k]))), k
        # the context stays usable
        W = to_host(ctx.polar(to_dev(np.eye(8)))[0])
        assert np.allclose(W, np.eye(8))
    finally:
        ctx.close()


def test_batch_reports_the_instance(B):
    """One such instance among good ones: its status says so, the others are right."""
    from paper_1804_09002_gb300 import inputs as I
    good = [I.haar_csd(n, seed=n) for n in (40, 70)]
    bad = _blocks(64, False)
    ctx = B.Context(0)
    try:
        plan = B.Batch(ctx, [40, 64, 70])
        a = [to_dev(good[0][0]), to_dev(bad[0]), to_dev(good[1][0])]
        b = [to_dev(good[0][1]), to_dev(bad[1]), to_dev(good[1][1])]
        plan.load(a, b)
        status = plan.run()
        R = plan.result(1)
        finite = all(np.all(np.isfinite(to_host(R[k]))) for k in ("U1", "U2", "V1", "theta"))
        assert finite or status[1] != 0
        for i, (_, _, th) in ((0, good[0]), (2, good[1])):
            assert status[i] == 0
            assert np.max(np.abs(to_host(plan.result(i)["theta"]) - th)) <= 1e-12 * 70
        plan.close()
    finally:
        ctx.close()
