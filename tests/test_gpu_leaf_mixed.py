"""Leaves of very different sizes in one call of the leaf eigensolver
(leaf.cu).  With a leaf of 257 to 512 floats per column in the call, a CTA of
the FP32 stage has 16 warps and each owns one column of the first block, while
a leaf of 33 to 96 rows still has blocks of up to 48 columns."""
import numpy as np
import pytest

from tests.gpu_util import U, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    return binding


def _two_groups(small, large, cplx):
    """Hermitian with `small` eigenvalues well above zero and `large` below,
    trace 0: its diagonal, and so the first shift, lies in the gap, and one
    split leaves two leaves of these sizes."""
    n = small + large
    rng = np.random.default_rng(n + 7 * cplx)
    X = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cplx else 0)
    Q = np.linalg.qr(X)[0]
    up = large / small
    ev = np.concatenate([up + 0.3 * rng.uniform(-1, 1, small), -1 + 0.3 * rng.uniform(-1, 1, large)])
    M = (Q * ev) @ Q.conj().T
    return (M + M.conj().T) / 2


def _launches(B, ctx, M):
    before = B.lib.csd_launch_count()
    lam, V, info = ctx.heig(to_dev(M))
    return to_host(lam), to_host(V), info, B.lib.csd_launch_count() - before


@pytest.mark.parametrize("small,large,cplx,leaf", [(90, 300, False, 320), (33, 300, False, 320), (96, 500, False, 512),
                                                   (90, 200, True, 256), (40, 150, True, 160)])
def test_small_leaf_beside_a_large_one(B, small, large, cplx, leaf):
    """Accuracy, and that the small leaf leaves the FP32 stage converged: a
    leaf that does not sends the call through the stage again, with one launch
    per sweep and round.  The reference is the same call with a leaf of 112 rows
    (four blocks, whose geometry does not depend on the other leaf) in the small
    one's place: it may differ by refinement steps of six launches each, but not
    by a pass (12 sweeps of at least 13 rounds)."""
    ctx = B.Context(0)
    try:
        ctx.set_eig_leaf(leaf)
        M = _two_groups(small, large, cplx)
        lam, V, info, count = _launches(B, ctx, M)
        assert info["eig_splits"] == 1 and info["eig_leaves"] == 2
        *_, ref = _launches(B, ctx, _two_groups(112, large, cplx))
    finally:
        ctx.close()
    n = small + large
    nb = np.linalg.norm(M, 2)
    assert np.max(np.abs(lam - np.linalg.eigvalsh(M))) <= 50 * n * U * nb
    assert np.linalg.norm(M @ V - V * lam) <= 50 * n * U * nb
    assert np.linalg.norm(V.conj().T @ V - np.eye(n), 2) <= 50 * n * U
    assert count <= ref + 12 * 13 // 2, (count, ref)
