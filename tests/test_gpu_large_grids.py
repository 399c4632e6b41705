"""Products with so many columns that their tiles do not fit a grid's second
dimension (65535): 8-column tiles of the FP64 pipe from 524 281 columns on,
16-column blocks of the tensor-core product's combination from 1 048 561 on."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1804_09002_gb300 import binding
    c = binding.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("engine,m,n", [(0, 1, 524281), (0, 3, 700001), (0, 33, 600001), (1, 3, 1048577)])
def test_very_wide_product(ctx, engine, m, n):
    """Small integers, so that every engine is exact."""
    k = 2
    g = torch.Generator(device="cuda:0").manual_seed(n)
    A = torch.randint(-9, 10, (k, m), device="cuda:0", generator=g).double().t()
    Bm = torch.randint(-9, 10, (n, k), device="cuda:0", generator=g).double().t()
    got = ctx.gemm(A, Bm, engine=engine)
    for j in range(0, n, 100000):  # in parts: the reference's own temporaries stay small
        b = Bm[:, j:j + 100000]
        want = A[:, :1] * b[:1, :] + A[:, 1:] * b[1:, :]
        assert torch.equal(got[:, j:j + 100000], want)
