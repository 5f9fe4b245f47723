"""Failures that a call has to report.  Every failure is made on the host: a
short limit of the kernels' bounded waits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2006_08498_gb300 as pkg  # noqa: E402


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_08498_gb300 import build
    build.build()
    c = pkg.Context(0)
    yield c
    c.close()


def _block(rows, cols, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((cols, rows), dtype=torch.complex128, device="cuda", generator=g).T


def _hermitian(n, seed):
    A = _block(n, n, seed)
    return (A + A.conj().T).T.contiguous().T


@pytest.mark.parametrize("n,kw", [
    (30, {}), (90, {}), (100, {}),       # four real products: each variant of the kernel
    (130, {}),                           # three
    (100, dict(precision=pkg.CHASE_MIXED_FP32)), (100, dict(half_storage=True))])
def test_expired_wait_in_every_product_kernel(ctx, n, kw):
    """Every variant winds down (its copies and MMAs land before its memory
    goes), reports, and leaves the context usable."""
    A, Y = _hermitian(700, 1), _block(700, n, 2)
    torch.cuda.synchronize()
    C = ctx.hemm(A, Y, **kw)
    ctx.set_wait_limit(1e-9)
    for _ in range(2):
        with pytest.raises(pkg.BseError) as ei:
            ctx.hemm(A, Y, **kw)
        assert ei.value.status == pkg.BSE_ETIMEOUT
    ctx.set_wait_limit(2.0)
    assert torch.equal(ctx.hemm(A, Y, **kw), C)
