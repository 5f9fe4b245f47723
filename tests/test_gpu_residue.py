"""The product in residue arithmetic (CHASE_FP64 on full storage) against FP64
at the edges of its tiles.

Tolerance.  Row i of A is scaled to a 2-norm in (2^50, 2^51] and rounded to
integers, column j of Y to one in (2^49, 2^50]; the integer product is exact.
Each rounding moves a complex element by at most sqrt(1/2) of a unit, so with
K columns of A

    ||dC_j|| <= sqrt(K/2) (2^-50 + 2^-49) ||A||_F ||y_j||,

and the result's own rounding (a 64-bit fraction of the range, then FP64) adds
at most 2^-49 ||A||_F ||y_j||.  The reference is an FP64 product, whose error
(about sqrt(K) 2^-53 of the same norms) is below that."""
import math

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2006_08498_gb300 as pkg  # noqa: E402


@pytest.fixture(scope="module")
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


def _hemm(ctx, A, Y):
    torch.cuda.synchronize()             # the context's stream is its own
    return ctx.hemm(A, Y)


def _check(A, Y, C):
    K = A.shape[1]
    tol = (math.sqrt(K / 2) * (2.0 ** -50 + 2.0 ** -49) + 2.0 ** -49) * torch.linalg.vector_norm(A)
    err = torch.linalg.vector_norm(C - A @ Y, dim=0)
    assert torch.all(err <= tol * torch.linalg.vector_norm(Y, dim=0))


@pytest.mark.parametrize("n", [1, 16, 17, 48, 49, 96, 97, 144, 145, 289, 512])
def test_column_tiles(ctx, n):
    """Every width of column tile, and one more column than fits."""
    A, Y = _hermitian(600, 1), _block(600, n, 2)
    _check(A, Y, _hemm(ctx, A, Y))


@pytest.mark.parametrize("N", [1, 2, 63, 64, 65, 127, 128, 129, 511, 513, 1025, 2049, 4097])
def test_rows_and_chunks(ctx, N):
    """Row tiles of 128, K chunks of 64, drains every 8 and 16 chunks, norm segments."""
    A, Y = _hermitian(N, 3), _block(N, 5, 4)
    _check(A, Y, _hemm(ctx, A, Y))


@pytest.mark.parametrize("N,n", [(4095, 97), (4095, 98), (4096, 97), (4096, 98), (4097, 98), (6001, 1)])
def test_rules_on_sizes(ctx, N, n):
    """Both sides of the lines between one row of the result per thread and four
    (N n = 400000), of column norms of their own (N = 4096), of row exponents in
    one launch (N = 4096)."""
    A, Y = _hermitian(N, 11), _block(N, n, 12)
    _check(A, Y, _hemm(ctx, A, Y))


def test_longest_unit(ctx):
    """More K chunks than one unit sums (224): K splits."""
    A, Y = _hermitian(14400, 5), _block(14400, 40, 6)
    _check(A, Y, _hemm(ctx, A, Y))


def test_scales_zeros_and_signs(ctx):
    """Rows and columns of very different size, zero ones, subnormal ones, and operands of
    one sign and size, whose residues all add up."""
    A, Y = _hermitian(300, 7), _block(300, 20, 8)
    d = torch.logspace(-30, 30, 300, dtype=torch.float64, device="cuda")
    A = (A * d[:, None] * d[None, :]).T.contiguous().T
    A[7, :] = 0
    A[:, 7] = 0
    Y[:, 3] = 0
    Y[:, 4] *= 1e-300
    Y[:, 5] *= 1e200
    C = _hemm(ctx, A, Y)
    assert torch.all(C[7, :] == 0) and torch.all(C[:, 3] == 0)
    K = A.shape[1]                       # row by row here: each row has a scale of its own
    tol = (math.sqrt(K / 2) * (2.0 ** -50 + 2.0 ** -49) + 2.0 ** -49)
    rows, size = torch.linalg.vector_norm(A, dim=1), Y.abs().amax(dim=0)
    cols = torch.linalg.vector_norm(Y / size.clamp(min=1e-306), dim=0) * size   # without over- or underflow
    assert torch.all((C - A @ Y).abs() <= 2 * tol * rows[:, None] * cols[None, :])
    B = torch.full((1100, 1100), 1.0 - 2.0 ** -52, dtype=torch.complex128, device="cuda").T
    X = torch.full((50, 1100), -1.0 + 1j, dtype=torch.complex128, device="cuda").T
    _check(B, X, _hemm(ctx, B, X))


def test_nonfinite_is_reported(ctx):
    for bad in (float("nan"), float("inf")):
        A, Y = _hermitian(200, 9), _block(200, 6, 10)
        A[150, 3] = bad
        with pytest.raises(pkg.BseError) as ei:
            _hemm(ctx, A, Y)
        assert ei.value.status == pkg.BSE_ENONFINITE
        A, Y = _hermitian(200, 9), _block(200, 6, 10)
        Y[199, 5] = bad
        with pytest.raises(pkg.BseError) as ei:
            _hemm(ctx, A, Y)
        assert ei.value.status == pkg.BSE_ENONFINITE
