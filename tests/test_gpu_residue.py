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

import numpy as np
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


@pytest.mark.parametrize("n", [111, 112, 113, 128, 129])
def test_three_and_four_products(ctx, n):
    """Both sides of the line between four real products and three (tiles of more
    than 112 columns), with every drain of a long unit."""
    A, Y = _hermitian(2100, 13), _block(2100, n, 14)
    _check(A, Y, _hemm(ctx, A, Y))


@pytest.mark.parametrize("n", [5, 97, 113])
def test_largest_sums(ctx, n):
    """Every operand's residue modulo 256 is -128 (integers 2^45 + 128 against
    2-norms of 45.25 times that, 2^44 + 128 for Y): the FP32 sums reach 2^24."""
    N = 1024
    A = torch.full((N, N), 1 + 2.0 ** -38, dtype=torch.complex128, device="cuda").T * (1 + 1j)
    Y = torch.full((n, N), 1 + 2.0 ** -37, dtype=torch.complex128, device="cuda").T * (1 + 1j)
    _check(A, Y, _hemm(ctx, A, Y))


# ---- the general products (Gram and QR entries)

def _integers(rows, cols, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.randint(-2 ** 17, 2 ** 17 + 1, (2, cols, rows), device="cuda", generator=g).double()
    return torch.complex(r[0], r[1]).T


@pytest.mark.parametrize("K,m1,m2", [(63, 4, 3), (64, 4, 3), (65, 1, 1), (64, 33, 40), (127, 129, 16), (1025, 17, 145),
                                     (4096, 31, 5), (4097, 97, 128), (20000, 140, 40), (4097, 512, 512)])
def test_gram_of_integers(ctx, K, m1, m2):
    """Integers of 18 bits are exact in the operands' 58 bits, so only the
    result's own rounding is left (one FP64 product of the 96-bit fraction:
    2^-52 of the element, and the fraction's 2^-70 of the norms); the FP64
    reference is exact: sums of 2 K products of 34 bits stay below 2^53."""
    A, B = _integers(K, m1, 5), _integers(K, m2, 6)
    A[:, 0] = 0.0
    torch.cuda.synchronize()
    for X, Y in ((A, B), (A, A)):
        G, ref = ctx.gram(X, Y), X.conj().T @ Y
        norms = torch.linalg.vector_norm(X, dim=0)[:, None] * torch.linalg.vector_norm(Y, dim=0)[None, :]
        assert torch.all((G - ref).abs() <= 2.0 ** -52 * ref.abs() + 2.0 ** -70 * norms)
    assert torch.equal(G, G.conj().T)


def test_gram_scales_and_nonfinite(ctx):
    """Column norms over the exponent range; non-finite entries give what IEEE
    arithmetic gives (native FP64), and the context stays usable."""
    K, m = 300, 6
    A = _integers(K, m, 7)
    s = 2.0 ** torch.tensor([-1060, -300, 0, 1, 300, 490], device="cuda", dtype=torch.float64)
    B = (A * s).T.contiguous().T
    torch.cuda.synchronize()
    G, ref = ctx.gram(A, B), (A.conj().T @ A) * s
    norms = torch.linalg.vector_norm(A, dim=0)[:, None] * torch.linalg.vector_norm(A, dim=0)[None, :]
    tol = (2.0 ** -52 * (A.conj().T @ A).abs() + 2.0 ** -70 * norms) * s + 2.0 ** -1073
    # the first column's entries lose bits below 2^-1074
    assert torch.all(((G - ref).abs() <= tol)[:, 1:])
    for bad in (float("nan"), float("inf")):
        C = A.clone(memory_format=torch.preserve_format)
        C[7, 2] = bad
        torch.cuda.synchronize()
        G = ctx.gram(C, A)
        fine = torch.isfinite(torch.view_as_real(G)).all(dim=-1)
        assert not fine[2].any() and fine[[0, 1, 3, 4, 5]].all()
    torch.cuda.synchronize()
    assert torch.all((ctx.gram(A, A) - A.conj().T @ A).abs() <= 2.0 ** -52 * norms)


@pytest.mark.parametrize("N,m,k", [(63, 5, 3), (64, 5, 3), (64, 64, 0), (65, 1, 1), (129, 17, 33), (1000, 97, 16),
                                   (4097, 100, 40), (1030, 290, 222)])
def test_qr_of_sizes(ctx, N, m, k):
    """Orthonormal to the bound of CholeskyQR2, 6 (N m + m (m + 1)) 2^-53 (its
    products are at least FP64's here), against L to the same; V R = the
    projected block to 2^-40 of its norm (three passes, each a product to FP64
    rounding over at most m = 290 columns)."""
    V0 = _block(N, m, 8)
    L = torch.linalg.qr(_block(N, k, 9))[0].T.contiguous().T if k else None
    V = V0.clone(memory_format=torch.preserve_format)
    torch.cuda.synchronize()
    out = ctx.qr(V, L)
    V = V if out is None else out
    bound = 6 * (N * m + m * (m + 1)) * 2.0 ** -53
    assert torch.linalg.matrix_norm(V.conj().T @ V - torch.eye(m, device="cuda")) <= bound
    P = V0
    if k:
        assert torch.linalg.matrix_norm(L.conj().T @ V) <= bound
        P = V0 - L @ (L.conj().T @ V0)
    assert torch.linalg.matrix_norm(V @ (V.conj().T @ P) - P) <= 2.0 ** -40 * torch.linalg.matrix_norm(P)


# ---- lines of subnormal numbers

def _down(X, e):
    """X 2^-e, exact where the result is a multiple of 2^-1074."""
    return ((X * 2.0 ** -1000) * 2.0 ** (1000 - e)).T.contiguous().T


@pytest.mark.parametrize("K", [300, 5000])
def test_gram_of_the_smallest_numbers(ctx, K):
    """Columns of entries below 2^-1042, which have no bits in a double's high word: integers of
    18 bits times 2^-1060, exact as operands.  The result as for other integers: 2^-52 of
    the element and 2^-70 of the norms, or a unit of 2^-1074."""
    A, B = _integers(K, 6, 8), _integers(K, 4, 9)
    Bt = _down(B, 1060)
    torch.cuda.synchronize()
    ref = A.conj().T @ B
    norms = torch.linalg.vector_norm(A, dim=0)[:, None] * torch.linalg.vector_norm(B, dim=0)[None, :]
    tol = 2.0 ** -52 * ref.abs() + 2.0 ** -70 * norms + 2.0 ** -13     # in units of 2^-1060
    up = lambda G: (G * 2.0 ** 1000) * 2.0 ** 60
    assert torch.all((up(ctx.gram(A, Bt)) - ref).abs() <= tol)
    assert torch.all((up(ctx.gram(Bt, A)) - ref.conj().T).abs() <= tol.T)


@pytest.mark.parametrize("N", [300, 4200])
def test_hemm_of_the_smallest_numbers(ctx, N):
    """A row of H, and the columns of Y, of such entries: exact as operands, so that only the
    result's own rounding is left (2^-49 of the norms, or a unit of 2^-1074)."""
    H, Y = _integers(N, N, 10), _integers(N, 3, 11)
    ref = H @ Y                          # of 18 bits both: exact
    tol = 2.0 ** -49 * torch.linalg.vector_norm(H, dim=1)[:, None] * torch.linalg.vector_norm(Y, dim=0)[None, :]
    Ht, Yt = H.clone(memory_format=torch.preserve_format), _down(Y, 1070)
    Ht[5] = _down(H, 1063)[5]
    torch.cuda.synchronize()
    C = (ctx.hemm(H, Yt) * 2.0 ** 1000) * 2.0 ** 70
    assert torch.all((C - ref).abs() <= tol + 2.0 ** -3)
    C = ctx.hemm(Ht, Y)
    C[5] = (C[5] * 2.0 ** 1000) * 2.0 ** 63
    assert torch.all((C - ref).abs() <= tol + 2.0 ** -10)


# ---- columns with entries far below their norm

def _graded_cases():
    def first(K, m, head, rest):
        A = _block(K, m, 31) * rest
        A[0] = head
        return A
    yield "one large entry against a zero", lambda K, m1, m2: (first(K, m1, 1.0, 1e-9), first(K, m2, 0.0, 1.0))
    yield "one entry against a tiny one", lambda K, m1, m2: (first(K, m1, 1.0, 0.0), first(K, m2, 1e-20, 1.0))
    def decay(K, m1, m2):
        d = torch.logspace(0, -18, K, dtype=torch.float64, device="cuda")[:, None]
        return _block(K, m1, 32) * d, _block(K, m2, 33) * d.flip(0)
    yield "opposite decays", decay
    def parts(K, m1, m2):
        B = _block(K, m2, 34)
        return _block(K, m1, 35).real.to(torch.complex128), torch.complex(B.real, 1e-15 * B.imag)
    yield "a small imaginary part", parts
    def one_pair(K, m1, m2):
        A, B = _block(K, m1, 36), _block(K, m2, 37)
        A[:, m1 - 1] = 0
        A[3, m1 - 1] = 1
        B[3, m2 - 1] = 1e-18
        return A, B
    yield "one pair among many", one_pair


@pytest.mark.parametrize("K,m1,m2", [(64, 3, 2), (400, 7, 20), (20000, 65, 70), (4097, 1, 130)])
@pytest.mark.parametrize("case", range(5))
def test_gram_of_graded_columns(ctx, K, m1, m2, case):
    """Real and imaginary part of every element to FP64 against the sum of their own
    products' magnitudes, as a sum of FP64 products has it in the worst case (2 K
    roundings, and as many in the reference); entries far below their column's norm
    count."""
    name, make = list(_graded_cases())[case]
    A, B = (x.T.contiguous().T for x in make(K, m1, m2))
    torch.cuda.synchronize()
    G = ctx.gram(A, B).cpu().numpy()
    a, b = A.cpu().numpy(), B.cpu().numpy()
    ar, ai, br, bi = (np.asfortranarray(x) for x in (a.real, a.imag, b.real, b.imag))
    re, im = ar.T @ br + ai.T @ bi, ar.T @ bi - ai.T @ br
    ar, ai, br, bi = abs(ar), abs(ai), abs(br), abs(bi)
    tol = 4 * K * 2.0 ** -53
    assert np.all(abs(G.real - re) <= tol * (ar.T @ br + ai.T @ bi)), name
    assert np.all(abs(G.imag - im) <= tol * (ar.T @ bi + ai.T @ br)), name


# ---- the operands' precision

def test_flat_matrix_keeps_the_precision_of_48_bit_slices(ctx):
    """Entries of even size.  An operand's unit is at most 2^-53 of its norm, a rounding
    moves a real number by a uniform half unit at most (variance 1/12): the two
    operands give an element's complex error an rms of at most sqrt(1/6 + 1/6)
    2^-53 = 2^-53.8 of the norms' product.  The reference sums FP64 products of 200
    columns (2^-56.8).  48-bit slices have about 2^-50.4 at this size."""
    N, n = 3000, 24
    A, Y = _hermitian(N, 15), _block(N, n, 16)
    torch.cuda.synchronize()
    C = ctx.hemm(A, Y)
    ref = sum(A[:, k:k + 200] @ Y[k:k + 200] for k in range(0, N, 200))
    e = (C - ref).abs() / (torch.linalg.vector_norm(A, dim=1)[:, None] * torch.linalg.vector_norm(Y, dim=0)[None, :])
    assert e.square().mean().sqrt() <= 2.0 ** -53.7


@pytest.mark.parametrize("n", [5, 97, 113])
def test_largest_sums_of_54_bits(ctx, n):
    """Every operand's residue modulo 256 is -128 (integers 2^48 + 128 against
    2-norms of 45.25 times that, both sides): the FP32 sums reach 2^24."""
    N = 1024
    A = torch.full((N, N), 1 + 2.0 ** -41, dtype=torch.complex128, device="cuda").T * (1 + 1j)
    Y = torch.full((n, N), 1 + 2.0 ** -41, dtype=torch.complex128, device="cuda").T * (1 + 1j)
    _check(A, Y, _hemm(ctx, A, Y))


# ---- the product on slices of all of H, which chase_hemm no longer reaches

@pytest.mark.parametrize("N,m", [(63, 1), (129, 33), (333, 7), (640, 96), (1000, 97), (2050, 40)])
def test_product_on_six_slices(ctx, N, m):
    """Rayleigh-Ritz keeps the products on six slices: H V of its vectors V = Q Y against its
    own H V = (H Q) Y.  An error of 2^-49.7 of ||h_i|| ||v_j|| (rms, entries of even size) in
    each of three products; a slice less costs 8 bits: 2^-42."""
    A = _hermitian(N, 61)
    Q = torch.linalg.qr(_block(N, m, 62))[0].T.contiguous().T
    torch.cuda.synchronize()
    _, V, HV, _ = ctx.rayleigh_ritz(A, Q)
    e = (HV - A @ V).abs() / torch.linalg.vector_norm(A, dim=1)[:, None]
    assert e.square().mean().sqrt() <= 2.0 ** -46
