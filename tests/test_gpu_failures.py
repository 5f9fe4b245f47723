"""Failures that a call has to report, and what it does where memory is short.  Every
failure is made on the host: a short limit of the kernels' bounded waits, set by the
caller or at one point of a call, an allocation that is refused (bsechase_inject)."""
import ctypes
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2006_08498_gb300 as pkg  # noqa: E402

LAST_PASS_WAIT_NS, PRODUCT_REFUSALS = 0, 1      # bsechase_inject


@pytest.fixture
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_08498_gb300 import build
    build.build()
    c = pkg.Context(0)
    yield c
    c.close()


def _inject(ctx, point, value):
    f = pkg.load().bsechase_inject
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_int64]
    assert f(ctx._h, point, value) == pkg.BSE_OK


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


def test_solve_reports_a_failure_of_its_last_pass(ctx):
    """The pass over the output vectors is the last thing that a solve does: a
    wait that expires there fails the call like one before it.  (A look at a barrier
    suspends a thread for some microseconds; the sums of this size take longer.)"""
    H = ctx.build_hamiltonian(0, 500, 4, 4)
    e, V, _, _ = ctx.solve(H, 100, 20)
    _inject(ctx, LAST_PASS_WAIT_NS, 1)
    with pytest.raises(pkg.BseError) as ei:
        ctx.solve(H, 100, 20)
    assert ei.value.status == pkg.BSE_ETIMEOUT
    _inject(ctx, LAST_PASS_WAIT_NS, 0)
    e2, V2, _, _ = ctx.solve(H, 100, 20)
    assert np.array_equal(e, e2) and torch.equal(V, V2)


def test_expired_wait_in_qr(ctx):
    """The products of chase_qr are tensor-core kernels: the context's limit holds for their waits."""
    N, m = 20000, 100                    # sums long enough for a wait to expire
    V = _block(N, m, 3)
    torch.cuda.synchronize()
    ctx.set_wait_limit(1e-9)
    with pytest.raises(pkg.BseError) as ei:
        ctx.qr(V.clone(memory_format=torch.preserve_format))
    assert ei.value.status == pkg.BSE_ETIMEOUT
    ctx.set_wait_limit(2.0)
    Q = ctx.qr(V)
    assert torch.linalg.matrix_norm(Q.conj().T @ Q - torch.eye(m, device="cuda")) <= 6 * (N * m + m * (m + 1)) * 2.0 ** -53


def test_expired_wait_in_gram(ctx):
    """An expired wait fails the call; only missing memory and non-finite operands are for native FP64."""
    A, B = _block(40000, 140, 4), _block(40000, 120, 5)
    torch.cuda.synchronize()
    G = ctx.gram(A, B)
    ctx.set_wait_limit(1e-9)
    with pytest.raises(pkg.BseError) as ei:
        ctx.gram(A, B)
    assert ei.value.status == pkg.BSE_ETIMEOUT
    ctx.set_wait_limit(2.0)
    assert torch.equal(ctx.gram(A, B), G)


@pytest.mark.parametrize("N,m,k", [(64, 5, 100), (100, 40, 129), (100, 129, 0), (64, 65, 3)])
def test_qr_of_more_columns_than_rows(ctx, N, m, k):
    """More kept columns than rows (zero ones, or repeated at no weight): projected like
    fewer.  More columns than rows have no orthonormal basis: BSE_ENONFINITE."""
    V0, L = _block(N, m, 6), None
    if k:
        L = torch.zeros((k, N), dtype=torch.complex128, device="cuda").T
        L[:, :3] = torch.linalg.qr(_block(N, 3, 7))[0]
    V = V0.clone(memory_format=torch.preserve_format)
    torch.cuda.synchronize()
    if m > N:
        with pytest.raises(pkg.BseError) as ei:
            ctx.qr(V, L)
        assert ei.value.status == pkg.BSE_ENONFINITE
        return
    ctx.qr(V, L)
    bound = 6 * (N * m + m * (m + 1)) * 2.0 ** -53
    assert torch.linalg.matrix_norm(V.conj().T @ V - torch.eye(m, device="cuda")) <= bound
    assert torch.linalg.matrix_norm(L.conj().T @ V) <= bound
    P = V0 - L @ (L.conj().T @ V0)
    assert torch.linalg.matrix_norm(V @ (V.conj().T @ P) - P) <= 2.0 ** -40 * torch.linalg.matrix_norm(P)


def test_gram_does_not_depend_on_earlier_calls(ctx):
    """Above 8 GB of workspace chase_gram stays in native FP64, whatever buffers
    other calls have left in the context: the same call gives the same bits."""
    A, B = _block(870000, 4, 41), _block(870000, 4, 42)   # 3.3 + 5.3 GB of residues
    torch.cuda.synchronize()
    fresh = ctx.gram(A, B)
    with pkg.Context(0) as other:
        other.gram(_block(291000, 300, 43), _block(291000, 1, 44))     # 3.4 GB of left operands
        X = _block(103000, 512, 45)
        torch.cuda.synchronize()
        other.gram(X, X.clone(memory_format=torch.preserve_format))    # 5.3 GB of right ones
        assert torch.equal(other.gram(A, B), fresh)


def test_products_without_memory_for_the_residues(ctx):
    """One refused allocation: the buffers are given back and taken anew, the same
    product.  Two: the product on slices, to its own bound (5e-11), and solves too; the
    solve without the stored H takes the same bits."""
    A, Y = _hermitian(1000, 51), _block(1000, 40, 52)
    torch.cuda.synchronize()
    C = ctx.hemm(A, Y)
    _inject(ctx, PRODUCT_REFUSALS, 1)
    assert torch.equal(ctx.hemm(A, Y), C)
    _inject(ctx, PRODUCT_REFUSALS, 2)
    D = ctx.hemm(A, Y)
    assert not torch.equal(D, C)
    norm = torch.linalg.matrix_norm(A, 2) * torch.linalg.vector_norm(Y, dim=0)
    assert torch.all(torch.linalg.vector_norm(D - C, dim=0) <= 5e-11 * norm)
    H = ctx.build_hamiltonian(3, 63, 4, 4)
    e, _, _, st = ctx.solve(H, 20, 10, seed=3)
    assert _flops(st, 1008) < 8 * 21
    _inject(ctx, PRODUCT_REFUSALS, 2)
    e2, V2, _, st = ctx.solve(H, 20, 10, seed=3)
    assert abs(_flops(st, 1008) - 8 * 21) < 1e-6 * 8 * 21
    assert np.max(np.abs(e2 - e) / np.abs(e)) <= 1e-10
    _inject(ctx, PRODUCT_REFUSALS, 2)
    e3, V3, _, _ = ctx.solve_bse(3, 63, 4, 4, 20, 10, seed_start=3)
    assert np.array_equal(e2, e3) and torch.equal(V2, V3)


def _flops(st, N):
    """Tensor flops per complex multiply-add of a solve's products with H."""
    return st["tc_kernel_tflops"] * st["tc_kernel_ms"] * 1e9 / (float(N) * N * st["matvecs"])


def test_request_whose_residues_exceed_the_budget(ctx):
    """The smallest budget that admits a request runs it on slices; one that holds
    the residues runs it as the direct solve, bit for bit."""
    R = dict(seed=3, Nk=63, Nv=4, Nc=4, nev=20, nex=10)
    H = ctx.build_hamiltonian(3, 63, 4, 4)
    e, _, _, _ = ctx.solve(H, 20, 10, seed=3)

    def run(budget):
        ctx.server_create(budget, 1)
        try:
            return ctx.wait(ctx.submit(**R))
        except pkg.BseError as err:
            assert err.status == pkg.BSE_ENOMEM
            return None
        finally:
            ctx.server_destroy()

    lo, hi = 1 << 20, 1 << 30                       # refused, admitted
    assert run(lo) is None
    full = run(hi)
    assert np.array_equal(full["evals"], e) and _flops(full["stats"], 1008) < 8 * 21
    while hi - lo > 1 << 16:
        mid = (lo + hi) // 2
        r = run(mid)
        if r is None:
            lo = mid
        else:
            hi, least = mid, r
    assert least["status"] == pkg.BSE_OK
    assert abs(_flops(least["stats"], 1008) - 8 * 21) < 1e-6 * 8 * 21
    assert np.max(np.abs(least["evals"] - e) / np.abs(e)) <= 1e-10


@pytest.mark.parametrize("model", [None, dict(rank_x=0), dict(rank_x=1)])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 1, 1), (1, 2, 3), (3, 1, 2), (31, 1, 1), (33, 1, 1)])
def test_generator_of_the_smallest_matrices(ctx, shape, model):
    """Matrices within one tile: the elements that the tile has beyond them have no ring distance (the
    generator read the distance table at down to -31 for them, before the tables' memory for N < 7)."""
    H = ctx.build_hamiltonian(5, *shape, model).cpu().numpy()
    ref = oracle.build_h(5, *shape, model)
    assert np.max(np.abs(H - ref)) <= 4e-15 * np.max(np.abs(ref))


@pytest.mark.parametrize("N,m,k", [(400, 20, 0), (400, 20, 9), (2000, 75, 30), (129, 60, 0), (63, 12, 4)])
@pytest.mark.parametrize("kind", ["equal", "half equal", "rank 5", "nearly equal", "kept"])
def test_qr_of_dependent_columns(ctx, N, m, k, kind):
    """Columns that depend on others (or on kept ones) get directions of their own: the basis is
    orthonormal to rounding, 2^-50 a column, and holds the columns to what is added to
    them, 2^-40 of each (2^-38 with the passes).  Native FP64 (N < 64) may keep a
    direction of less than its rounding over the square root of the first pass' shift
    without failing, and holds the columns to that."""
    V0 = _block(N, m, 71)
    L = torch.linalg.qr(_block(N, k, 72))[0].T.contiguous().T if k else None
    if kind == "equal":
        V0[:, 4] = V0[:, 5]
    elif kind == "half equal":
        V0[:, m // 2:] = V0[:, :m - m // 2].clone()
    elif kind == "rank 5":
        V0 = (_block(N, 5, 73) @ _block(5, m, 74)).T.contiguous().T
    elif kind == "nearly equal":
        V0[:, 4] = V0[:, 5] + 1e-10 * V0[:, 6]
    elif k:
        V0[:, 2] = L[:, 1]
    V = V0.clone(memory_format=torch.preserve_format)
    torch.cuda.synchronize()
    ctx.qr(V, L)
    assert torch.linalg.matrix_norm(V.conj().T @ V - torch.eye(m, device="cuda")) <= m * 2.0 ** -50
    P = V0
    if k:
        assert torch.linalg.matrix_norm(L.conj().T @ V) <= m * 2.0 ** -50
        P = V0 - L @ (L.conj().T @ V0)
    span = 2.0 ** -38 if N >= 64 else 2.0 ** -53 / math.sqrt(11 * (N * m + m * (m + 1)) * 2.0 ** -53 * m)
    assert torch.linalg.matrix_norm(V @ (V.conj().T @ P) - P) <= span * torch.linalg.matrix_norm(P)


@pytest.mark.parametrize("kw", [{}, dict(precision=pkg.CHASE_MIXED_FP32), dict(half_storage=True),
                                dict(precision=pkg.CHASE_FP64_DFMA)])
def test_solve_from_a_dependent_start_block(ctx, kw):
    H = ctx.build_hamiltonian(0, 63, 4, 4)
    e, _, _, _ = ctx.solve(H, 20, 10)
    X = _block(1008, 30, 75)
    X[:, 10:20] = X[:, :10].clone()
    torch.cuda.synchronize()
    e2, V, _, _ = ctx.solve(H, 20, 10, V0=X, **kw)
    assert np.max(np.abs(e2 - e) / np.abs(e)) <= 1e-10
    assert torch.linalg.matrix_norm(V.conj().T @ V - torch.eye(20, device="cuda")) <= 20 * 2.0 ** -50
