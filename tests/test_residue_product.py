"""The FP64-class product by residues (spin_gemm_ozaki with 4 slices and more,
the mixed form's Schur complements and residuals): exact on integers that the
fixed point holds, at the edges of its tiles, exact runs and TMA padding; the
same bits whatever panels its arena allows; rows and columns with infinities,
NaN, zeros, subnormals and extreme exponents."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spin():
    import paper_1801_04723_gb300 as s

    s.build()
    s.lib()
    return s


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()


@pytest.mark.parametrize("slices", [4, 5, 6, 7])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (127, 255, 63), (128, 256, 64), (129, 257, 65), (5, 700, 1023),
                                   (260, 3, 1024), (130, 300, 1025), (64, 513, 5000), (1000, 16, 8200)])
def test_integers_exact(spin, m, n, k, slices):
    """Integers up to 2^19: every sum is below 2^53, so the FP64 result is the integer itself."""
    rng = np.random.default_rng(m + 3 * n + 7 * k + slices)
    A, B = rng.integers(-2 ** 19, 2 ** 19 + 1, (m, k)), rng.integers(-2 ** 19, 2 ** 19 + 1, (k, n))
    C = rng.integers(-1000, 1000, (m, n))
    want = C - A @ B
    want[np.arange(min(m, n)), np.arange(min(m, n))] += 1
    D = spin.gemm_ozaki(dev(A), dev(B), slices=slices, alpha=-1.0, beta=1.0, C=dev(C), add_identity=True)
    torch.cuda.synchronize()
    assert spin.take_device_error() == 0
    np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), want)


def test_largest_inner_dimension_and_beyond(spin):
    """k = 98304 (96 exact runs) is the residue form's largest; above it the digit form runs."""
    for k in (98304, 98305):
        rng = np.random.default_rng(k)
        A, B = rng.integers(-1000, 1001, (40, k)), rng.integers(-1000, 1001, (k, 24))
        D = spin.gemm_ozaki(dev(A), dev(B), slices=5)
        torch.cuda.synchronize()
        assert spin.take_device_error() == 0
        np.testing.assert_array_equal(D.cpu().numpy().astype(np.int64), A @ B)


def test_extreme_rows_and_columns(spin):
    """Rows and columns scaled by powers of two scale the result exactly; a
    zero row gives zeros; a row or column with an infinity or NaN gives
    non-finite values there and nowhere else."""
    rng = np.random.default_rng(5)
    m, n, k = 200, 300, 400
    A, B = rng.integers(-2 ** 18, 2 ** 18 + 1, (m, k)), rng.integers(-2 ** 18, 2 ** 18 + 1, (k, n))
    er, ec = rng.integers(-400, 401, m), rng.integers(-400, 401, n)
    er[3] = -1060  # a row of subnormals
    ec[:] = np.where(rng.random(n) < 0.1, 0, ec)
    Af, Bf = np.ldexp(A.astype(float), er[:, None]), np.ldexp(B.astype(float), ec)
    Af[7] = 0.0
    exact = (A @ B).astype(float)
    want = np.ldexp(np.where(np.arange(m)[:, None] == 7, 0.0, exact), er[:, None] + ec)
    keep = np.arange(m) != 3  # the subnormal row's integers are shortened: finite, nothing more
    D = spin.gemm_ozaki(dev(Af), dev(Bf), slices=7).cpu().numpy()
    np.testing.assert_array_equal(D[keep], want[keep])
    assert np.isfinite(D[3]).all()
    Af[11, 5], Bf[17, 13] = np.nan, np.inf
    D = spin.gemm_ozaki(dev(Af), dev(Bf), slices=7).cpu().numpy()
    bad = (np.arange(m)[:, None] == 11) | (np.arange(n) == 13)
    assert not np.isfinite(D[bad]).any()
    np.testing.assert_array_equal(D[keep][~bad[keep]], want[keep][~bad[keep]])


@pytest.mark.parametrize("n", [600, 1100, 2048])
def test_panels_change_no_bit(spin, n):
    """A mixed inversion in a caller's workspace of the least size (several
    panels) and in the library's (one panel pair)."""
    g = torch.Generator(device="cuda:0").manual_seed(n)
    G = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda:0")
    A = (G @ G.T).div_(n)
    A = (A + A.T).mul_(0.5)
    A.diagonal().add_(0.5)
    X, info = spin.invert(A, precision="bf16x3")
    ws = torch.empty(spin.workspace_bytes(n, precision="bf16x3") // 8 + 1, dtype=torch.float64, device="cuda:0")
    Y, info2 = spin.invert(A, precision="bf16x3", workspace=ws)
    assert info["refine_iters"] == info2["refine_iters"]
    assert torch.equal(X, Y)


def exact_product(A, B):
    """A B in extended precision, rows in blocks."""
    L = np.longdouble
    return np.stack([(A[i].astype(L)[:, None] * B.astype(L)).sum(axis=0) for i in range(A.shape[0])])


@pytest.mark.parametrize("slices", [4, 5, 6, 7])
@pytest.mark.parametrize("k", [64, 128, 256, 512, 2048, 8192])
def test_bits_of_the_digit_slices(spin, k, slices):
    """Dense operands: the error is that of rounding them to the 8 s - 1 bits of
    s digit slices, nothing more: independent uniform errors of up to half a
    unit u = 2^-(8 s - 1) of the row's (column's) power of two, so a standard
    deviation of u / sqrt(12) sqrt(4^e_i |b_j|^2 + 4^f_j |a_i|^2) per output,
    plus the rounding of the result.  The digit form has that error and the
    pairs it leaves out."""
    rng = np.random.default_rng(k + slices)
    m, n = 96, 80
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    D = spin.gemm_ozaki(dev(A), dev(B), slices=slices)
    torch.cuda.synchronize()
    want = exact_product(A, B)
    u = 2.0 ** -(8 * slices - 1)
    ei, fj = np.frexp(np.abs(A).max(axis=1))[1], np.frexp(np.abs(B).max(axis=0))[1]
    var = u * u / 12 * (4.0 ** ei[:, None] * (B * B).sum(axis=0) + 4.0 ** fj * (A * A).sum(axis=1)[:, None])
    var += (2.0 ** -53 * np.abs(want.astype(float))) ** 2
    z = (D.cpu().numpy() - want).astype(float) / np.sqrt(var)
    # 7680 outputs sharing 176 rows and columns: the root mean square is within 3 % of its expectation
    assert np.sqrt(np.mean(z * z)) <= 1.05
    assert np.abs(z).max() <= 7.0


@pytest.mark.parametrize("slices", [4, 5, 6])
@pytest.mark.parametrize("family", ["spd", "sdd"])
@pytest.mark.parametrize("n", [64, 80, 96, 130, 160, 300])
def test_residual_within_its_error_model(spin, n, family, slices):
    """The refinement certifies with 0.7 sqrt(n) 2^-(8 s - 1) as the residual's
    error relative to |A|_F |X|_F."""
    rng = np.random.default_rng(n + slices)
    if family == "spd":
        G = rng.standard_normal((n, n))
        A = G @ G.T / n + 0.3 * np.eye(n)
    else:
        A = rng.uniform(-1, 1, (n, n)) + n * np.eye(n)
    X = np.linalg.inv(A)
    R = spin.gemm_ozaki(dev(A), dev(X), slices=slices, alpha=-1.0, add_identity=True)
    torch.cuda.synchronize()
    want = np.eye(n) - exact_product(A, X)
    err = np.linalg.norm((R.cpu().numpy() - want).astype(float)) / np.linalg.norm(A) / np.linalg.norm(X)
    assert err <= 0.7 * np.sqrt(n) * 2.0 ** -(8 * slices - 1)


@pytest.mark.parametrize("n", [3, 16, 20, 32, 33, 34, 35, 36, 37, 38, 39, 40, 48, 64, 65, 96, 127])
def test_small_orders_in_the_least_workspace(spin, n):
    """The form of the residual depends on the order alone: the certified residual is that of the
    library's own buffer, up to the order in which its n^2 squares are added (n^2 2^-53)."""
    g = torch.Generator(device="cuda:0").manual_seed(n)
    G = torch.randn((n, n), generator=g, dtype=torch.float64, device="cuda:0")
    A = G @ G.T / n + 0.5 * torch.eye(n, dtype=torch.float64, device="cuda:0")
    for tol, slices in ((1e-4, 0), (1e-10, 0), (1e-13, 7)):
        kw = dict(precision="bf16x3", leaf=16, residual_slices=slices)
        X, info = spin.invert(A, tol=tol, **kw)
        ws = torch.empty(spin.workspace_bytes(n, **kw), dtype=torch.uint8, device="cuda:0")
        Y, info2 = spin.invert(A, tol=tol, workspace=ws, **kw)
        assert info["refine_iters"] == info2["refine_iters"]
        assert abs(info["rel_residual"] - info2["rel_residual"]) <= 1e-10 * info["rel_residual"]
        assert torch.equal(X, Y)
