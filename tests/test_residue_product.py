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
