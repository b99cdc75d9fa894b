"""The single inversions' leaf with its columns over a cluster (orders up to
256) at the edges of its layout (rows per lane, columns per CTA, panels in the
slot ring) and of its pivot search and reciprocal: bit for bit the batched
paths' leaf, which shares none of that code (rows in one CTA up to 128, rows
over a cluster above), with the same status."""
import time

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


def matrix(kind, L, rng):
    if kind == "uniform":
        return rng.uniform(-1, 1, (L, L))
    if kind == "ties":  # equal magnitudes everywhere: the lowest position wins
        return rng.choice([-1.0, 1.0], (L, L)) + np.diag(np.full(L, 2.0))
    if kind == "low_words":  # rows that differ in the last bits of |a| only
        return rng.choice([-1.0, 1.0], (L, L)) * (1.0 + rng.integers(0, 4, (L, L)) * 2.0 ** -52) + np.diag(
            np.full(L, 3.0))
    if kind == "range":  # pivots near both ends of the exponent range
        d = 2.0 ** rng.choice([-1015.0, -1000.0, -3.0, 0.0, 7.0, 1000.0, 1022.0], L)
        return rng.uniform(0.5, 1, (L, L)) * 2.0 ** -1020 + np.diag(d)
    if kind == "powers":  # reciprocals that are exact, and significands of all ones
        return np.diag(rng.choice([2.0 ** -60, 1.0, 2.0 - 2.0 ** -52, -(2.0 - 2.0 ** -52) * 2.0 ** 40], L))
    A = rng.uniform(-1, 1, (L, L))
    if kind == "zero_column":
        A[:, L // 2] = 0.0
    else:
        A[L // 3, L // 2] = np.nan if kind == "nan" else np.inf
    return A


@pytest.mark.parametrize("kind", ["uniform", "ties", "low_words", "range", "powers", "zero_column", "nan", "inf"])
@pytest.mark.parametrize("L", [1, 2, 4, 5, 16, 17, 31, 32, 33, 63, 64, 65, 80, 127, 128, 129, 144, 145, 255, 256])
def test_same_bits_as_the_batched_leaf(spin, L, kind):
    A = torch.from_numpy(np.ascontiguousarray(matrix(kind, L, np.random.default_rng(1000 * L + len(kind))))).cuda()
    info = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    start = time.perf_counter()
    X = spin.leaf_inverse(A, info_dev=info)
    torch.cuda.synchronize()
    assert time.perf_counter() - start < 2.0  # a bad pivot ends every warp, none waits for its limit (4 s)
    # enough leaves that the batch does not take clusters of columns as well
    Y, status = spin.invert_batched([A] * 80, leaf=L, schedule="lockstep")
    torch.cuda.synchronize()
    assert info[0].item() == status[0].item()
    Z, few = spin.invert_batched([A] * 3, leaf=L, schedule="lockstep")  # clusters of columns, up to 152 CTAs
    torch.cuda.synchronize()
    assert few[2].item() == status[0].item()
    if info[0].item() == 0:
        assert torch.equal(X, Y[0]) and torch.equal(X, Z[2])


@pytest.mark.parametrize("apart", [0.0, 2.0 ** -52, -(2.0 ** -52)])
@pytest.mark.parametrize("L,row", [(L, row) for L in (33, 64, 65, 128, 256) for row in (32, 64, 96, 224) if row < L])
def test_first_pivot_tied_with_a_row_of_its_lane(spin, L, row, apart):
    """Rows 0 and 32 t, which one lane holds, have the largest entries of column
    0: equal ones (the lower row is the pivot) or one unit in the last place apart."""
    A = np.random.default_rng(L + row).uniform(-0.5, 0.5, (L, L))
    A[0, 0], A[row, 0] = 1.0 + 2.0 ** -50, -(1.0 + 2.0 ** -50 + apart)
    A = torch.from_numpy(A).cuda()
    X = spin.leaf_inverse(A)
    Y, _ = spin.invert_batched([A] * 80, leaf=L, schedule="lockstep")  # no clusters of columns
    torch.cuda.synchronize()
    assert torch.equal(X, Y[0])


@pytest.mark.parametrize("count", [12, 20, 38, 76])
@pytest.mark.parametrize("kind", ["uniform", "ties", "zero_column"])
@pytest.mark.parametrize("L", [16, 17, 32, 33, 50, 64, 65, 100, 127, 128, 200])
def test_narrow_clusters_of_a_batch(spin, L, kind, count):
    """More leaves at once take narrower clusters with wider panels (16 columns a
    CTA at most), up to the count that takes one CTA a leaf."""
    As = [torch.from_numpy(np.ascontiguousarray(matrix(kind, L, np.random.default_rng(z + L)))).cuda() for z in range(4)]
    As = (As * 20)[:80]
    Y, want = spin.invert_batched(As, leaf=L, schedule="lockstep")
    X, status = spin.invert_batched(As[:count], leaf=L, schedule="lockstep")
    torch.cuda.synchronize()
    assert status.tolist() == want.tolist()[:count]
    if status[0].item() == 0:
        assert all(torch.equal(x, y) for x, y in zip(X, Y))
