"""Plain inversions above order 4096, whose large products run by residues on
the tensor cores where that is at least as accurate as the FP64 kernel, decided
on the device from the operands' exponents.  An inversion in a caller's
workspace of exactly spin_workspace_bytes has no room for the residues: it is
the FP64 kernel's result, to compare with."""
import numpy as np
import pytest

import bounds
import oracle
from paper_1801_04723_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = 4161  # split 2112 + 2049: every product of the top level is above 2048
LEAF = 128
LINE = 256  # products above it in every dimension, in inversions whose top products are above 2048


@pytest.fixture(scope="module")
def spin():
    import paper_1801_04723_gb300 as s

    s.build()
    s.lib()
    return s


def fp64_kernel_inverse(spin, A, schedule="default", check=True):
    n = A.shape[0]
    size = spin.workspace_bytes(n, leaf=LEAF, schedule=schedule)
    ws = torch.empty(size, dtype=torch.uint8, device="cuda:0")
    X, info = spin.invert(A, leaf=LEAF, workspace=ws, schedule=schedule, check=check)
    torch.cuda.synchronize()
    return X, info


def products_by_residues(spin, A, **kw):
    spin.profile_start()
    X, info = spin.invert(A, leaf=LEAF, **kw)
    rec = spin.profile_collect()
    torch.cuda.synchronize()
    small = [r for r in rec if r["kind"] in ("gemm_tc", "gemm_f64") and min(r["m"], r["n"], r["k"]) <= LINE]
    assert small and all(r["kind"] == "gemm_f64" for r in small)
    large = [r for r in rec if r["kind"] in ("gemm_tc", "gemm_f64") and r not in small]
    assert sum(r["depth"] == 0 for r in large) == 6
    return X, info, [sum(r["kind"] == "gemm_tc" and (r["depth"] == 0 or not top) for r in large)
                     for top in (True, False)], len(large)


@pytest.mark.parametrize("family", ["spd", "sdd"])
def test_as_accurate_as_the_fp64_kernel(spin, family):
    A = (inputs.spd_gram_device(N, 5, "cuda:0", alpha=0.3) if family == "spd" else inputs.sdd_device(N, 6, "cuda:0"))
    X, info, (top, count), large = products_by_residues(spin, A)
    assert info["status"] == 0 and top == 6
    assert count == large or family == "sdd"  # a diagonally dominant inverse's short products are refused
    Y, _ = fp64_kernel_inverse(spin, A)
    assert not torch.equal(X, Y)  # another rounding, so the other form did run
    Ah, Xh, Yh = A.cpu().numpy(), X.cpu().numpy(), Y.cpu().numpy()
    ref, _ = oracle.strassen_inv(Ah, LEAF)
    assert bounds.elementwise_ok(Xh, ref, Ah)
    rx, ry = oracle.residual(Ah, Xh)[0], oracle.residual(Ah, Yh)[0]
    assert rx <= 1e-13 and rx <= 1.5 * ry


def test_same_bits_on_one_stream_and_in_panels(spin):
    """The same products on one or two streams, and in an arena a caller's
    workspace leaves (several panels)."""
    A = inputs.spd_gram_device(N, 7, "cuda:0", alpha=0.5)
    X, _, _, large = products_by_residues(spin, A)
    Y, _, _, _ = products_by_residues(spin, A, schedule="lockstep")
    assert torch.equal(X, Y)
    ws = torch.empty(spin.workspace_bytes(N, leaf=LEAF) + (400 << 20), dtype=torch.uint8, device="cuda:0")
    Z, _, (_, count), _ = products_by_residues(spin, A, workspace=ws)
    assert count == large and torch.equal(X, Z)


def test_widely_spread_operands_keep_the_fp64_kernel(spin):
    """Rows and columns scaled by powers of two over a range of 2^80: fixed
    point relative to the largest entry would lose the small ones."""
    A = inputs.spd_gram_device(N, 8, "cuda:0", alpha=0.5)
    g = torch.Generator(device="cuda:0").manual_seed(3)
    d = torch.exp2(torch.randint(-40, 41, (N,), generator=g, device="cuda:0").double())
    A = (A * d[:, None]) * d[None, :]
    X, info, (_, count), _ = products_by_residues(spin, A)
    assert info["status"] == 0 and count == 0
    Y, _ = fp64_kernel_inverse(spin, A)
    assert torch.equal(X, Y)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_non_finite_entries(spin, bad):
    A = inputs.spd_gram_device(N, 9, "cuda:0", alpha=0.5)
    A[17, N - 5] = bad
    X, info, _, _ = products_by_residues(spin, A, check=False)
    Y, info2 = fp64_kernel_inverse(spin, A, check=False)
    assert info["status"] == info2["status"] == 2
    assert (info["fail_leaf"], info["fail_col"]) == (info2["fail_leaf"], info2["fail_col"])


def test_entries_just_below_a_power_of_two(spin):
    """Positive entries within 8 units of their last place below the power of
    two that bounds their row (column): the largest 63-bit integers."""
    g = torch.Generator(device="cuda:0").manual_seed(11)
    A = torch.rand((N, N), generator=g, dtype=torch.float64, device="cuda:0").mul_(2.0).sub_(1.0)
    A.diagonal().add_(200.0)
    for j in range(1, 10):
        x = 1.0 - j * 2.0 ** -53
        A[2200 + 64 * j, 7 * j] = x
        A[2210 + 64 * j, 7 * j] = -x
        A[9 * j, 2300 + 32 * j] = x
        A[9 * j, 2310 + 32 * j] = -x
    X, info, (top, _), _ = products_by_residues(spin, A)
    assert info["status"] == 0 and top == 6
    Y, _ = fp64_kernel_inverse(spin, A)
    assert not torch.equal(X, Y)
    assert bounds.elementwise_ok(X.cpu().numpy(), Y.cpu().numpy(), A.cpu().numpy())
