"""The bounded exchange waits of the batched paths' leaf with its rows over a
cluster (128 < L <= 256, batches whose leaves do not fit the GPU as clusters of
columns): a CTA that sends nothing ends in a status, not in a hang, and leaves
the GPU usable."""
import time

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def spin():
    import paper_1801_04723_gb300 as s

    s.build()
    s.lib()
    return s


@pytest.mark.parametrize("L,mute", [(160, 0), (160, 1), (256, 0), (256, 3)])
def test_muted_cta_times_out(spin, L, mute):
    start = time.perf_counter()
    assert spin.batched_leaf_exchange_timeout(L, mute, 50.0) == 6
    assert time.perf_counter() - start < 2.0
    A = torch.eye(L, dtype=torch.float64, device="cuda:0") * 4.0
    X, status = spin.invert_batched([A] * 80, leaf=L, schedule="lockstep")
    torch.cuda.synchronize()
    assert status.tolist() == [0] * 80 and torch.equal(X[7], A / 16.0)


@pytest.mark.parametrize("L,mute,limit", [(1, 0, 50.0), (300, 0, 50.0), (64, 0, 50.0), (256, 4, 50.0), (256, -1, 50.0),
                                          (256, 0, 0.0), (256, 0, 5000.0)])
def test_bad_arguments(spin, L, mute, limit):
    assert spin.batched_leaf_exchange_timeout(L, mute, limit) == 1
