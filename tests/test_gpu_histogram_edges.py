"""Ensemble histograms at the edges of their kernels: unaligned views, counts
fewer than a load, one bin, the last shared and first global bin count, all
counts equal, series longer than the shared counters, one and two samples."""
import numpy as np
import pytest

from oracle import stats as ost

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


@pytest.mark.parametrize("dtype", [np.int32, np.int16])
@pytest.mark.parametrize("bins", [1, 2, 512, 8192, 8193])
@pytest.mark.parametrize("n", [1, 3, 7, 8, 9, 4097, 65535, 65536, 1000003])
@pytest.mark.parametrize("skip", [0, 1, 3, 7])
def test_count_histogram(ssa, dtype, bins, n, skip):
    rng = np.random.default_rng(n + bins + skip)
    v = rng.integers(-3, bins + 3, size=n + skip).astype(dtype)
    if n == 4097:
        v[:] = bins // 2
    h, c = ssa.count_histogram(torch.from_numpy(v).cuda()[skip:], bins)
    o, oc = ost.count_histogram(v[skip:], bins)
    np.testing.assert_array_equal(h.cpu().numpy(), o)
    assert int(c.item()) == oc


@pytest.mark.parametrize("dtype", [np.int32, np.int16])
@pytest.mark.parametrize("K,n", [(1, 5), (2, 33), (9, 600), (10, 1), (101, 70001), (8192, 40), (9000, 40)])
def test_dwell_histogram(ssa, dtype, K, n):
    rng = np.random.default_rng(K + n)
    s = ((rng.random((K, 2, n)) < 0.3).cumsum(axis=0) % 2).astype(dtype)
    h = ssa.dwell_histogram(torch.from_numpy(s).cuda(), 1).cpu().numpy()
    want = np.zeros(K, np.int64)
    for j in range(n if n < 2000 else 0):
        x, start = s[:, 1, j] != 0, -1
        for k in range(1, K):
            if x[k] and not x[k - 1]:
                start = k
            elif not x[k] and x[k - 1] and start >= 0:
                want[k - start] += 1
                start = -1
    if n >= 2000:
        x = s[:, 1, :] != 0
        start = np.full(n, -1)
        for k in range(1, K):
            ends = ~x[k] & x[k - 1] & (start >= 0)
            np.add.at(want, k - start[ends], 1)
            start[ends] = -1
            start[x[k] & ~x[k - 1]] = k
    np.testing.assert_array_equal(h, want)
