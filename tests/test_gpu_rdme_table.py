"""Voxel sums from the table and from the chains: counts on both sides of the
table's last row (4095) that cross it both ways in one trajectory, voxels that
start on both sides, beside empty ones.  Exact agreement with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "rn"), ("uniform_f16", "rn"),
         ("uniform_bf16", "rn"), ("mixed_bf16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def both(ssa, md, dims, D, x0, n, t_end, samples, prec, rnd, norm=False, cap=2000):
    g = ssa.rdme_run(ssa.Model.from_dict(md), dims, D, x0, n, t_end, samples, prec, rnd, norm, 5, cap)
    torch.cuda.synchronize()
    o = oracle.rdme_run(md, dims, D, x0, n, t_end, samples, precision=prec, rounding=rnd, normalise=norm, seed=5,
                        max_events=cap)
    np.testing.assert_array_equal(g["snapshots"].cpu().numpy(), o["snapshots"])
    np.testing.assert_array_equal(g["status"].cpu().numpy().view(np.uint32), o["status"])
    np.testing.assert_array_equal(g["n_events"].cpu().numpy(), o["n_events"])
    return o["snapshots"]


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("x0", [4094, 4095, 4096, 4097])
def test_counts_around_the_last_row(ssa, prec, rnd, x0):
    # about 600 events: birth and death in balance, hops between four voxels
    lat = np.full((4, 1), x0, np.int32)
    s = both(ssa, P.birth_death(float(x0), 1.0), (2, 2), [0.05], lat, 48, 0.016, np.linspace(0, 0.016, 9), prec, rnd)
    if prec in ("fp64", "fp32"):
        assert s.min() < 4096 <= s.max()
    m = P.schlogl()
    lat = np.tile(np.array([x0, 100000, 200000], np.int32), (2, 1))
    both(ssa, m, (2,), [0.5, 0.0, 0.0], lat, 32, 2e-4, [1e-4, 2e-4], prec, rnd, True)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_voxels_on_both_sides(ssa, prec, rnd):
    lat = np.array([[0], [4090], [4095], [4096], [4100], [20000]], np.int32)
    both(ssa, P.birth_death(4096.0, 1.0), (3, 2), [0.4], lat, 48, 0.02, [0.01, 0.02], prec, rnd)
