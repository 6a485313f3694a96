"""RDME events of the compiled structures at the edges of their domain: odd event
caps, propensity sums outside the fast division's range, counts beyond 2^24,
Hill amplitudes far from 1, constants that overflow binary16, one voxel, two
voxels (a hop between siblings), odd extents, 257 voxels, samples at 0.  Exact
agreement with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "sr"), ("uniform_f16", "rn"),
         ("uniform_f16", "sr"), ("uniform_bf16", "rn"), ("uniform_bf16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def both(ssa, md, dims, D, x0, n, t_end, samples, prec, rnd, norm=False, seed=5, cap=2000, state_bytes=4):
    S = int(np.prod(dims))
    x0 = np.ascontiguousarray(np.broadcast_to(np.asarray(x0, np.int32), (S, md["order"].shape[1])))
    g = ssa.rdme_run(ssa.Model.from_dict(md), dims, D, x0, n, t_end, samples, prec, rnd, norm, seed, cap, state_bytes)
    torch.cuda.synchronize()
    o = oracle.rdme_run(md, dims, D, x0, n, t_end, samples, precision=prec, rounding=rnd, normalise=norm, seed=seed,
                        max_events=cap, state_bytes=state_bytes)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    np.testing.assert_array_equal(g["snapshots"], o["snapshots"])
    np.testing.assert_array_equal(g["status"].view(np.uint32), o["status"])
    np.testing.assert_array_equal(g["n_events"], o["n_events"])
    gt, ot = g["t_final"], o["t_final"]
    ok = ~(np.isnan(gt) & np.isnan(ot))
    np.testing.assert_array_equal(gt.view(np.uint64)[ok], ot.view(np.uint64)[ok])


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("cap", [0, 1, 7, 8, 9, 501])
def test_event_caps(ssa, prec, rnd, cap):
    both(ssa, P.dimer(), (3, 2), [0.5, 0.2], [40, 3], 45, 4.0, [0.0, 1.0, 4.0], prec, rnd, cap=cap)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("dims", [(1,), (2,), (3,), (5, 3), (257,)])
def test_lattice_shapes(ssa, prec, rnd, dims):
    m = P.schlogl()
    if prec == "fp64" and dims == (257,):   # 1024 binary64 nodes a lane: beyond shared memory, refused
        with pytest.raises(ssa.SSAError, match="does not fit in shared memory"):
            both(ssa, m, dims, [2.0, 0.0, 0.0], P.schlogl_x0(m), 40, 0.02, [0.01, 0.02], prec, rnd, True, cap=600)
        return
    both(ssa, m, dims, [2.0, 0.0, 0.0], P.schlogl_x0(m), 40, 0.02, [0.01, 0.02], prec, rnd, True, cap=600)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("rate", [2.0**-95, 2.0**-91, 1e-20, 2.0**88, 2.0**91, 1e38])
def test_propensity_sums_at_the_division_bounds(ssa, prec, rnd, rate):
    both(ssa, P.birth_death(rate, rate), (4,), [rate], [2], 40, 4.0 / rate, [0.0, 1.0 / rate, 4.0 / rate], prec, rnd,
         cap=150)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("x0", [0, 1, 2**23, 2**24 + 1])
def test_counts(ssa, prec, rnd, x0):
    both(ssa, P.birth_death(x0 + 1.0, 1.0), (4,), [0.7], [x0], 40, 1.0, [1e-6, 1.0], prec, rnd, cap=150)
    both(ssa, P.dimer(2e5, 1e5), (2, 2), [1e4, 1e4], [min(x0, 3), 1], 40, 1e-4, [1e-4], prec, rnd, cap=150)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("alpha", [0.0, 1e-12, 216.0, 1e12])
def test_hill_amplitudes(ssa, prec, rnd, alpha):
    md = P.repressilator(alpha=alpha)
    both(ssa, md, (2, 1, 2), [0.3, 0, 0, 0.1, 0, 0], [3, 0, 2, 5, 300, 2000], 40, 0.5, [0.3, 0.5], prec, rnd, cap=300)
    m = P.schlogl()     # reservoirs not folded: 1e5 overflows binary16
    both(ssa, m, (2,), [1.0, 0, 0], P.schlogl_x0(m), 40, 0.02, [0.02], prec, rnd, cap=200)
