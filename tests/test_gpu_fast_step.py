"""The direct-method step of the compiled structures at the edges of its domain:
quotients and logarithms over many draws, propensity sums at the bounds of the
fast division, counts around 2^23, event caps around a slice, constants that
overflow the 16-bit formats, Hill amplitudes far from 1, samples at -0 and 0.
Exact agreement with the oracle (both sides round every operation identically)."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "sr"), ("uniform_f16", "rn"),
         ("uniform_f16", "sr"), ("uniform_bf16", "rn"), ("uniform_bf16", "sr"), ("uniform_f16", "sra"),
         ("uniform_bf16", "sra")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def both(ssa, md, x0, n, t_end, samples, prec, rnd, norm, seed, cap, state_bytes=4):
    m = ssa.Model.from_dict(md)
    assert m.family != "general"
    g = ssa.ensemble_run(m, n, x0, t_end, samples, prec, rnd, norm, seed, cap, state_bytes)
    torch.cuda.synchronize()
    o = oracle.run(md, x0, n, t_end, samples, prec, rnd, norm, seed, cap, state_bytes)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    np.testing.assert_array_equal(g["snapshots"], o["snapshots"])
    np.testing.assert_array_equal(g["status"].view(np.uint32), o["status"])
    np.testing.assert_array_equal(g["n_events"], o["n_events"])
    gt, ot = g["t_final"], o["t_final"]
    ok = ~(np.isnan(gt) & np.isnan(ot))
    np.testing.assert_array_equal(gt.view(np.uint64)[ok], ot.view(np.uint64)[ok])


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("k,gamma", [(1.0, 0.0), (3.0, 0.7)])
def test_first_waiting_times(ssa, prec, rnd, k, gamma):
    # a few events of many trajectories: -log u and the quotient for 2^18 draws
    both(ssa, P.birth_death(k, gamma), [1], 2**18, 1e3, [1e3], prec, rnd, False, 5, 2)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("rate", [2.0**-95, 2.0**-90, 2.0**-89, 1e-20, 2.0**60, 2.0**89, 2.0**90, 2.0**91, 1e38, 1e300])
def test_propensity_sums_at_the_division_bounds(ssa, prec, rnd, rate):
    both(ssa, P.birth_death(rate, rate), [2], 70, 8.0 / rate, [0.0, 1.0 / rate, 4.0 / rate], prec, rnd, False, 6, 300)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("x0", [2**23 - 30, 2**23 - 1, 2**23, 2**24 - 40, 2**24 + 1, 2**31 - 1])
def test_counts_around_the_float_range(ssa, prec, rnd, x0):
    both(ssa, P.birth_death(2.0 * x0, 1.0), [x0], 40, 1.0, [1e-6, 1.0], prec, rnd, False, 7, 333)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("cap", [0, 1, 2, 3, 63, 64, 65, 127, 200])
def test_event_caps_around_a_slice(ssa, prec, rnd, cap):
    both(ssa, P.dimer(), P.dimer_x0(300), 45, 50.0, P.even_samples(50.0, 7), prec, rnd, False, 8, cap)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_constants_beyond_the_16_bit_range(ssa, prec, rnd):
    # c' overflows binary16 (and 0 * inf meets counts below the order)
    both(ssa, P.dimer(2e5, 1e5), [1, 0], 40, 1e-4, [1e-4], prec, rnd, False, 9, 100)
    both(ssa, P.dimer(2e5, 1e5), [3, 2], 40, 1e-4, [1e-4], prec, rnd, False, 9, 100)
    m = P.schlogl()   # reservoirs not folded: 1e5 overflows binary16
    both(ssa, m, P.schlogl_x0(m), 40, 0.05, [0.01, 0.05], prec, rnd, False, 10, 400)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("alpha", [0.0, 1e-12, 216.0, 7e4, 1e12])
def test_hill_amplitudes(ssa, prec, rnd, alpha):
    md = P.repressilator(alpha=alpha)
    both(ssa, md, [3, 0, 2, 5, 300, 2000], 40, 1.0, [0.3, 1.0], prec, rnd, False, 11, 500)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_absorbing_state_and_samples_at_zero(ssa, prec, rnd):
    both(ssa, P.birth_death(0.0, 1.0), [3], 100, 1e4, [-0.0, 0.0, 1.0, 1e4], prec, rnd, False, 12, 1000)
    both(ssa, P.telegraph(), P.TELEGRAPH_X0, 100, 3.0, P.even_samples(3.0, 400), prec, rnd, False, 13, 3000, 2)
