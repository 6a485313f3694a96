"""Networks without a compiled structure on either side of the rule that picks
their kernel: changes of 1024 and 1025, counts that start at 2^23 - 1 and 2^23
(moving, reactant only, held and unread), Hill amplitudes at the format's bounds,
sweeps over several parameter sets, each also split and with hand-offs that give
up.  Exact agreement with the oracle."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "sr"), ("uniform_f16", "sr"),
         ("uniform_bf16", "rn"), ("uniform_bf16", "sra")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def net(order, stoich, rate, hill=None, constant=None):
    order = np.asarray(order, np.int32)
    law = np.zeros(len(order), np.int32)
    if hill is not None:
        law = np.array([1 if h else 0 for h in hill], np.int32)
        hill = np.array([h if h else [0, 0, 1, 0] for h in hill], np.float64)
    return {"order": order, "stoich": np.asarray(stoich, np.int32), "rate": np.asarray(rate, np.float64), "law": law,
            "hill": hill, "constant": None if constant is None else np.asarray(constant, np.uint8)}


def same(g, o, cols=slice(None)):
    g = {k: v.cpu().numpy() for k, v in g.items()}
    np.testing.assert_array_equal(g["snapshots"][..., cols], o["snapshots"])
    np.testing.assert_array_equal(g["status"].view(np.uint32)[cols], o["status"])
    np.testing.assert_array_equal(g["n_events"][cols], o["n_events"])
    gt, ot = g["t_final"][cols], o["t_final"]
    ok = ~(np.isnan(gt) & np.isnan(ot))
    np.testing.assert_array_equal(gt.view(np.uint64)[ok], ot.view(np.uint64)[ok])


def both(ssa, md, x0, n, t_end, samples, prec, rnd, norm=False, cap=1500, seed=17):
    m = ssa.Model.from_dict(md)
    assert m.family == "general"
    g = ssa.ensemble_run(m, n, x0, t_end, samples, prec, rnd, norm, seed, cap)
    torch.cuda.synchronize()
    same(g, oracle.run(md, x0, n, t_end, samples, prec, rnd, norm, seed, cap))


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("jump", [1024, 1025, -1024, -1025])
def test_largest_change(ssa, prec, rnd, jump):
    md = net([[0], [1]], [[abs(jump)], [-1 if jump > 0 else jump]], [1.0, 0.2])
    both(ssa, md, [3000], 40, 3.0, [1.0, 3.0], prec, rnd)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("x0", [2**23 - 1, 2**23])
def test_first_counts(ssa, prec, rnd, x0):
    r = 2.0 / x0
    both(ssa, net([[0, 0], [1, 0]], [[1, 1], [-1, 0]], [1.0, r]), [x0, 7], 40, 60.0, [9.0, 60.0], prec, rnd)   # moves
    both(ssa, net([[1, 0], [0, 1]], [[0, 1], [0, -1]], [r, 0.5]), [x0, 7], 40, 60.0, [9.0, 60.0], prec, rnd)   # reactant
    held = net([[1, 0], [0, 1]], [[0, 1], [0, -1]], [r, 0.5], constant=[1, 0])
    both(ssa, held, [x0, 7], 40, 60.0, [9.0, 60.0], prec, rnd, norm=True)                                      # unread


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("alpha", [2.0**-30, np.nextafter(2.0**-29, 0), 2.0**-29, 65504.0, 65505.0, 65519.9, 65520.0, 2.0**30,
                                   2.0**31])
def test_hill_amplitude_bounds(ssa, prec, rnd, alpha):
    md = net([[0, 0], [1, 0], [0, 1]], [[1, 1], [-1, 0], [0, -1]], [1.0, 1.0, 1.0],
             hill=[[0.5, alpha, 4, 1], None, None])
    both(ssa, md, [4, 40], 40, min(4.0, 50.0 / alpha), [min(2.0, 20.0 / alpha)], prec, rnd, cap=400)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("split,spins", [(False, 0), (True, 0), (True, 1)])
def test_sweep_and_plain_runs(ssa, prec, rnd, split, spins):
    md = net([[1, 0, 1], [2, 0, 0], [0, 1, 0], [0, 0, 0]], [[1, 0, -1], [-2, 1, 0], [1, -1, 0], [0, 1, 0]],
             [0.02, 0.01, 0.5, 2.0], constant=[0, 0, 1])
    rates = np.ascontiguousarray(md["rate"][None, :] * np.array([[0.5], [1.0], [2.0]]))
    x0 = np.ascontiguousarray([[10, 5, 50], [0, 0, 60], [3, 1, 20]], np.int32)
    n, T, smp = 3 * 37, 37, np.array([2.0, 8.0])
    m = ssa.Model.from_dict(md)
    out = {"snapshots": torch.empty((2, 3, n), dtype=torch.int32, device="cuda"),
           "status": torch.empty(n, dtype=torch.int32, device="cuda"),
           "n_events": torch.empty(n, dtype=torch.int64, device="cuda"),
           "t_final": torch.empty(n, dtype=torch.float64, device="cuda")}
    wide = net([[0], [1]], [[1500], [-1]], [1.0, 0.5])
    try:
        if split:
            ssa.set_longest_first(2, 64)
        ssa.set_tail_lock_limit(spins)
        rc = ssa.lib().ssa_sweep_run_noalloc(
            m.handle, 3, T, ssa._np_ptr(rates), None, ssa._np_ptr(x0), 5, 8.0, 2, ssa._np_ptr(smp), ssa.PRECISION[prec],
            ssa.ROUNDING[rnd], 1, 23, 1500, 4, *[ssa._dev_ptr(out[k]) for k in ("snapshots", "status", "n_events", "t_final")],
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        torch.cuda.synchronize()
        both(ssa, wide, [10], 600, 3.0, [1.0, 3.0], prec, rnd)
    finally:
        ssa.set_longest_first()
        ssa.set_tail_lock_limit()
    for q in range(3):
        o = oracle.run(dict(md, rate=rates[q]), x0[q], T, 8.0, smp, prec, rnd, True, 23, 1500, g0=5 + q * T)
        same(out, o, slice(q * T, (q + 1) * T))
