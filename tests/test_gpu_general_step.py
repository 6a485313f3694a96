"""Networks without a compiled structure at the edges of their step: reservoirs
folded and not, counts of reservoirs beyond 2^24, counts around 2^23, jumps that
take a count negative, changes of more than 1024, Hill laws of every exponent,
eight species and sixteen reactions, event caps, int16 storage and species
masks, split scheduling.  Exact agreement with the oracle."""
import numpy as np
import pytest

import oracle

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


def net(order, stoich, rate, hill=None, constant=None):
    order = np.asarray(order, np.int32)
    law = np.zeros(len(order), np.int32)
    if hill is not None:
        law = np.array([1 if h else 0 for h in hill], np.int32)
        hill = np.array([h if h else [0, 0, 1, 0] for h in hill], np.float64)
    return {"order": order, "stoich": np.asarray(stoich, np.int32), "rate": np.asarray(rate, np.float64), "law": law,
            "hill": hill, "constant": None if constant is None else np.asarray(constant, np.uint8)}


def both(ssa, md, x0, n, t_end, samples, prec, rnd, norm=False, seed=3, cap=3000, state_bytes=4, mask=0):
    m = ssa.Model.from_dict(md)
    assert m.family == "general"
    g = ssa.ensemble_run(m, n, x0, t_end, samples, prec, rnd, norm, seed, cap, state_bytes, out_species=mask)
    torch.cuda.synchronize()
    o = oracle.run(md, x0, n, t_end, samples, prec, rnd, norm, seed, cap, state_bytes, out_species=mask)
    g = {k: v.cpu().numpy() for k, v in g.items()}
    np.testing.assert_array_equal(g["snapshots"], o["snapshots"])
    np.testing.assert_array_equal(g["status"].view(np.uint32), o["status"])
    np.testing.assert_array_equal(g["n_events"], o["n_events"])
    gt, ot = g["t_final"], o["t_final"]
    ok = ~(np.isnan(gt) & np.isnan(ot))
    np.testing.assert_array_equal(gt.view(np.uint64)[ok], ot.view(np.uint64)[ok])
    return o


EXCHANGE = net([[1, 0, 1], [2, 0, 0], [0, 1, 0], [0, 3, 0], [0, 0, 0], [1, 0, 0]],
               [[1, 0, -1], [-2, 1, 0], [1, -1, 0], [0, -3, 0], [0, 1, 0], [-1, 0, 0]],
               [0.02, 0.01, 0.5, 0.001, 2.0, 0.1], constant=[0, 0, 1])


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("z", [50, 40000, 2**24 + 3, 2**31 - 1])
def test_reservoir(ssa, prec, rnd, norm, z):
    md = dict(EXCHANGE, rate=np.array([1.0 / z, 0.01, 0.5, 0.001, 2.0, 0.1]))
    both(ssa, md, [10, 5, z], 70, 4.0, [0.0, 1.0, 4.0], prec, rnd, norm, mask=5)
    both(ssa, md, [10, 5, z], 70, 4.0, [0.0, 1.0, 4.0], prec, rnd, norm, state_bytes=2)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_negative_counts_and_large_changes(ssa, prec, rnd):
    md = net([[1], [0]], [[-3], [1]], [1.0, 2.0])          # fires at x >= 1, takes 3
    o = both(ssa, md, [20], 90, 30.0, [1.0, 5.0, 30.0], prec, rnd)
    assert np.any(o["status"] & 4)
    md = net([[0], [1]], [[1500], [-1]], [1.0, 0.5])
    both(ssa, md, [10], 60, 4.0, [2.0, 4.0], prec, rnd)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("x0", [2**23 - 20, 2**23 + 5, 2**24 + 1])
def test_counts_around_the_float_range(ssa, prec, rnd, x0):
    md = net([[0, 0], [1, 0]], [[1, 1], [-1, 0]], [2.0 * x0, 1.0])
    both(ssa, md, [x0, 7], 40, 1.0, [1e-6, 1.0], prec, rnd, cap=333)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("h", [1, 2, 3, 4])
@pytest.mark.parametrize("alpha", [0.0, 30.0, 1e11])
def test_hill_laws(ssa, prec, rnd, h, alpha):
    md = net([[0, 0], [1, 0], [0, 0], [0, 1]], [[1, 0], [-1, 0], [0, 1], [0, -1]], [1.0, 1.0, 1.0, 1.0],
             hill=[[1.0, alpha, h, 1], None, [0.5, 20.0, 5 - h, 0], None])
    both(ssa, md, [4, 300], 64, 2.0, [1.0, 2.0], prec, rnd, cap=700)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("cap", [0, 1, 65, 3000])
def test_largest_network(ssa, prec, rnd, cap):
    rng = np.random.default_rng(1)
    order = np.zeros((16, 8), np.int32)
    stoich = np.zeros((16, 8), np.int32)
    for j in range(16):
        i, k = j % 8, (3 * j + 1) % 8
        if j < 8:
            stoich[j, i] = 1
        else:
            order[j, i] = 1 + j % 3
            order[j, k] = max(order[j, k], 1)
            stoich[j, i] -= 1
            stoich[j, (i + 1) % 8] += 1
    rate = np.concatenate([rng.uniform(1.0, 8.0, 8), rng.uniform(1e-3, 1e-1, 8)])
    both(ssa, net(order, stoich, rate), [3, 0, 9, 1, 4, 2, 0, 6], 50, 6.0, np.linspace(0, 6, 40), prec, rnd, cap=cap)


def test_split_scheduling(ssa):
    ssa.set_longest_first(2, 64)
    try:
        for prec, rnd in MODES[1:6]:
            both(ssa, EXCHANGE, [10, 5, 50], 1000, 20.0, [5.0, 20.0], prec, rnd, True)
    finally:
        ssa.set_longest_first()
