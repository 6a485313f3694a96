"""Tau-leaping draws at the edges of the two-phase sampler: lambda at and around
10, draws that need many blocks or rounds, lambda far beyond 2^22 (64-bit
counts), zero and negative-free channels, sixteen channels, 1024 samples and
every block size.  Exact agreement with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_bf16", "rn"), ("uniform_bf16", "sr"), ("mixed_f16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def both(ssa, md, x0, n, t_end, tau, samples, prec, rnd, seed=1, state_bytes=4):
    g = ssa.tau_run(ssa.Model.from_dict(md), n, x0, t_end, tau, samples, prec, rnd, False, seed, state_bytes)
    torch.cuda.synchronize()
    o = oracle.tau_run(md, x0, n, t_end, tau, samples, precision=prec, rounding=rnd, seed=seed, state_bytes=state_bytes)
    for k, v in g.items():
        np.testing.assert_array_equal(v.cpu().numpy().view(np.uint8), np.ascontiguousarray(o[k]).view(np.uint8))


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("lam", [1e-6, 0.5, 9.0, 9.999, 10.0, 10.001, 12.0, 40.0, 1000.0, 2.0**21, 2.0**23, 1e12, 1e20])
def test_one_channel(ssa, prec, rnd, lam):
    md = {"order": np.array([[0]], np.int32), "stoich": np.array([[1]], np.int32), "rate": np.array([lam])}
    both(ssa, md, [0], 1000, 3.0, 1.0, [0.0, 1.0, 3.0], prec, rnd)
    bd = P.birth_death(lam, 0.5)         # compiled structure: birth lambda, death lambda from the count
    both(ssa, bd, [25], 333, 4.0, 1.0, [2.0, 4.0], prec, rnd, seed=2)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_sixteen_channels_and_many_samples(ssa, prec, rnd):
    rate = np.array([0.0, 1e-3, 0.3, 2.0, 5.0, 8.0, 9.99, 10.0, 11.0, 15.0, 25.0, 60.0, 200.0, 1e3, 1e5, 1e7])
    order = np.zeros((16, 8), np.int32)
    order[1::2, 0] = 1
    stoich = np.zeros((16, 8), np.int32)
    for j in range(16):
        stoich[j, j % 8] = 1 if j % 3 else -1
    md = {"order": order, "stoich": stoich, "rate": rate}
    both(ssa, md, [1, 2, 3, 4, 5, 6, 7, 8], 100, 2.0, 0.25, P.even_samples(2.0, 1024), prec, rnd, seed=3)


@pytest.mark.parametrize("block", [32, 96, 256])
def test_block_sizes(ssa, block):
    ssa.set_launch_config(block, 0, 16)
    try:
        m = P.schlogl()
        both(ssa, P.repressilator(), P.REPRESSILATOR_X0, 301, 2.0, 0.02, [1.0, 2.0], "fp64", "rn", seed=4)
        both(ssa, P.repressilator(h=3), P.REPRESSILATOR_X0, 301, 2.0, 0.02, [1.0, 2.0], "mixed_f16", "sr", seed=4)
    finally:
        ssa.set_launch_config()


@pytest.mark.parametrize("lam", [10.0, 11.3, 14.0, 20.0, 47.0, 150.0, 1000.0, 1999.0, 2500.0])
def test_many_draws_of_the_rejection_method(ssa, lam):
    # every acceptance decision of 2^18 draws: the approximate test must never
    # decide differently from the contract's
    md = {"order": np.array([[0]], np.int32), "stoich": np.array([[1]], np.int32), "rate": np.array([lam])}
    both(ssa, md, [0], 2**16, 4.0, 1.0, [1.0, 2.0, 3.0, 4.0], "fp32", "rn", seed=9)
