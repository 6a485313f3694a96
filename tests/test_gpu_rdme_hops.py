"""Lattices where some species of several hop: the destination and the species of
a hop are found from one channel number, for every subset of hopping species and
for voxels with one to six neighbours.  Exact agreement with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("mixed_f16", "rn"), ("uniform_bf16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    mod.lib()
    return mod


def both(ssa, md, dims, D, x0, prec, rnd, fold=False):
    lat = np.tile(np.asarray(x0, np.int32), (int(np.prod(dims)), 1))
    lat[::2] += np.asarray(D, np.float64)[None, :].astype(bool).astype(np.int32)   # not the same everywhere
    kw = dict(normalise=fold, seed=13, max_events=400)
    g = ssa.rdme_run(ssa.Model.from_dict(md), dims, D, lat, 45, 2.0, [0.5, 2.0], prec, rnd, **kw)
    torch.cuda.synchronize()
    o = oracle.rdme_run(md, dims, D, lat, 45, 2.0, [0.5, 2.0], precision=prec, rounding=rnd, **kw)
    for k in ("snapshots", "n_events"):
        np.testing.assert_array_equal(g[k].cpu().numpy(), o[k])
    np.testing.assert_array_equal(g["status"].cpu().numpy().view(np.uint32), o["status"])


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("dims", [(2,), (3, 2), (3, 3, 3)])
@pytest.mark.parametrize("hopping", [1, 2, 3, 4, 5, 6, 7])
def test_subsets_of_three_species(ssa, prec, rnd, dims, hopping):
    D = [0.7 * (i + 1) if (hopping >> i) & 1 else 0.0 for i in range(3)]
    both(ssa, P.telegraph(0.5, 0.5, 20.0, 1.0), dims, D, P.TELEGRAPH_X0, prec, rnd)


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("D", [[0, 0, 0, 0, 0, 2.0], [0.3, 0, 0.2, 0, 0, 0.1], [0.5] * 6])
def test_six_species(ssa, prec, rnd, D):
    both(ssa, P.repressilator(), (3, 3), D, P.REPRESSILATOR_X0, prec, rnd)


@pytest.mark.parametrize("prec,rnd", MODES)
def test_one_moving_species_between_held_ones(ssa, prec, rnd):
    m = P.schlogl()
    D = [0.0 if c else 1.5 for c in m["constant"]]
    both(ssa, m, (2, 2, 2), D, P.schlogl_x0(m), prec, rnd, True)
