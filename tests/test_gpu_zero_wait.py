"""A first uniform of exactly 1 (all 32 bits of the word set), so that the waiting
time is zero: the event fires at time zero and the snapshot there shows it.  One in
2^32 trajectories of a seed starts so; these two of seed 1 do."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "sr"), ("uniform_f16", "rn"), ("uniform_bf16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    mod.lib()
    return mod


def same(g, o):
    torch.cuda.synchronize()
    for k in ("snapshots", "n_events"):
        np.testing.assert_array_equal(g[k].cpu().numpy(), o[k])
    np.testing.assert_array_equal(g["t_final"].cpu().numpy().view(np.uint64), o["t_final"].view(np.uint64))


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("traj", [1205451635, 1348758320])
@pytest.mark.parametrize("net", ["birth_death", "general", "lattice"])
def test_event_at_time_zero(ssa, prec, rnd, traj, net):
    assert int(oracle.philox((0, 0, traj, 0), (1, 0)).reshape(-1)[0]) == 0xFFFFFFFF
    md = P.repressilator(h=3) if net == "general" else P.birth_death(10.0, 0.5)
    x0 = list(P.REPRESSILATOR_X0) if net == "general" else [4]
    m = ssa.Model.from_dict(md)
    for cap in (1, 50):
        kw = dict(normalise=False, seed=1, max_events=cap)
        first = traj - 3
        if net == "lattice":
            lat = np.array([[4], [3]], np.int32)
            same(ssa.rdme_run(m, (2,), [1.0], lat, 33, 2.0, [0.0, 1.0], prec, rnd, traj_offset=first, **kw),
                 oracle.rdme_run(md, (2,), [1.0], lat, 33, 2.0, [0.0, 1.0], precision=prec, rounding=rnd, g0=first,
                                 **kw))
        else:
            same(ssa.ensemble_run(m, 33, x0, 2.0, [0.0, 1.0], prec, rnd, traj_offset=first, **kw),
                 oracle.run(md, x0, 33, 2.0, [0.0, 1.0], prec, rnd, g0=first, **kw))
