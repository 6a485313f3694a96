"""Hill amplitudes of the compiled repressilator at the bounds of the fast
division (2^-60 and 2^90) and at the narrower ones it had: the direct method and
the lattice, exact agreement with the oracle."""
import numpy as np
import pytest

import oracle
from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MODES = [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "rn"), ("mixed_bf16", "sr"), ("uniform_f16", "sr"),
         ("uniform_bf16", "rn"), ("uniform_bf16", "sr")]


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    assert torch.cuda.is_available()
    mod.lib()
    return mod


def same(g, o):
    torch.cuda.synchronize()
    for k in ("snapshots", "n_events"):
        np.testing.assert_array_equal(g[k].cpu().numpy(), o[k])
    np.testing.assert_array_equal(g["status"].cpu().numpy().view(np.uint32), o["status"])


@pytest.mark.parametrize("prec,rnd", MODES)
@pytest.mark.parametrize("alpha", [0.99 * 2.0**-60, 2.0**-60, 2.0**-31, 2.0**-30, 2.0**31, 1.5 * 2.0**31, 2.0**89, 2.0**90,
                                   2.0**91])
def test_amplitudes(ssa, prec, rnd, alpha):
    md = P.repressilator(alpha0=min(0.2, alpha), alpha=alpha)
    x0 = [3, 0, 2, 0, 300, 2**22 + 5]
    t = min(1.0, 30.0 / alpha)
    m = ssa.Model.from_dict(md)
    assert m.family == "repressilator"
    same(ssa.ensemble_run(m, 40, x0, t, [0.3 * t, t], prec, rnd, False, 11, 300),
         oracle.run(md, x0, 40, t, [0.3 * t, t], prec, rnd, False, 11, 300))
    lat = np.tile(np.array([3, 0, 2, 2**31 - 900, 300, 0], np.int32), (2, 1))
    D = [0.3, 0, 0, 0.0, 0, 0]
    same(ssa.rdme_run(m, (2,), D, lat, 40, t, [t], prec, rnd, False, 11, 120),
         oracle.rdme_run(md, (2,), D, lat, 40, t, [t], precision=prec, rounding=rnd, seed=11, max_events=120))
