"""A network runs on a compiled structure only where every table agrees with it:
each change vector entry of each reaction (Hill rows too), each reactant order,
each law, Hill exponent, regulator and held species.  Anything else is general."""
import numpy as np
import pytest

from paper_2605_00479_gb300 import presets as P

NETWORKS = {"birth_death": P.birth_death, "schlogl": P.schlogl, "telegraph": P.telegraph, "dimer": P.dimer,
            "repressilator": P.repressilator}


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    return mod


@pytest.mark.parametrize("name", sorted(NETWORKS))
def test_every_table_entry_decides(ssa, name):
    base = NETWORKS[name]()
    assert ssa.Model.from_dict(base).family == name
    M, N = base["order"].shape
    held = np.zeros(N) if base["constant"] is None else base["constant"]
    for j in range(M):
        for i in range(N):
            m = {**base, "stoich": base["stoich"].copy()}
            m["stoich"][j, i] += 1
            # the change of a held species is never applied: it does not matter
            assert ssa.Model.from_dict(m).family == (name if held[i] else "general"), ("stoich", j, i)
            if base["law"][j] == P.MASS_ACTION:
                m = {**base, "order": base["order"].copy()}
                m["order"][j, i] = (m["order"][j, i] + 1) % 4
                assert ssa.Model.from_dict(m).family == "general", ("order", j, i)
    for i in range(N):
        c = held.astype(np.uint8).copy()
        c[i] ^= 1
        assert ssa.Model.from_dict({**base, "constant": c}).family == "general"


@pytest.mark.gpu
@pytest.mark.parametrize("prec,rnd", [("fp64", "rn"), ("fp32", "rn"), ("mixed_f16", "sr"), ("uniform_bf16", "sr")])
def test_transcription_bursts(ssa, prec, rnd):
    import oracle
    torch = pytest.importorskip("torch")
    md = P.repressilator()
    md["stoich"] = md["stoich"].copy()
    md["stoich"][[0, 4, 8], [0, 1, 2]] = 3      # three mRNAs a transcription
    smp = P.even_samples(2.0, 5)
    g = ssa.ensemble_run(ssa.Model.from_dict(md), 70, P.REPRESSILATOR_X0, 2.0, smp, prec, rnd, False, 3, 5000)
    torch.cuda.synchronize()
    o = oracle.run(md, P.REPRESSILATOR_X0, 70, 2.0, smp, prec, rnd, False, 3, 5000)
    np.testing.assert_array_equal(g["snapshots"].cpu().numpy(), o["snapshots"])
    np.testing.assert_array_equal(g["n_events"].cpu().numpy(), o["n_events"])
