"""Calls from several host threads that need different amounts of shared memory
of the same kernel: none may fail, and each gives what it gives alone."""
import threading

import numpy as np
import pytest

from paper_2605_00479_gb300 import presets as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    mod.lib()
    return mod


def together(jobs):
    """Each job in a thread of its own, on a stream of its own, started at once."""
    errors, gate = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                gate.wait()
                job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:   # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("net", ["schlogl", "general"])
def test_lattices_of_different_sizes(ssa, net):
    if net == "schlogl":
        md, x0, fold = P.schlogl(), P.schlogl_x0(P.schlogl()), True
    else:
        md, x0, fold = P.repressilator(h=3), P.REPRESSILATOR_X0, False
    m = ssa.Model.from_dict(md)
    D = [0.5] + [0.0] * (m.N - 1)

    def run(voxels):
        lat = np.tile(np.asarray(x0, np.int32), (voxels, 1))
        return ssa.rdme_run(m, (voxels,), D, lat, 32, 0.01, [0.01], "mixed_bf16", "rn", fold, 5, max_events=40)

    sizes = (1, 32)
    alone = [run(v) for v in sizes]
    torch.cuda.synchronize()

    def many(i):
        for _ in range(200):
            g = run(sizes[i])
        torch.cuda.current_stream().synchronize()
        assert torch.equal(g["snapshots"], alone[i]["snapshots"])

    together([lambda: many(0), lambda: many(1)])


def test_surrogates_of_different_batches(ssa):
    sizes = (1, 4096)
    nets = [ssa.Surrogate(b, seed=1) for b in sizes]
    rng = np.random.default_rng(0)
    feats = [torch.from_numpy(rng.uniform(-1, 1, (b, 4)).astype(np.float32)).cuda() for b in sizes]
    alone = [n.predict(f) for n, f in zip(nets, feats)]
    targets = [a.clone() for a in alone]
    torch.cuda.synchronize()

    def many(i):
        for _ in range(200):
            got = nets[i].predict(feats[i])
            nets[i].train_step(feats[i], targets[i], 0.0, weight_decay=0.0)
        torch.cuda.current_stream().synchronize()
        assert torch.equal(got, alone[i])
        nets[i].status()

    together([lambda: many(0), lambda: many(1)])
