"""Gradients and steps after earlier ones: the buffers that the backward pass
adds to (bias gradients, loss) are cleared for every call, block by block."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ssa():
    from paper_2605_00479_gb300 import build, ssa as mod
    build.build()
    mod.lib()
    return mod


def data(rows, seed):
    rng = np.random.default_rng(seed)
    f = rng.uniform(-1, 1, size=(rows, 4)).astype(np.float32)
    t = rng.random((rows, 128)) ** 8
    t = (t / t.sum(axis=1, keepdims=True)).astype(np.float32)
    return f, t, torch.from_numpy(f).cuda(), torch.from_numpy(t).cuda()


def blocks(theta):
    at = 0
    for name, shape in mlp.SHAPES:
        n = int(np.prod(shape))
        yield name, np.asarray(theta[at:at + n])
        at += n


def bias_allowance(theta, f, t):
    """Twice what one fp32 sum over the rows may be off, for each bias: B
    additions of 2^-23 of the terms' sizes; again twice, because the terms of
    the binary64 oracle may differ from the kernel's by a flipped bf16."""
    tr = {}
    mlp.loss_and_grad(theta.astype(np.float64), f.astype(np.float64), t.astype(np.float64), bf16=True, trace=tr)
    return {f"b{l}": 4 * f.shape[0] * 2.0**-23 * np.abs(tr[f"dz{l}"]).sum(axis=0) for l in (1, 2, 3, 4)}


def same_gradient(g, ref, allow):
    """Weight gradients are formed without atomics: the same bits.  Bias
    gradients are added up in any order."""
    for (name, a), (_, b) in zip(blocks(g), blocks(ref)):
        if name.startswith("W"):
            np.testing.assert_array_equal(a.view(np.uint32), b.view(np.uint32), err_msg=name)
        else:
            d = np.abs(a.astype(np.float64) - b.astype(np.float64))
            assert np.all(d <= allow[name]), (name, float((d / allow[name]).max()))


@pytest.mark.parametrize("B", [1, 9, 300])
def test_gradients_after_earlier_passes(ssa, B):
    f, t, fd, td = data(B, B)
    _, _, f2, t2 = data(300, 77)
    net = ssa.Surrogate(300, seed=5)
    theta = net.get_params()
    allow = bias_allowance(theta, f, t)
    loss, ref = net.gradients(fd, td)
    tol = 2 * (B + 8) * 2.0**-23 * loss
    again, g = net.gradients(fd, td)
    same_gradient(g, ref, allow)
    assert abs(again - loss) <= tol
    net.gradients(f2, t2)
    net.train_step(f2, t2, 1e-2)
    net.set_params(theta)
    again, g = net.gradients(fd, td)
    same_gradient(g, ref, allow)
    assert abs(again - loss) <= tol
    net.train(f2, t2, 3, 200, 1e-2, 1e-3)
    net.predict(f2)
    net.set_params(theta)
    again, g = net.gradients(fd, td)
    same_gradient(g, ref, allow)
    assert abs(again - loss) <= tol
    net.status()


@pytest.mark.parametrize("rows,batch", [(1, 1), (5, 7), (64, 8)])
def test_training_run_is_the_single_steps(ssa, rows, batch):
    """Up to eight rows every sum has one order (zeros apart), so nothing may differ."""
    _, _, f, t = data(rows, rows + 1)
    a, b = ssa.Surrogate(batch, seed=3), ssa.Surrogate(batch, seed=3)
    a.train(f, t, 4, batch, 1e-3, 1e-3)
    for k in range(4):
        idx = (k * batch + torch.arange(batch, device="cuda")) % rows
        b.train_step(f[idx].contiguous(), t[idx].contiguous(), 1e-3)
    torch.cuda.synchronize()
    for (name, x), (_, y) in zip(blocks(a.get_params()), blocks(b.get_params())):
        np.testing.assert_array_equal(x, y, err_msg=name)
    for x, y in zip(a.get_state()[1:4], b.get_state()[1:4]):
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("rows,batch", [(100, 250), (300, 257), (2048, 1024)])
def test_first_step_of_a_training_run(ssa, rows, batch):
    """Larger batches: the weights after one step have the same bits, the bias
    gradients agree within their sums' rounding."""
    f, t, fd, td = data(rows, rows + 2)
    idx = np.arange(batch) % rows
    a, b = ssa.Surrogate(batch, seed=4), ssa.Surrogate(batch, seed=4)
    allow = bias_allowance(a.get_params(), f[idx], t[idx])
    a.train(fd, td, 1, batch, 1e-3, 1e-3)
    b.train_step(fd[idx].contiguous(), td[idx].contiguous(), 1e-3)
    torch.cuda.synchronize()
    for (name, x), (_, y) in zip(blocks(a.get_params()), blocks(b.get_params())):
        if name.startswith("W"):
            np.testing.assert_array_equal(x, y, err_msg=name)
    same_gradient(a.get_state()[3], b.get_state()[3], allow)
