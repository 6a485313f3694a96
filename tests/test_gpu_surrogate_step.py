"""The surrogate's device-driven training at the edges of its kernels: batches of
one row, below, at and above a block's rows, not a multiple of the padding,
data sets smaller than the batch (rows wrap); each equal to the same steps taken
one by one.  The softmax kernel's block sums against binary64."""
import numpy as np
import pytest

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
    f = torch.from_numpy(rng.uniform(-1, 1, size=(rows, 4)).astype(np.float32)).cuda()
    t = rng.random((rows, 128)) ** 8
    return f, torch.from_numpy((t / t.sum(axis=1, keepdims=True)).astype(np.float32)).cuda()


@pytest.mark.parametrize("rows,batch", [(1, 1), (5, 7), (64, 8), (300, 257), (100, 250), (2048, 1024)])
def test_train_equals_single_steps(ssa, rows, batch):
    f, t = data(rows, rows)
    a, b = ssa.Surrogate(batch, seed=3), ssa.Surrogate(batch, seed=3)
    trace = torch.full((4,), float("nan"), device="cuda")
    a.train(f, t, 4, batch, 1e-3, 1e-3, loss_every=1, loss_trace=trace)
    losses = torch.zeros(4, device="cuda")
    for k in range(4):
        idx = (k * batch + torch.arange(batch, device="cuda")) % rows
        b.train_step(f[idx].contiguous(), t[idx].contiguous(), 1e-3, loss=losses[k:k + 1])
    torch.cuda.synchronize()
    a.status(), b.status()
    # the bias gradients and the loss are summed by fp32 atomics in any order;
    # AdamW's first steps divide them by their own size, so a bias whose
    # gradient is at rounding level may move by up to its step (4 * lr)
    # elsewhere: nothing beyond what four steps can move, and almost all equal
    ta, tb = a.get_params(), b.get_params()
    assert np.max(np.abs(ta - tb)) <= 4.2e-3
    assert np.mean(np.abs(ta - tb) <= 1e-5) >= 0.97
    np.testing.assert_allclose(trace.cpu().numpy(), losses.cpu().numpy(), rtol=1e-4)


@pytest.mark.parametrize("B", [1, 7, 8, 9, 255, 257, 1000])
def test_softmax_block_sums(ssa, B):
    rng = np.random.default_rng(B)
    z = torch.from_numpy(rng.normal(size=(B, 128)).astype(np.float32)).cuda()
    _, t = data(B, B + 1)
    dz = torch.zeros((B, 128), dtype=torch.bfloat16, device="cuda")
    bg, loss = torch.zeros(128, device="cuda"), torch.zeros(1, device="cuda")
    rc = ssa.lib().ssa_mlp_softmax_xent(B, ssa._dev_ptr(z), ssa._dev_ptr(t), None, ssa._dev_ptr(dz), ssa._dev_ptr(bg),
                                        ssa._dev_ptr(loss), None)
    assert rc == 0
    q = torch.softmax(z.double(), 1)
    d = (q - t.double()) / B
    eps = 2.0 ** -23 * (B + 200)     # one rounding an addition, softmax within a few ulp
    assert torch.all((bg.double() - d.sum(0)).abs() <= eps * d.abs().sum(0) + 1e-9)
    ce = -(t.double() * torch.log_softmax(z.double(), 1)).sum() / B
    assert abs(float(loss) - float(ce)) <= eps * float(ce) + 1e-6
    assert torch.all((dz.double() - d).abs() <= 2.0 ** -8 * d.abs() + 1e-9)
