"""Training steps of the preconditioner's network at the edges of its blocks (128
samples, 1,024 with eight samples a lane group) and beyond one pass of the
grid, against the same steps in FP64.

Bars: a loss is a mean of FP32 squares, within 2e-5 of itself.  A step moves a
weight by lr times a ratio of order one whose relative error is that of an
FP32 gradient sum (1e-6 of its terms), so weights agree to 3e-5 (1 % of lr)
unless the terms cancel to a few parts in 1e5: two in a hundred may differ
more, none by more than the steps themselves."""
import numpy as np
import pytest

from paper_1810_03358_gb300 import learn
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


def rows_of(seed, step, batch, rows):
    """sampled rows: splitmix64 of the sample's index, scaled to the row count"""
    z = [(seed + (step * batch + 1 + k) * 0x9E3779B97F4A7C15) % 2 ** 64 for k in range(batch)]
    out = np.empty(batch, dtype=np.int64)
    for k, v in enumerate(z):
        v = ((v ^ (v >> 30)) * 0xBF58476D1CE4E5B9) % 2 ** 64
        v = ((v ^ (v >> 27)) * 0x94D049BB133111EB) % 2 ** 64
        out[k] = ((v ^ (v >> 31)) * rows) >> 64
    return out


def reference(feat, target, w0, steps, batch, lr, seed):
    f, t = torch.tensor(feat, dtype=torch.float64), torch.tensor(target, dtype=torch.float64)
    w = torch.tensor(w0, dtype=torch.float64)
    m, v, losses = torch.zeros_like(w), torch.zeros_like(w), []
    for step in range(steps):
        row = torch.tensor(rows_of(seed, step, batch, len(target)))
        y = w.clone().requires_grad_(True)
        h = torch.relu(f[row] @ y[:320].view(64, 5).T + y[320:384])
        loss = ((h @ y[384:448] + y[448] - t[row]) ** 2).mean()
        loss.backward()
        m, v = 0.9 * m + 0.1 * y.grad, 0.999 * v + 0.001 * y.grad ** 2
        w = w - lr * (m / (1 - 0.9 ** (step + 1))) / ((v / (1 - 0.999 ** (step + 1))).sqrt() + 1e-8)
        losses.append(float(loss.detach()))
    return w.numpy(), np.array(losses)


@pytest.mark.parametrize("batch", [1, 31, 127, 128, 129, 1000, 1025, 16385, 40000])
def test_steps_match_reference(ff, batch):
    rng = np.random.default_rng(batch)
    rows, steps, lr, seed = 50000, 3, 3e-3, 17
    feat = rng.normal(size=(rows, 5)).astype(np.float32)
    target = np.sin(feat.sum(axis=1)).astype(np.float32)
    w0 = learn.init_weights(5).astype(np.float32)
    dev = dict(dtype=torch.float32, device="cuda")
    w, adam = torch.tensor(w0, **dev), torch.zeros(2 * learn.N_PARAMS, **dev)
    work = torch.zeros(ff.ffmin_mlp_work_floats(), **dev)
    losses = np.asarray(ff.ffmin_mlp_train(torch.tensor(feat, **dev), torch.tensor(target, **dev), steps, batch, lr,
                                           seed, w, adam, work))
    wr, lref = reference(feat, target, w0, steps, batch, lr, seed)
    assert np.all(np.abs(losses - lref) <= 2e-5 * np.abs(lref) + 1e-9)
    d = np.abs(w.cpu().numpy() - wr)
    assert d.max() <= 2 * steps * lr
    assert np.mean(d > 3e-5) <= 0.02
