"""The preconditioner network's training kernel in forms that a plain call on a
whole GPU does not reach: mlp.cu compiled by itself with other values of its
build-time constants.

A wait that runs out: with a single poll at the grid barrier some block gives
up within a few steps (the first cluster to arrive finds the other 15 missing),
while blocks of the same cluster that poll later see the count complete.  The
call reports the timeout, the weights are those of some step (a step moves a
weight by at most about lr), and the context still computes what it did.

Runs of several launches (more than 4,096 steps): weights, moments, the sample
stream and the bias corrections go on where the launch before ended, so the
losses and weights have the bits of one launch, and of launches of seven steps.

A grid that is not resident at once: with 64 clusters (512 blocks, of which the
SMs hold two each) the first launch is refused, and the call goes on with fewer
clusters; so it goes where a process has a share of the SMs, down to blocks
without clusters.  The gradient over all rows against FP64: a thread adds 128
rows' terms in FP32 (2,048 in the 16 blocks without clusters), the rest is a
tree, so at the worst 2^11 2^-24 = 1.2e-4 of the terms' magnitudes: a bar of 2e-4
of the largest component, where a lost block would show as 1 / 512.

The largest batch, 2^31 - 1 samples (of one row): every thread adds up 2^17 equal
terms in FP32, each addition off by at most 2^-24 of the sum, so the loss is
within 2^17 2^-24 = 1 % of the row's; the first Adam step moves a weight by lr
towards the gradient's sign, whatever its size."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_1810_03358_gb300 import build, learn
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


@pytest.fixture(scope="module")
def variant(ff, tmp_path_factory):
    """variant(FFMIN_X=1, ...) -> a train function like ffmin.ffmin_mlp_train
    that returns (status, losses), from mlp.cu with those constants"""
    def make(**macros):
        out = str(tmp_path_factory.mktemp("mlp") / "libmlp.so")
        cmd = [build.nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.ROOT + "/include", "-I",
               build.CSRC] + build.ARCH + [f"-D{k}={v}" for k, v in macros.items()] + ["-o", out, build.CSRC + "/mlp.cu"]
        subprocess.run(cmd, check=True, capture_output=True, text=True)
        L = C.CDLL(out)
        L.ffmin_mlp_train.argtypes = ff.lib().ffmin_mlp_train.argtypes

        def train(feat, target, steps, batch, lr, seed, w, adam, work):
            losses = np.zeros(max(steps, 1), dtype=np.float32)
            st = L.ffmin_mlp_train(feat.data_ptr(), target.data_ptr(), target.numel(), steps, batch, lr, seed,
                                   w.data_ptr(), adam.data_ptr(), work.data_ptr(),
                                   losses.ctypes.data_as(C.POINTER(C.c_float)), None,
                                   torch.cuda.current_stream().cuda_stream)
            return st, losses
        return train
    return make


def inputs(rows, seed=3):
    rng = np.random.default_rng(seed)
    feat = rng.normal(size=(rows, 5)).astype(np.float32)
    target = np.sin(feat.sum(axis=1)).astype(np.float32)
    dev = dict(dtype=torch.float32, device="cuda")
    return torch.tensor(feat, **dev), torch.tensor(target, **dev)


def fresh(ff):
    dev = dict(dtype=torch.float32, device="cuda")
    return (torch.tensor(learn.init_weights(5).astype(np.float32), **dev), torch.zeros(2 * learn.N_PARAMS, **dev),
            torch.zeros(ff.ffmin_mlp_work_floats(), **dev))


def test_a_wait_that_runs_out_is_reported(ff, variant):
    feat, target = inputs(50000)
    lr, steps = 3e-3, 50

    def plain():
        w, adam, work = fresh(ff)
        return ff.ffmin_mlp_train(feat, target, 5, 16384, lr, 9, w, adam, work), w.cpu().numpy()
    before = plain()
    impatient = variant(FFMIN_MLP_POLLS=1)
    for _ in range(3):
        w, adam, work = fresh(ff)
        w0 = w.cpu().numpy()
        st, _ = impatient(feat, target, steps, 16384, lr, 9, w, adam, work)
        assert st == ff.FFMIN_ERR_TIMEOUT
        assert np.abs(w.cpu().numpy() - w0).max() <= 2 * steps * lr
    after = plain()
    assert np.array_equal(before[0], after[0]) and np.array_equal(before[1], after[1])


@pytest.mark.parametrize("macros", [dict(FFMIN_MLP_CLUSTERS=64), dict(FFMIN_MLP_CLUSTER=1)])
def test_other_grids(ff, variant, macros):
    feat, target = inputs(1 << 17)
    w, adam, work = fresh(ff)
    w[384:448] = 0.1
    y = w.double().requires_grad_(True)
    h = torch.relu(feat.double() @ y[:320].view(64, 5).T + y[320:384])
    loss = ((h @ y[384:448] + y[448] - target.double()) ** 2).mean()
    loss.backward()
    st, got = variant(**macros)(feat, target, 0, 1 << 17, 0.0, 0, w, adam, work)
    assert st == ff.FFMIN_OK
    assert abs(got[0] - float(loss.detach())) <= 2e-4 * float(loss.detach())
    g = work[-learn.N_PARAMS:].double()
    assert (g - y.grad).abs().max() <= 2e-4 * y.grad.abs().max()


def test_largest_batch(ff):
    feat, target = inputs(1)
    lr = 3e-3
    w, adam, work = fresh(ff)
    w[384:448] = 0.1  # every unit reaches the output
    y = w.double().requires_grad_(True)
    h = torch.relu(feat[0].double() @ y[:320].view(64, 5).T + y[320:384])
    loss = (h @ y[384:448] + y[448] - target[0]) ** 2
    loss.backward()
    got = ff.ffmin_mlp_train(feat, target, 1, 2 ** 31 - 1, lr, 9, w, adam, work)
    assert abs(got[0] - float(loss.detach())) <= 0.01 * float(loss.detach())
    step, sign = w.double() - y.detach(), y.grad.sign()
    big = y.grad.abs() > 1e-4  # beside Adam's epsilon of 1e-8
    assert int(big.sum()) > 100
    assert (step + lr * sign)[big].abs().max() <= 1e-3 * lr
    assert step[y.grad == 0].abs().max() == 0.0


@pytest.mark.parametrize("steps,split", [(4100, 8192), (50, 7)])
def test_runs_of_several_launches(ff, variant, steps, split):
    feat, target = inputs(5000)
    one, two = fresh(ff), fresh(ff)
    st, la = variant(FFMIN_MLP_STEPS=split)(feat, target, steps, 300, 1e-3, 21, *one)
    lb = ff.ffmin_mlp_train(feat, target, steps, 300, 1e-3, 21, *two)
    assert st == ff.FFMIN_OK and np.isfinite(la).all() and la[-5:].mean() < la[:5].mean()
    assert np.array_equal(la, lb)
    for a, b in zip(one[:2], two[:2]):
        assert torch.equal(a, b)
