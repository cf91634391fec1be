"""Batches of more than five tiles per SM, where one block finalizes a whole tile,
and of more systems than the work queues' lists take at once: systems of one
and of two tiles with ragged ends, each many times.  Copies of a system do the
same sums in the same order, so they agree bit for bit; E + grad, E and ten
L-BFGS steps against the oracle with the FP64 bars of the other tests (E within
2e-11 of the terms, the gradient within 1e-9 of the largest force; after ten
steps E within 1e-8 and coordinates within 1e-6 A)."""
import numpy as np
import pytest

from paper_1810_03358_gb300 import synth
from tests.gpu_util import need_gpu, split, to_dev

pytestmark = pytest.mark.gpu
SIZES = (1, 2, 31, 33, 64, 97, 128, 129, 200)


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


def test_one_block_per_tile(ff, oracle_mod):
    import torch
    kinds = [synth.make_system(n, 900 + n) for n in SIZES]
    tiles = sum(-(-n // 128) for n in SIZES)
    copies = 5 * torch.cuda.get_device_properties(0).multi_processor_count // tiles + 2
    systems = kinds * copies
    assert len(systems) > 300
    S = ff.System(systems, 0)
    x0 = to_dev([s.x for s in systems])
    e, g = S.energy_grad(x0)
    e_only = S.energy(x0)
    x = x0.clone()
    r = S.minimize(x, method="LBFGS", max_iter=10)
    S.close()
    gs, xs = split(g.cpu().numpy(), systems), split(x.cpu().numpy(), systems)
    for k, s in enumerate(kinds):
        d, _, go = oracle_mod.energy_terms(s, s.x, grad=True)
        assert abs(e[k] - d["total"]) <= 2e-11 * d["sum_abs"] + 1e-300
        assert abs(e_only[k] - d["total"]) <= 2e-11 * d["sum_abs"] + 1e-300
        assert np.abs(gs[k] - go).max() <= 1e-9 * np.abs(go).max()
        xo, ro = oracle_mod.minimize(s, s.x, method=oracle_mod.LBFGS, max_iter=10)
        assert r[k]["iterations"] == ro["iterations"] and r[k]["status_name"] == ro["status_name"]
        assert abs(r[k]["energy"] - ro["energy"]) <= 1e-8 * abs(ro["energy"]) + 1e-300
        assert np.abs(xs[k] - xo).max() < 1e-6
        for c in range(1, copies):
            q = c * len(kinds) + k
            assert e[q] == e[k] and e_only[q] == e_only[k] and np.array_equal(gs[q], gs[k])
            assert r[q] == r[k] and np.array_equal(xs[q], xs[k])
