"""Gradient-free moves with FP64 terms on clusters, in the forms that the sizes
of the other tests do not reach: private copies of the positions in global
memory (too many atoms for shared memory), clusters of four, two and one block
a part, and rows in plain FP64 (offsets above 0.2 A, coordinates beyond 112 A).
Against the oracle with the bars of the epoch tests: coordinates within 1e-8 A
(a parabola's vertex carries the rounding of its row energies), in proportion
to the spacing of the coordinates where they are larger than 32 A."""
import dataclasses

import numpy as np
import pytest

from paper_1810_03358_gb300 import synth
from tests.gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


@pytest.fixture(scope="module")
def oracle_mod():
    from oracle import build, oracle
    build.build()
    return oracle


def system(n, seed, shift=0.0):
    s = synth.make_system(min(n, 1000), seed)
    x = s.x
    if n > 1000:  # copies of one chain side by side
        rng = np.random.default_rng(seed)
        k = -(-n // 1000)
        grid = np.array([(a, b, c) for a in range(3) for b in range(3) for c in range(3)][:k])
        x = (x[None] + 70.0 * (grid[:, None, :] - 1)).reshape(-1, 3)[:n]
        s = dataclasses.replace(s, charge=rng.uniform(-0.8, 0.8, n), sigma=rng.uniform(2.5, 3.8, n),
                                epsilon=rng.uniform(0.02, 0.2, n))
    x = np.ascontiguousarray(x + shift)
    return dataclasses.replace(s, x=x, x_ref=x)


# (atoms, parts, moves, delta, shift): sequential and epochs in global memory;
# clusters of four (20 parts), two (40) and one (80); plain rows
@pytest.mark.parametrize("n,parts,moves,delta,shift", [
    (7300, 0, 24, 0.05, 0.0), (4700, 64, 300, 0.05, 0.0), (700, 20, 600, 0.05, 0.0), (700, 40, 600, 0.05, 0.0),
    (700, 80, 600, 0.05, 0.0), (90, 0, 200, 0.3, 0.0), (90, 0, 200, 0.05, 150.0), (300, 4, 400, 0.05, 100.0)])
def test_moves_match_oracle(ff, oracle_mod, n, parts, moves, delta, shift):
    s = system(n, 840 + n, shift)
    kw = dict(method=4, max_iter=moves, gtol_inf=1e-9, seed=31, gradfree_delta=delta)
    if parts:
        kw.update(gradfree_parts=parts, gradfree_margin=0.5)
    S = ff.System([s], 0)
    x = to_dev([s.x])
    r = S.minimize(x, **kw)[0]
    S.close()
    xo, ro = oracle_mod.minimize(s, s.x, **kw)
    assert r["iterations"] == ro["iterations"]
    bar = 1e-8 * max(1.0, np.spacing(np.abs(s.x).max()) / np.spacing(31.0))
    assert np.abs(x.cpu().numpy().reshape(-1, 3) - xo).max() < bar
    assert abs(r["energy"] - ro["energy"]) <= 1e-10 * abs(ro["energy"])
