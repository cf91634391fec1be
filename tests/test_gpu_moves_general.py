"""Gradient-free moves with FP64 terms where their rows leave the fixed-point
form: offsets above 0.2 A, the far field and systems beyond 112 A in rows from
FP64 differences (positions in shared memory, in global memory, parts of one
block, of a cluster), single atoms out there, and the sequential search on
the whole grid above 8,000 atoms.  Against the oracle with the bars of the
epoch tests (coordinates within 1e-8 A, in proportion to the spacing of the
coordinates where they are larger than 32 A).

And what they cost: the work of a move is that of the plain rows plus nine
differences a pair in FP64, about 1.4 times (1.6 with the far field), or
two launches over all SMs; three times leaves room for both, where a row
evaluated position by position took 4.8 times."""
import dataclasses
import time

import numpy as np
import pytest

from tests.gpu_util import need_gpu, to_dev
from tests.test_gpu_moves64 import system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


@pytest.fixture(scope="module")
def oracle_mod():
    from oracle import build, oracle
    build.build()
    return oracle


def against_oracle(ff, oracle_mod, s, **kw):
    kw = dict(method=4, gtol_inf=1e-9, seed=31, **kw)
    S = ff.System([s], 0)
    x = to_dev([s.x])
    r = S.minimize(x, **kw)[0]
    S.close()
    xo, ro = oracle_mod.minimize(s, s.x, **kw)
    assert r["iterations"] == ro["iterations"]
    bar = 1e-8 * max(1.0, np.spacing(np.abs(s.x).max()) / np.spacing(31.0))
    assert np.abs(x.cpu().numpy().reshape(-1, 3) - xo).max() < bar
    assert abs(r["energy"] - ro["energy"]) <= 1e-10 * abs(ro["energy"])


FAR = dict(gradfree_taylor_r=8.0)


@pytest.mark.parametrize("n,parts,moves,shift,kw", [
    (5, 0, 40, 0.0, FAR), (700, 20, 600, 0.0, FAR), (700, 80, 600, 0.0, FAR), (700, 80, 600, 130.0, {}),
    (7300, 0, 24, 0.0, dict(gradfree_delta=0.3)), (7300, 0, 24, 0.0, FAR), (4700, 64, 300, 0.0, FAR),
    (8000, 0, 16, 0.0, FAR), (8001, 0, 16, 0.0, FAR), (8100, 0, 16, 0.0, dict(gradfree_delta=0.3))])
def test_general_rows_match_oracle(ff, oracle_mod, n, parts, moves, shift, kw):
    s = system(n, 840 + n, shift)
    if parts:
        kw = dict(kw, gradfree_parts=parts, gradfree_margin=0.5)
    against_oracle(ff, oracle_mod, s, max_iter=moves, **kw)


@pytest.mark.parametrize("n,parts", [(700, 0), (700, 20), (90, 0)])
def test_few_atoms_far_out(ff, oracle_mod, n, parts):
    # a bonded pair of atoms beyond the range (up to n / 256 such atoms keep the
    # fixed-point rows; at 90 atoms none): they move, and are partners of the
    # others' moves.  A change of any start coordinate by one place moves the
    # oracle's result by 1e-11 A at most
    s = system(n, 77)
    x = s.x.copy()
    x[-1], x[-2] = (121.3, 2.0, -1.0), (122.0, 3.1, -0.2)
    whole = {k: ~np.any((i >= n - 2) & (i.min(axis=1, keepdims=True) < n - 2), axis=1)
             for k, i in (("bond", s.bond_idx), ("angle", s.angle_idx), ("dihedral", s.dihedral_idx))}
    s = dataclasses.replace(
        s, x=x, x_ref=x, bond_idx=s.bond_idx[whole["bond"]], bond_k=s.bond_k[whole["bond"]],
        bond_r0=s.bond_r0[whole["bond"]], angle_idx=s.angle_idx[whole["angle"]], angle_k=s.angle_k[whole["angle"]],
        angle_theta0=s.angle_theta0[whole["angle"]], dihedral_idx=s.dihedral_idx[whole["dihedral"]],
        dihedral_v=s.dihedral_v[whole["dihedral"]])
    kw = dict(gradfree_parts=parts, gradfree_margin=0.5) if parts else {}
    against_oracle(ff, oracle_mod, s, max_iter=2 * n, **kw)


@pytest.mark.parametrize("n,kw", [(3334, FAR), (3334, dict(gradfree_delta=0.3)), (12000, FAR),
                                  (12000, dict(gradfree_delta=0.3))])
def test_general_rows_cost(ff, n, kw):
    import torch
    s = system(n, 5)
    S = ff.System([s], 0)
    x0 = to_dev([s.x])
    x = x0.clone()

    def move_time(kw):  # of one move: 640 moves less 128 (both with two evaluations)
        t = {}
        for m in (128, 640):
            runs = []
            for _ in range(5):
                x.copy_(x0)
                torch.cuda.synchronize()
                a = time.perf_counter()
                S.minimize(x, method=4, gtol_inf=1e-9, seed=31, max_iter=m, **kw)
                runs.append(time.perf_counter() - a)
            t[m] = min(runs)
        return (t[640] - t[128]) / 512
    plain, general = move_time({}), move_time(kw)
    S.close()
    assert general < 3.0 * plain, (plain, general)
