"""MIXED exclusion variant with scaled partners anywhere: the FP32 sweeps walk an
atom's sorted partners along a j tile 32 atoms at a time, so partners sit at the
edges of those windows and of tiles, in far tiles, and many on one atom.  Bars:
those of the MIXED exclusion tests."""
import dataclasses

import numpy as np
import pytest

from paper_1810_03358_gb300 import synth
from tests.gpu_util import need_gpu
from tests.test_gpu_exclusions import check_mixed, excl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


@pytest.fixture(scope="module")
def oracle_mod():
    from oracle import build, oracle
    build.build()
    return oracle


def with_bonds(s, pairs):
    """s with further bonds at their present length (excluded pairs without force)"""
    pairs = np.array(pairs, dtype=np.int32)
    r = np.linalg.norm(s.x[pairs[:, 0]] - s.x[pairs[:, 1]], axis=1)
    return dataclasses.replace(s, bond_idx=np.ascontiguousarray(np.concatenate([s.bond_idx, pairs])),
                               bond_k=np.concatenate([s.bond_k, np.full(len(pairs), 1.0)]),
                               bond_r0=np.concatenate([s.bond_r0, r]))


@pytest.mark.parametrize("n", [130, 300, 1000])
def test_partners_at_window_and_tile_edges(ff, oracle_mod, n):
    s = synth.make_system(n, 70 + n)
    edges = [0, 31, 32, 63, 64, 95, 96, 127, 128, n - 1]
    pairs = [(a, b) for a in edges for b in edges if a + 3 < b]
    pairs += [(5, int(b)) for b in range(40, min(n, 120), 2)]  # many partners of one atom
    check_mixed(ff, oracle_mod, [excl(with_bonds(s, pairs))])
