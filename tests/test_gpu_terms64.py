"""FP64 pair terms formed on 64-bit significands: whole tiles, tiles in two
and in four parts, and coordinates or parameters outside the range of the
integer forms (those pairs take the FP64 formula), against the oracle.

Bars: the plain FP64 bars (tests/test_gpu_energy.py): E within 2e-11 of
sum |terms|, the gradient within 1e-9 of the largest force; a term's rounding
error is below 2 units of 2^-53, so they are not tight."""
import dataclasses
import math

import numpy as np
import pytest

from paper_1810_03358_gb300 import synth
from tests.gpu_util import need_gpu, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    return need_gpu()


@pytest.fixture(scope="module")
def orc():
    from oracle import build, oracle
    build.build()
    return oracle


def check(ff, orc, s):
    S = ff.System([s], 0)
    x = to_dev([s.x])
    e, g = S.energy_grad(x)
    e_only = S.energy(x)
    S.close()
    # the oracle by blocks of 50 rows: one running sum of 4e7 terms, most of
    # them far below its last place, would be off by more than the bar itself
    blocks = [orc.energy_rows(s, s.x, i, min(i + 50, s.n_atoms)) for i in range(0, s.n_atoms, 50)]
    d = {k: math.fsum(b[0][k] for b in blocks) for k in ("total", "sum_abs")}
    assert all(b[1] == 0 for b in blocks)
    go = sum(b[2] for b in blocks)
    g = g.cpu().numpy().reshape(-1, 3)
    assert abs(e[0] - d["total"]) <= 2e-11 * d["sum_abs"]
    assert abs(e_only[0] - d["total"]) <= 2e-11 * d["sum_abs"]
    assert np.abs(g - go).max() <= 1e-9 * np.abs(go).max()


# 1 to 3 tiles, ragged last parts, sizes with four parts a tile pair (up to 2,000,
# 6,200 and 6,273), two (3,400 and 9,000) and whole tiles (4,352 and 4,481);
# clusters of eight blocks a part up to 257, of four (1,000 and 1,101) and two (2,000)
@pytest.mark.parametrize("n", [31, 33, 96, 97, 257, 1000, 1101, 2000, 3400, 4352, 4481, 6200, 6273, 9000])
def test_tiles_and_parts(ff, orc, n):
    rng = np.random.default_rng(n)
    s = synth.make_system(min(n, 2000), 900 + n)
    if n > 2000:  # copies of one chain side by side
        k = -(-n // 2000)
        shift = np.arange(k)[:, None] * np.array([[60.0, 0.0, 0.0]])
        x = (s.x[None] + shift[:, None, :]).reshape(-1, 3)[:n]
        s = dataclasses.replace(s, x=np.ascontiguousarray(x), x_ref=x, charge=rng.uniform(-0.8, 0.8, n),
                                sigma=rng.uniform(2.5, 3.8, n), epsilon=rng.uniform(0.02, 0.2, n))
    check(ff, orc, s)


@pytest.mark.parametrize("what", ["zeros", "tiny", "huge", "far", "axis", "denormal_d"])
def test_out_of_range_and_special_values(ff, orc, what):
    s = synth.make_system(200, 77)
    x, q, ep = s.x.copy(), s.charge.copy(), s.epsilon.copy()
    if what == "zeros":      # uncharged atoms, atoms without Lennard-Jones
        q[::3] = 0.0
        ep[1::4] = 0.0
        q[7] = -0.0
    elif what == "tiny":     # below 2^-200
        q[5] = 1e-70
        ep[9] = 1e-150
    elif what == "huge":     # above 2^200
        q[5] = 1e62
    elif what == "far":      # beyond 2^41 A
        x[150:] += 1e13
    elif what == "axis":     # differences along one axis only
        x = np.stack([np.arange(200) * 1.5, np.zeros(200), np.zeros(200)], axis=1)
        s = dataclasses.replace(s, dihedral_v=np.zeros_like(s.dihedral_v), angle_k=np.zeros_like(s.angle_k))
    else:                    # one difference far below the others
        x[1::2, 2] = x[::2, 2] + 1e-310
    check(ff, orc, dataclasses.replace(s, x=np.ascontiguousarray(x), charge=q, epsilon=ep))


@pytest.mark.parametrize("what", ["plain", "zeros", "tiny", "huge", "far", "negative_sigma"])
@pytest.mark.parametrize("n", [31, 32, 33, 150, 2049])
def test_noalloc_special_values(ff, n, what):
    """The allocation-free entry point against the same sums in numpy; it
    takes parameters unchecked, a negative sigma among them."""
    import torch
    rng = np.random.default_rng(n)
    x = synth.make_system(n, 5).x
    q, sg, ep = rng.uniform(-0.8, 0.8, n), rng.uniform(2.5, 3.8, n), rng.uniform(0.02, 0.2, n)
    if what == "zeros":
        q[::3] = 0.0
        ep[1::4] = 0.0
    elif what == "tiny":
        ep[9] = 1e-150
    elif what == "huge":
        q[5] = 1e62
    elif what == "far":
        x[n // 2:] += 1e13
    elif what == "negative_sigma":
        sg[::5] *= -1.0

    def dev(a):
        return torch.tensor(np.ascontiguousarray(a).reshape(-1), dtype=torch.float64, device="cuda")

    g, e = torch.empty(3 * n, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.float64, device="cuda")
    ff.ffmin_pair_energy_grad_noalloc(dev(x), dev(q), dev(sg), dev(ep), g, e, coulomb_c=332.0)
    d = x[None] - x[:, None]
    r2 = (d * d).sum(-1)
    np.fill_diagonal(r2, 1.0)
    w = 1.0 - np.eye(n)
    ec = 332.0 * np.outer(q, q) / np.sqrt(r2) * w
    s6, e4 = (np.outer(sg, sg) / r2) ** 3, 4.0 * np.sqrt(np.outer(ep, ep)) * w
    e_ref = 0.5 * (ec + e4 * (s6 * s6 - s6)).sum()
    f = (ec + e4 * (12.0 * s6 * s6 - 6.0 * s6)) / r2
    g_ref = (f[:, :, None] * d).sum(1)
    total = 0.5 * (np.abs(ec) + e4 * (s6 * s6 + np.abs(s6))).sum()
    assert abs(e.item() - e_ref) <= 2e-11 * total
    assert np.abs(g.cpu().numpy().reshape(n, 3) - g_ref).max() <= 1e-9 * np.abs(g_ref).max()


@pytest.mark.parametrize("sizes", [(1,), (2, 127, 128, 129), (700, 5, 1025, 300)])
def test_neighbour_counts(ff, orc, sizes):
    """Counts within 8 A at tile edges and in a ragged batch, by brute force in
    the FP32 arithmetic of the kernel."""
    import torch
    systems = [synth.make_system(n, 300 + n) for n in sizes]
    S = ff.System(systems, 0)
    counts = torch.full((S.n_atoms,), -1, dtype=torch.int32, device="cuda")
    ff.ffmin_neighbour_counts(S.handle, to_dev([s.x for s in systems]), counts)
    S.close()
    want = []
    for s in systems:
        x = s.x.astype(np.float32)
        d = x[:, None] - x[None]
        near = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2] < np.float32(64.0)
        want.append(near.sum(1) - 1)
    assert np.array_equal(counts.cpu().numpy(), np.concatenate(want))
