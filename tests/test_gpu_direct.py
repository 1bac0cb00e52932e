"""Direct summation (tg_direct_forces) at the sizes where its split of the sources can go wrong: fewer
sources than the eight blocks of a cluster, ragged eighths, tiles of sinks that are not full, each tile
width, masks and both kernels -- against the oracle's direct sum.

Tolerance: both sides add the same n float64 terms in different orders, each term a few roundings off, so
the difference is below (n + 16) u times the sum of the terms' magnitudes (u = 2^-53)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n,n_sink", [(1, 1), (2, 2), (7, 3), (300, 1), (2047, 33), (2049, 700), (5000, 4999)])
@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("masked", [False, True])
def test_direct_split_matches_oracle(n, n_sink, kernel, masked):
    eps = 0.2   # a good part of the pairs is softened
    pos, _, _ = ics.clustered(n, 1007)
    mass = ics.random_masses(n, 3)
    fast = ics.random_fast_mask(n, 5) if masked else None
    sinks = np.random.default_rng(n).permutation(n)[:n_sink].astype(np.int64)
    s = tg.Solver(tg.Params(p=3, eps=eps, kernel=kernel))
    up = lambda a: None if a is None else torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    acc, pot = s.direct_forces(up(pos), up(mass), up(fast), up(sinks))
    only, _ = tg.tg_direct_forces(s.ctx, up(pos), up(mass), up(fast), up(sinks))
    a_o, p_o = oracle.direct(pos, mass, eps, kernel, fast, sinks)
    u = 2.0 ** -53
    # terms are at most m g r <= m * max(g r) and m |phi| <= m |phi(0)|
    grid = np.linspace(1e-6, 3.0, 20001)
    if kernel == 1:
        top_f, top_p = (grid * (grid * grid + eps * eps) ** -1.5).max(), 1.0 / eps
    else:
        w = np.minimum(grid / eps, 1.0)
        g = np.where(grid < eps, (21 * w ** 5 - 90 * w ** 4 + 140 * w ** 3 - 84 * w ** 2 + 14) / eps ** 3, grid ** -3.0)
        top_f, top_p = (g * grid).max(), 3.0 / eps
    tol = (n + 16) * u * mass.sum()
    assert np.abs(acc.cpu().numpy() - a_o).max() <= tol * top_f
    assert np.abs(pot.cpu().numpy() - p_o).max() <= tol * top_p
    assert torch.equal(only, acc)   # the sums are added in a fixed order: two calls agree bit for bit
    s.close()


def test_direct_pairs_outside_the_float64_cube_range():
    # squared distances far outside the range of the series: the Newtonian force underflows to zero at 1e170
    # and is finite at 1e-100
    for sep, want in ((1e170, 0.0), (1e-100, 0.5e200)):
        pos = torch.zeros((3, 2), dtype=torch.float64, device=DEV)
        pos[0, 1] = sep
        mass = torch.tensor([0.5, 0.5], dtype=torch.float64, device=DEV)
        s = tg.Solver(tg.Params(p=3, eps=1e-120, kernel=0))
        acc, _ = s.direct_forces(pos, mass)
        got = float(acc[0, 0])
        assert got == want if want == 0.0 else abs(got - want) < 1e-14 * want
        s.close()
