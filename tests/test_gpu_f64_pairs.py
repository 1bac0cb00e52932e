"""The float64 P2P and M2L kernels at the sizes where their packing can go wrong: work units whose last rows take
64, 32, 16 or 8 slots, columns that are no multiple of four, leaves of one particle and leaves wider than a
tile, few slow or few fast particles, trees with fewer M2L blocks than warps and rounds that are not full, every
order with a kernel of its own and the generic one above -- against the oracle.

Tolerance: each particle against 1e-12 of the force it would feel if every pull were aligned (the float64 parity
bound of the other tests, taken from a scale that no cancellation shrinks)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


def _up(a):
    return None if a is None else torch.tensor(np.ascontiguousarray(a), device=DEV)


def _pull(pos, mass, eps, kernel):
    d = pos[:, :, None] - pos[:, None, :]
    r = np.sqrt((d * d).sum(0))
    if kernel == 1:
        g = (r * r + eps * eps) ** -1.5
    else:
        u = np.minimum(r / eps, 1.0)
        g = np.where(r < eps, (21 * u ** 5 - 90 * u ** 4 + 140 * u ** 3 - 84 * u ** 2 + 14) / eps ** 3,
                     np.maximum(r, eps) ** -3.0)
    return (mass[None, :] * g * r).sum(1)


def _check(pos, mass, fast, p, theta, eps, kernel, n_crit):
    s = tg.Solver(tg.Params(p=p, theta=theta, eps=eps, kernel=kernel, precision=tg.TG_PREC_FP64, n_crit=n_crit))
    acc, pot = s.fmm_forces(_up(pos), _up(mass), _up(fast))
    only, _ = s.fmm_forces(_up(pos), _up(mass), _up(fast), want_pot=False)
    pairs = s.stats()["m2l_pairs"]
    s.close()
    a_o, p_o = oracle.fmm(pos, mass, oracle.params(p=p, theta=theta, eps=eps, kernel=kernel, n_crit=n_crit), fast)
    scale = 1e-12 * _pull(pos, mass, eps, kernel)
    for a in (acc, only):
        assert (np.linalg.norm(a.cpu().numpy() - a_o, axis=0) <= scale).all()
    assert np.abs(pot.cpu().numpy() - p_o).max() <= 1e-12 * np.abs(p_o).max()
    return pairs


@pytest.mark.parametrize("n,n_crit", [(2, 1), (9, 1), (40, 8), (130, 33), (300, 256), (700, 130), (900, 17), (1500, 49)])
@pytest.mark.parametrize("fraction", [0.0, 0.02, 0.5, 0.98])
@pytest.mark.parametrize("kernel", [0, 1])
def test_f64_p2p_packing(n, n_crit, fraction, kernel):
    # theta so small that no cell pair is accepted: every pair goes through P2P
    pos, _, _ = ics.clustered(n, 1007)
    fast = ics.random_fast_mask(n, 11, fraction) if fraction else None
    assert _check(pos, ics.random_masses(n, 3), fast, 2, 0.01, 0.05, kernel, n_crit) == 0


@pytest.mark.parametrize("p", [1, 2, 3, 4, 5, 6, 7])
@pytest.mark.parametrize("n,n_crit", [(60, 2), (700, 20), (2500, 3)])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("kernel", [0, 1])
def test_f64_m2l_rounds(p, n, n_crit, masked, kernel):
    pos, _, _ = ics.plummer(n, 1001)
    fast = ics.random_fast_mask(n, 11, 0.6) if masked else None
    assert _check(pos, ics.random_masses(n, 3), fast, p, 0.7, 0.01, kernel, n_crit) > 0


def test_f64_leaf_of_many_coincident_particles():
    # a deepest-level leaf far beyond n_crit: its self pair and its pairs take several column tiles
    pos, _, _ = ics.plummer(600, 1001)
    pos[:, :300] = pos[:, :1]
    mass = ics.random_masses(600, 3)
    fast = ics.random_fast_mask(600, 11, 0.4)
    _check(pos, mass, fast, 3, 0.5, 0.05, 0, 16)
