"""Float64 P2P with a softening whose inverse cube leaves float64's range: the particle itself, masked pairs and the
empty slots of the packed rows and columns contribute nothing, whatever the value of a pair at r = 0 would be.

Tolerance: the sums of n float64 terms in two orders, each term a few roundings off: (n + 16) 2^-53 times the sum of
the terms' magnitudes (no cell pair is accepted at this opening angle, so the reference is the direct sum)."""
import numpy as np
import pytest
import torch

from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


def _newton(pos, mass, fast):
    """Accelerations, potentials and the sums of their terms' magnitudes of point masses."""
    n = mass.size
    d = pos[:, None, :] - pos[:, :, None]
    r = np.sqrt((d * d).sum(0)) + np.eye(n)
    use = ~np.eye(n, dtype=bool)
    if fast is not None:
        use &= ~(fast[:, None].astype(bool) & fast[None, :].astype(bool))
    w = np.where(use, mass[None, :], 0.0)
    return (w * d / r ** 3).sum(2), -(w / r).sum(1), (w / r ** 2).sum(1), (w / r).sum(1)


@pytest.mark.parametrize("n,n_crit", [(1, 8), (2, 8), (5, 2), (40, 7), (300, 33), (500, 256)])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("scale", [1.0, 1e8])
def test_f64_p2p_tiny_softening(n, n_crit, masked, kernel, scale):
    pos = ics.clustered(n, 1007)[0] * scale
    if scale > 1.0 and n > 2:   # round coordinates, such as a slot without a particle might hold
        pos[:, 0], pos[:, 1], pos[:, 2] = scale, -scale, 0.0
    mass = ics.random_masses(n, 3)
    fast = ics.random_fast_mask(n, 11, 0.5) if masked else None
    up = lambda a: None if a is None else torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    s = tg.Solver(tg.Params(p=2, theta=0.01, eps=1e-120, kernel=kernel, precision=tg.TG_PREC_FP64, n_crit=n_crit))
    acc, pot = s.fmm_forces(up(pos), up(mass), up(fast))
    only, _ = s.fmm_forces(up(pos), up(mass), up(fast), want_pot=False)
    a, p, a_top, p_top = _newton(pos, mass, fast)
    tol = (n + 16) * 2.0 ** -53
    for got in (acc, only):
        assert (np.linalg.norm(got.cpu().numpy() - a, axis=0) <= 2 * tol * a_top).all()   # both sides round
    assert (np.abs(pot.cpu().numpy() - p) <= 2 * tol * p_top).all()
    s.close()


@pytest.mark.parametrize("kernel", [0, 1])
def test_f64_masked_coincident_particles(kernel):
    # fast particles at one place: their pairs are left out, also where their value would not be finite
    pos, _, _ = ics.plummer(64, 1001)
    pos[:, 5:9] = pos[:, 4:5]
    mass = ics.random_masses(64, 3)
    fast = np.zeros(64, dtype=np.uint8)
    fast[4:20] = 1
    up = lambda x: torch.tensor(np.ascontiguousarray(x), device=DEV)  # noqa: E731
    s = tg.Solver(tg.Params(p=2, theta=0.01, eps=1e-120, kernel=kernel, precision=tg.TG_PREC_FP64, n_crit=16))
    acc, _ = s.fmm_forces(up(pos), up(mass), up(fast))
    d = pos[:, None, :] - pos[:, :, None]
    r = np.sqrt((d * d).sum(0))
    use = ~np.eye(64, dtype=bool) & ~(fast[:, None].astype(bool) & fast[None, :].astype(bool))
    r = np.where(use, r, 1.0)
    w = np.where(use, mass[None, :], 0.0)
    a, top = (w * d / r ** 3).sum(2), (w / r ** 2).sum(1)
    assert (np.linalg.norm(acc.cpu().numpy() - a, axis=0) <= 2 * 80 * 2.0 ** -53 * top).all()
    s.close()
