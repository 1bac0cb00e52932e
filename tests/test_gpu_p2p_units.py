"""P2P on both sides of the pair counts where its work units change size (8192 leaf pairs in float32, 16,384 and 32,768
in float64), against the oracle: one particle per leaf and no accepted cell pair make n (n - 1) / 2 leaf pairs.

Tolerance: the float32 and float64 parity bounds of the other tests (1e-5 and 1e-12), of the force that a particle
would feel if every pull were aligned."""
import numpy as np
import pytest
import torch

import oracle
from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n", [2, 127, 128, 129, 130, 181, 182, 256, 257])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_unit_sizes(n, masked, kernel, precision):
    eps = 0.05
    pos, _, _ = ics.clustered(n, 1007)
    mass = ics.random_masses(n, 3)
    fast = ics.random_fast_mask(n, 11, 0.4) if masked else None
    up = lambda a: None if a is None else torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    s = tg.Solver(tg.Params(p=2, theta=0.01, eps=eps, kernel=kernel, n_crit=1,
                            precision=tg.TG_PREC_FP64 if precision == "fp64" else tg.TG_PREC_FP32))
    acc, pot = s.fmm_forces(up(pos), up(mass), up(fast))
    only, _ = s.fmm_forces(up(pos), up(mass), up(fast), want_pot=False)
    stats = s.stats()
    assert stats["m2l_pairs"] == 0 and stats["p2p_cell_pairs"] == 2 * (n * (n - 1) // 2 + n)   # two calls, self pairs
    s.close()
    a_o, p_o = oracle.direct(pos, mass, eps, kernel, fast)
    d = pos[:, :, None] - pos[:, None, :]
    r = np.sqrt((d * d).sum(0))
    pull = (mass[None, :] * r * np.maximum(r, 0.3 * eps) ** -3.0).sum(1)   # no pair pulls harder than at 0.3 eps
    bound = 1e-12 if precision == "fp64" else 1e-5
    for a in (acc, only):
        assert (np.linalg.norm(a.cpu().numpy() - a_o, axis=0) <= bound * pull).all()
    assert np.abs(pot.cpu().numpy() - p_o).max() <= bound * np.abs(p_o).max()
