"""How far two runs of one float32 step may differ.  The sums of an evaluation are added in an order that changes from
run to run, so accelerations repeat to float32 rounding; a step repeats as well as that as long as no particle's
timestep lies within that rounding of a rung's pivot step.  (One that does may take either rung, and a deep rung's few
particles then follow another path.)  Here the pivot lies in a gap of the timesteps: the rungs have to be equal, and
the velocities within the kicks' rounding."""
import numpy as np
import pytest
import torch

from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


@pytest.mark.parametrize("n", [3000, 12001])
@pytest.mark.parametrize("kernel", [0, 1])
def test_float32_step_repeats_to_rounding_away_from_the_pivot(n, kernel):
    pos, vel, mass = (torch.tensor(np.ascontiguousarray(a), device=DEV) for a in ics.plummer(n, 1001))
    base = dict(p=5, theta=0.5, n_crit=64, eps=0.01, kernel=kernel, precision=tg.TG_PREC_FP32, k_max=1)
    s = tg.Solver(tg.Params(dt_max=1.0, **base))
    s.hhs_init(pos.clone(), vel.clone(), mass)
    a = tg.tg_hhs_state(s.ctx, n, DEV)[2]
    eta = tg.Params(**base).eta
    s.close()
    dt = np.sort(np.sqrt(eta * base["eps"] / a.cpu().numpy()))
    mid = dt[n // 4: 3 * n // 4]
    gap = mid[1:] / mid[:-1]
    k = int(gap.argmax())
    assert gap[k] - 1.0 > 1e-4   # ten times the bound of an acceleration on each side
    dt_max = float(np.sqrt(mid[k] * mid[k + 1]))
    runs = []
    for batched in (0, 0, 1, 1):
        s, P, V = tg.Solver(tg.Params(dt_max=dt_max, batched=batched, **base)), pos.clone(), vel.clone()
        s.hhs_init(P, V, mass)
        s.hhs_step()
        runs.append((P, V, tg.tg_hhs_state(s.ctx, n, DEV)[0]))
        s.close()
    assert 0 < int(runs[0][2].sum()) < n
    # two sums (slow and fast sources) of accelerations, each within 1e-5 of the exact ones in both runs
    tol = 4e-5 * dt_max * float(a.max())
    for P, V, rung in runs[1:]:
        assert torch.equal(rung, runs[0][2])
        assert float((V - runs[0][1]).abs().max()) <= tol
        assert float((P - runs[0][0]).abs().max()) <= tol * dt_max
