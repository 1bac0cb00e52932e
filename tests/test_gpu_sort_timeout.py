"""A bounded wait of the particle sort that runs out (made to by TG_DEBUG_SORT_HOLD: one tile publishes nothing, and
the waits for it are short): the error on every path, untouched outputs, the restored state, and a correct next call."""
import numpy as np
import pytest
import torch

from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")

N = 20001   # ten tiles, the last one ragged
BOTH = ["fp32", "fp64"]


def _prec(name):
    return tg.TG_PREC_FP64 if name == "fp64" else tg.TG_PREC_FP32


def _system(n, seed=1001):
    return tuple(torch.tensor(np.ascontiguousarray(a), device=DEV) for a in ics.plummer(n, seed))


def _close(a, ref, precision):
    """Two runs of one evaluation: they differ by the order of their sums (the bounds of the parity tests)."""
    nb = torch.linalg.norm(ref, dim=0)
    scale = nb if precision == "fp64" else torch.maximum(nb, 0.1 * nb.median())
    rel = (torch.linalg.norm(a - ref, dim=0) / scale).max().item()
    assert rel < (1e-13 if precision == "fp64" else 1e-5), rel


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("tile", [0, 4, 8])
@pytest.mark.parametrize("before", [0, 60000])   # a new context, and one whose buffers hold a larger sort's indices
def test_evaluation(precision, tile, before):
    P, _, M = _system(N)
    fast = (torch.arange(N, device=DEV) % 3 == 0).to(torch.uint8)
    prm = tg.Params(p=4, n_crit=64, precision=_prec(precision))
    ref, _ = tg.Solver(prm).fmm_forces(P, M, fast)
    s = tg.Solver(prm)
    if before:
        Pb, _, Mb = _system(before, 1002)
        s.fmm_forces(Pb, Mb)
    acc = torch.full((3, N), 12345.0, dtype=torch.float64, device=DEV)
    pot = torch.full((N,), 12345.0, dtype=torch.float64, device=DEV)
    tg.tg_debug_control(s.ctx, tg.TG_DEBUG_SORT_HOLD, tile)
    for _ in range(2):
        with pytest.raises(tg.TGError, match="TIMEOUT"):
            tg.tg_fmm_forces(s.ctx, P, M, fast, acc, pot)
        torch.cuda.synchronize()
        assert bool((acc == 12345.0).all()) and bool((pot == 12345.0).all())
    with pytest.raises(tg.TGError, match="TIMEOUT"):
        tg.tg_build_tree(s.ctx, P)
    tg.tg_debug_control(s.ctx, tg.TG_DEBUG_SORT_HOLD, -1)
    a, _ = s.fmm_forces(P, M, fast)
    _close(a, ref, precision)
    s.close()


def _step_params(precision, batched):
    # float32: a single rung, so that no rung decision turns the rounding of two runs into different steps
    return tg.Params(p=4, n_crit=64, dt_max=1 / 64, k_max=3 if precision == "fp64" else 0, eps=0.01,
                     precision=_prec(precision), batched=batched)


def _state(s, n):
    return tg.tg_hhs_state(s.ctx, n, DEV, with_total=True)


def _bound(prm, system):
    P0, V0, M = system
    s, P, V = tg.Solver(prm), P0.clone(), V0.clone()
    s.hhs_init(P, V, M)
    return s, P, V


def _same_step(P, V, Pr, Vr, prm, a):
    """Two kicks of dt/2 with accelerations that agree to the parity bounds."""
    tol = 1e-12 if prm.precision == tg.TG_PREC_FP64 else 1e-5 * prm.dt_max * float(a.max())
    assert float((V - Vr).abs().max()) <= tol and float((P - Pr).abs().max()) <= tol


@pytest.mark.parametrize("precision", BOTH)
@pytest.mark.parametrize("batched", [0, 1])
def test_step_is_restored(precision, batched):
    prm = _step_params(precision, batched)
    system = _system(N)
    ref, Pr, Vr = _bound(prm, system)
    ref.hhs_step()
    s, P, V = _bound(prm, system)
    before = _state(s, N)
    a = before[2]
    s.hhs_step()   # the graph of the batched step is there when the tile is held
    _same_step(P, V, Pr, Vr, prm, a)
    P1, V1, before = P.clone(), V.clone(), _state(s, N)
    ref.hhs_step()
    tg.tg_debug_control(s.ctx, tg.TG_DEBUG_SORT_HOLD, 2)
    for _ in range(2):
        with pytest.raises(tg.TGError, match="TIMEOUT"):
            s.hhs_step()
        torch.cuda.synchronize()
        assert torch.equal(P, P1) and torch.equal(V, V1)
        for x, y in zip(_state(s, N), before):
            assert torch.equal(x, y)
    tg.tg_debug_control(s.ctx, tg.TG_DEBUG_SORT_HOLD, -1)
    s.hhs_step()
    torch.cuda.synchronize()
    if precision == "fp32":   # two steps: the second starts from states that differ already
        prm = tg.Params(**{**prm.__dict__, "dt_max": 4 * prm.dt_max})
    _same_step(P, V, Pr, Vr, prm, a)
    s.close()
    ref.close()


def test_ensemble_restores_the_member_and_steps_the_others():
    prm = _step_params("fp64", 1)
    systems = [_system(3000, 1001), _system(N, 1002), _system(9000, 1003)]
    alone = [_bound(prm, x) for x in systems]
    members = [_bound(prm, x) for x in systems]
    ctxs = [m[0].ctx for m in members]
    held = ctxs[1]
    # the first call sizes the members' buffers with an evaluation of its own, before anything is stepped
    tg.tg_debug_control(held, tg.TG_DEBUG_SORT_HOLD, 0)
    with pytest.raises(tg.TGError, match="TIMEOUT"):
        tg.tg_ensemble_step(ctxs)
    torch.cuda.synchronize()
    for (_, P, V), (P0, V0, _) in zip(members, systems):
        assert torch.equal(P, P0) and torch.equal(V, V0)
    tg.tg_debug_control(held, tg.TG_DEBUG_SORT_HOLD, -1)
    tg.tg_ensemble_step(ctxs)
    # now the wait runs out inside the graph
    P1, V1, before = members[1][1].clone(), members[1][2].clone(), _state(members[1][0], N)
    tg.tg_debug_control(held, tg.TG_DEBUG_SORT_HOLD, 0)
    with pytest.raises(tg.TGError, match="TIMEOUT.*member 1"):
        tg.tg_ensemble_step(ctxs)
    torch.cuda.synchronize()
    assert torch.equal(members[1][1], P1) and torch.equal(members[1][2], V1)
    for x, y in zip(_state(members[1][0], N), before):
        assert torch.equal(x, y)
    for k, steps in ((0, 2), (1, 1), (2, 2)):
        for _ in range(steps):
            alone[k][0].hhs_step()
        _same_step(*members[k][1:], *alone[k][1:], prm, None)
    tg.tg_debug_control(held, tg.TG_DEBUG_SORT_HOLD, -1)
    members[1][0].hhs_step()
    alone[1][0].hhs_step()
    torch.cuda.synchronize()
    _same_step(*members[1][1:], *alone[1][1:], prm, None)
    for m in members + alone:
        m[0].close()


@pytest.mark.parametrize("tile", [0, 4, 8])
def test_allocation_free_sort(tile):
    P, _, _ = _system(N)
    keys, perm = tg.tg_morton_sort_noalloc(P)
    k, p = torch.empty_like(keys), torch.empty_like(perm)
    rc = tg.load().tg_debug_morton_sort_noalloc(N, tg._ptr(P), tg._ptr(k), tg._ptr(p), None, tile)
    torch.cuda.synchronize()
    assert rc == 0 and bool((p == -1).all())
    for hold in (-1, None):   # the call behind it is whole again
        if hold is None:
            k, p = tg.tg_morton_sort_noalloc(P)
        else:
            assert tg.load().tg_debug_morton_sort_noalloc(N, tg._ptr(P), tg._ptr(k), tg._ptr(p), None, hold) == 0
        torch.cuda.synchronize()
        assert torch.equal(k, keys) and torch.equal(p, perm)
