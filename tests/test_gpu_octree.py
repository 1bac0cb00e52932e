"""The particle sort at its edges (one block up to 8192 particles, tiles of 2048 above, equal keys in input order)
and the octree build (windows of n_crit + 1 keys, cells ranked per level) against the oracle's tree, bit for bit, at
the sizes where it can go wrong: one particle, tiles of 1024 positions and their neighbours, the smallest and
the largest leaves, few levels, coincident particles (keys equal to the last level) and a far outlier (every
other particle in one deep corner)."""
import numpy as np
import pytest
import torch

import oracle
from paper_1712_10116_gb300 import ics

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_1712_10116_gb300 import binding as tg
    DEV = torch.device("cuda:0")


def _points(kind, n):
    pos = ics.clustered(n, 1007)[0] if kind != "sphere" else ics.uniform_sphere(n, 1002)[0]
    if kind == "coincident":
        pos[:, : (2 * n) // 3] = pos[:, :1]
    if kind == "outlier":
        pos[:, 0] = 4000.0
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("n", [1, 2, 31, 1022, 1023, 1024, 1025, 2047, 2048, 5000])
@pytest.mark.parametrize("n_crit", [1, 2, 7, 64, 255, 256])
@pytest.mark.parametrize("kind", ["sphere", "clustered", "coincident", "outlier"])
def test_tree_matches_oracle(n, n_crit, kind):
    pos = _points(kind, n)
    for max_level in (21, 3, 1) if n_crit in (2, 64) else (21,):
        s = tg.Solver(tg.Params(p=2, n_crit=n_crit, max_level=max_level))
        tg.tg_build_tree(s.ctx, torch.tensor(pos, device=DEV))
        t = tg.tg_get_tree(s.ctx)
        s.close()
        o = oracle.Tree(pos, oracle.params(n_crit=n_crit, max_level=max_level))
        assert np.array_equal(t["keys"], o.keys) and np.array_equal(t["perm"], o.perm)
        for name in ("level", "coords", "first", "count", "nchild"):
            assert np.array_equal(t[name], getattr(o, name)), name


@pytest.mark.parametrize("n", [8191, 8192, 8193, 10240, 10241, 40959, 100001])
@pytest.mark.parametrize("kind", ["clustered", "coincident", "outlier"])
def test_sort_matches_oracle(n, kind):
    pos = _points(kind, n)
    if kind == "coincident":
        pos[:, n // 2:] = pos[:, :1]   # one key for almost every particle: the order is the input order
    s = tg.Solver(tg.Params(p=2, n_crit=64))
    d = torch.tensor(pos, device=DEV)
    for _ in range(2):
        tg.tg_build_tree(s.ctx, d)
        t = tg.tg_get_tree(s.ctx)
        k, p = tg.tg_morton_sort_noalloc(d)
        o = oracle.Tree(pos, oracle.params(n_crit=64))
        assert np.array_equal(t["keys"], o.keys) and np.array_equal(t["perm"], o.perm)
        assert np.array_equal(k.cpu().numpy().view(np.uint64), o.keys) and np.array_equal(p.cpu().numpy(), o.perm)
    s.close()
