"""The pair search's list has room for 20 pairs a member wherever its blocks
take their chunks: levels of one and of a few small nodes, which have fewer
blocks than the list has regions, are not searched for friends a second time
(rf_lvl_link), and the trees equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

from gpu_util import compare_trees, gpu_tree_dict, oracle_tree_dict

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _nfw_groups(sizes, seed):
    """NFW groups (concentration 10, radius 1, one velocity dispersion) on a lattice of the box."""
    rng = np.random.default_rng([seed, len(sizes)])
    box = 50.0
    at = np.stack(np.meshgrid(*[np.arange(5) * 10.0 + 5.0] * 3), -1).reshape(-1, 3)[:len(sizes)]
    x = np.concatenate([[0.0], np.logspace(-5, 1, 4000)])
    m = np.log1p(x) - x / (1 + x)
    n = sum(sizes)
    d = rng.standard_normal((n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    pos = np.repeat(at, sizes, 0) + d * np.interp(rng.random(n), m / m[-1], x / x[-1])[:, None]
    vel = rng.standard_normal((n, 3)) * 300.0
    perm = rng.permutation(n).astype(np.int32)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p, v = np.empty_like(pos), np.empty_like(vel)
    p[perm], v[perm] = pos, vel
    return synth.wrap(p, box), v.astype(np.float32), box, perm, off


@pytest.mark.parametrize("sizes", [[1025], [1100], [1500], [2000], [3000], [4000], [2000] * 20])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_small_levels_fit_the_list(sizes, seed):
    from paper_1110_4372_gb300 import rsgpu as rs
    ctx = rs.Context()
    rs.rs_profile_enable(ctx)
    pos, vel, box, perm, off = _nfw_groups(sizes, seed)
    tree = rs.rs_refine6d(ctx, *(torch.from_numpy(a).cuda() for a in (pos, vel)), box,
                          *(torch.from_numpy(a).cuda() for a in (perm, off)))
    ran = rs.rs_profile_read(ctx)
    assert "rf_lvl_pairs" in ran and "rf_lvl_link" not in ran
    compare_trees(gpu_tree_dict(tree), oracle_tree_dict(oracle.refine(pos, vel, box, perm, off)), box)
