"""A linking length whose square is subnormal in float32 (members a few 1e-20
apart on a lattice, far from a few others): no weight of the half-precision
screen holds it, and every friend must be found all the same."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

from gpu_util import gpu_tree_dict, oracle_tree_dict

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [500, 1500, 6000])
@pytest.mark.parametrize("spacing", [2.0 ** -62, 2.0 ** -66, 2.0 ** -68])
def test_lattice_of_subnormal_squares(n, spacing):
    from paper_1110_4372_gb300 import rsgpu as rs
    rng = np.random.default_rng(n)
    side = int(np.ceil((0.95 * n) ** (1 / 3)))
    grid = np.stack(np.meshgrid(*[np.arange(side)] * 3), -1).reshape(-1, 3)[:int(0.95 * n)] * spacing
    pos = synth.wrap(np.concatenate([grid, rng.standard_normal((n - len(grid), 3)) * 0.15]), 20.0)
    vel = np.full((n, 3), 7.0, np.float32)
    perm, off = rng.permutation(n).astype(np.int32), np.array([0, n], np.int64)
    tree = rs.rs_refine6d(rs.Context(), *(torch.from_numpy(a).cuda() for a in (pos, vel)), 20.0,
                          *(torch.from_numpy(a).cuda() for a in (perm, off)))
    g, o = gpu_tree_dict(tree), oracle_tree_dict(oracle.refine(pos, vel, 20.0, perm, off))
    assert set(g) == set(o) and len(o) > 1
    for k in g:
        for q in ("members", "parent_key", "nchild"):
            assert g[k][q] == o[k][q], (k, q)
