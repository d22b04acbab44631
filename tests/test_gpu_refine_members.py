"""The refinement's passes over the members of all groups: group edges inside
a warp's 32 slots, empty groups, offsets that start after the first slot,
groups across each face of the box, and nodes at the edges of the 1024
members whose moments one block adds up.  The trees, moments included, must
equal the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

from gpu_util import compare_trees, gpu_tree_dict, oracle_tree_dict

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EDGES = [0, 10, 31, 32, 33, 1, 0, 0, 64, 65, 12, 100, 2, 15, 300, 0]


@pytest.mark.parametrize("sizes,skip,stride", [(EDGES, 0, 3), (EDGES, 37, 4), ([1] * 70 + [40], 0, 3),
                                               ([1025, 1279, 1280, 11], 5, 3), ([2047, 2048, 2049, 5121], 0, 4)])
def test_group_members_match_oracle(sizes, skip, stride):
    from paper_1110_4372_gb300 import rsgpu
    rng = np.random.default_rng([len(sizes), skip])
    box, n = 20.0, sum(sizes) + skip
    corners = np.stack(np.meshgrid(*[[0.0, 7.0, 14.0]] * 3), -1).reshape(-1, 3)
    pos, vel = rng.random((n, 3)) * box, rng.standard_normal((n, 3)) * 60.0
    perm, at = rng.permutation(n).astype(np.int32), skip
    for k, s in enumerate(sizes):
        pos[perm[at:at + s]] = corners[k % 27] + rng.standard_normal((s, 3)) * 0.15
        at += s
    pos, vel = synth.wrap(pos, box), vel.astype(np.float32)
    off = skip + np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p, v = torch.from_numpy(pos).cuda(), torch.from_numpy(vel).cuda()
    if stride == 4:
        p, v = (torch.nn.functional.pad(a, (0, 1)).contiguous() for a in (p, v))
    tree = rsgpu.rs_refine6d(rsgpu.Context(), p, v, box, torch.from_numpy(perm).cuda(), torch.from_numpy(off).cuda())
    o = oracle.refine(pos, vel, box, perm, off)
    assert o.n_nodes > 0
    compare_trees(gpu_tree_dict(tree), oracle_tree_dict(o), box)


@pytest.mark.parametrize("n,f,bracket_min", [(1025, 0.02, 4096), (1025, 0.99, 4096), (4096, 0.99, 4096),
                                             (4097, 0.02, 4096), (9000, 0.7, 1 << 30), (1500, 0.98, 1024)])
def test_sampled_brackets_match_oracle(n, f, bracket_min):
    """Both sample sizes, where the bracket's quantiles are cut off at the
    sample's ends (below the first or above the last value)."""
    from paper_1110_4372_gb300 import rsgpu
    rng = np.random.default_rng([n, bracket_min])
    box = 20.0
    pos = synth.wrap(rng.standard_normal((n, 3)) * 0.15, box)
    vel = (rng.standard_normal((n, 3)) * 60.0).astype(np.float32)
    perm, off = np.arange(n, dtype=np.int32), np.array([0, n], np.int64)
    ctx = rsgpu.Context()
    rsgpu.rs_set_tuning(ctx, bracket_min=bracket_min)
    tree = rsgpu.rs_refine6d(ctx, *(torch.from_numpy(a).cuda() for a in (pos, vel)), box,
                             torch.from_numpy(perm).cuda(), torch.from_numpy(off).cuda(), f)
    compare_trees(gpu_tree_dict(tree), oracle_tree_dict(oracle.refine(pos, vel, box, perm, off, f)), box)


@pytest.mark.parametrize("n", [2000, 6000])
def test_more_pairs_than_listed_match_oracle(n):
    """The bracket spans the gap between a core's neighbour distances and the
    sparse rest's, so the core's pairs (n^2 / 5) lie inside it: far more than
    the 20 a member that the pair search lists."""
    from paper_1110_4372_gb300 import rsgpu
    rng = np.random.default_rng(n)
    box, f = 20.0, 0.7
    scale = np.where(np.arange(n) < f * n, 0.05, 1.0)[:, None]
    pos = synth.wrap(rng.standard_normal((n, 3)) * 0.15 * scale + 10.0, box)
    vel = (rng.standard_normal((n, 3)) * 60.0 * scale).astype(np.float32)
    perm, off = rng.permutation(n).astype(np.int32), np.array([0, n], np.int64)
    tree = rsgpu.rs_refine6d(rsgpu.Context(), *(torch.from_numpy(a).cuda() for a in (pos, vel)), box,
                             torch.from_numpy(perm).cuda(), torch.from_numpy(off).cuda(), f)
    compare_trees(gpu_tree_dict(tree), oracle_tree_dict(oracle.refine(pos, vel, box, perm, off, f)), box)


@pytest.mark.parametrize("bad", [-1, 500])
def test_index_out_of_range_is_an_error(bad):
    from paper_1110_4372_gb300 import rsgpu
    rng = np.random.default_rng(5)
    pos = torch.from_numpy(rng.random((500, 3)).astype(np.float32)).cuda()
    perm = torch.arange(500, dtype=torch.int32, device="cuda")
    perm[[40, 499]] = bad
    off = torch.tensor([0, 37, 500], dtype=torch.int64, device="cuda")
    ctx = rsgpu.Context()
    with pytest.raises(rsgpu.RsError):
        rsgpu.rs_refine6d(ctx, pos, pos, 20.0, perm, off)
