"""The refinement without its list of pairs, as when the list would pass its
limit (levels of about 104 million members and more) or finds no memory: every
member searches its nearest neighbour within the sampled bracket, and every
node's friends are searched once the linking length is known.  RS_FAULT=pairs
leaves the list out at any size; trees must equal the oracle's exactly."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

from gpu_util import compare_trees, gpu_tree_dict, oracle_tree_dict
from test_gpu_leaf_search import _members

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _groups(kinds, sizes, seed):
    """Groups on a lattice of the box, members shuffled: what rs_refine6d takes."""
    rng = np.random.default_rng(seed)
    box = 40.0
    at = np.stack(np.meshgrid(*[np.arange(4) * 10.0] * 3), -1).reshape(-1, 3)
    parts = [_members(k, n, rng) for k, n in zip(kinds, sizes)]
    pos = np.vstack([p + c for (p, _), c in zip(parts, at)])
    vel = np.vstack([v for _, v in parts])
    perm = rng.permutation(len(pos))
    shuffled = np.empty(len(pos), np.int32)
    shuffled[perm] = np.arange(len(pos))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return synth.wrap(pos[perm], box), vel[perm].astype(np.float32), box, shuffled, off


def _refine(rs, ctx, g, f):
    pos, vel, box, perm, off = g
    rs.rs_profile_reset(ctx)
    tree = rs.rs_refine6d(ctx, *(torch.from_numpy(a).cuda() for a in (pos, vel)), box,
                          *(torch.from_numpy(a).cuda() for a in (perm, off)), f)
    return gpu_tree_dict(tree), rs.rs_profile_read(ctx)


@pytest.mark.parametrize("kinds,sizes,f", [
    (["blob"], [1025], 0.7), (["blob"], [33_000], 0.7), (["pairs", "copies", "still"], [5001, 6000, 1100], 0.7),
    (["blob", "copies", "blob"], [4096, 4097, 2049], 0.9), (["blob"] * 20, [1500 + 37 * k for k in range(20)], 0.5)])
def test_trees_without_the_pair_list_match_oracle(monkeypatch, kinds, sizes, f):
    from paper_1110_4372_gb300 import rsgpu as rs
    ctx = rs.Context()
    rs.rs_profile_enable(ctx)
    g = _groups(kinds, sizes, len(sizes))
    monkeypatch.setenv("RS_FAULT", "pairs")
    got, ran = _refine(rs, ctx, g, f)
    assert "rf_lvl_pairs" not in ran and "rf_lvl_nn" in ran and "rf_lvl_link" in ran
    pos, vel, box, perm, off = g
    compare_trees(got, oracle_tree_dict(oracle.refine(pos, vel, box, perm, off, f)), box)


def test_a_list_without_memory_is_no_error(monkeypatch):
    """The list's allocation alone fails (the other slots are there from a
    call without the list): the call succeeds and rs_last_error says nothing."""
    from paper_1110_4372_gb300 import rsgpu as rs
    ctx = rs.Context()
    rs.rs_profile_enable(ctx)
    g = _groups(["blob"] * 2, [5000, 3000], 1)
    monkeypatch.setenv("RS_FAULT", "pairs")
    ref, _ = _refine(rs, ctx, g, 0.7)
    monkeypatch.setenv("RS_FAULT", "alloc")
    got, ran = _refine(rs, ctx, g, 0.7)
    assert "rf_lvl_pairs" not in ran
    compare_trees(got, ref, g[2])
    assert rs.lib().rs_last_error(ctx.handle) == b""
