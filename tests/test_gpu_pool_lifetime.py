"""Contexts destroyed before the trees and halo tables that they made (as a
collector may order it): the blocks stay valid, are freed afterwards in any
order, and other contexts are untouched."""
import random

import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

from gpu_util import cuda_inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_contexts_go_before_their_trees(seed):
    from paper_1110_4372_gb300 import rsgpu as rs
    c = synth.generate("c1")
    o = oracle.run_all(c.pos, c.vel, c.box)
    pos, vel = cuda_inputs(c)
    labels = torch.from_numpy(o["labels"]).cuda()
    order = random.Random(seed)
    kept = rs.Context()
    for _ in range(4):
        made = []
        for _ in range(3):
            ctx = rs.Context()
            rs.rs_profile_enable(ctx)
            perm, off = rs.rs_group_sort(ctx, labels)
            tree = rs.rs_refine6d(ctx, pos, vel, c.box, perm, off)
            hid, halos = rs.rs_assign_ex(ctx, tree, pos, vel, c.box)
            assert np.array_equal(hid.cpu().numpy(), o["halo_id"])
            made.append([ctx.close, tree.free, halos.__del__])
        for m in made:
            m[0]()  # the context first
        rest = [f for m in made for f in m[1:]]
        order.shuffle(rest)
        for f in rest:
            f()
            hid, _, _ = rs.rs_find_halos(kept, pos, vel, c.box)
            assert np.array_equal(hid.cpu().numpy(), o["halo_id"])
