"""The refinement's list of pairs is optional memory: a later call that finds
the device full gets it.  (RS_FAULT=full: every allocation's first try fails
for as long as the list is held.)"""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _group(n, seed):
    rng = np.random.default_rng(seed)
    pos = synth.wrap(rng.standard_normal((n, 3)) * 0.15, 20.0)
    vel = (rng.standard_normal((n, 3)) * 60.0).astype(np.float32)
    return pos, vel, np.arange(n, dtype=np.int32), np.array([0, n], np.int64)


def test_the_pair_list_makes_room_for_later_calls(monkeypatch):
    from paper_1110_4372_gb300 import rsgpu as rs
    ctx, box = rs.Context(), 20.0
    pos, vel, perm, off = _group(30_000, 3)
    p, v, m, o = (torch.from_numpy(a).cuda() for a in (pos, vel, perm, off))
    tree = rs.rs_refine6d(ctx, p, v, box, m, o)
    held = rs.rs_workspace_bytes(ctx)
    ref = oracle.refine(pos, vel, box, perm, off)
    hid_o, halos = oracle.assign(ref, len(pos), box, 360.0, len(pos) / box ** 3)
    monkeypatch.setenv("RS_FAULT", "full")
    hid, nh = rs.rs_assign(ctx, tree, p, v, box)  # needs slots that the refinement did not
    assert np.array_equal(hid.cpu().numpy(), hid_o) and nh == len(halos.id)
    assert rs.rs_workspace_bytes(ctx) < held
    tree2 = rs.rs_refine6d(ctx, p, v, box, m, o)  # allocates the list again
    hid, nh = rs.rs_assign(ctx, tree2, p, v, box)
    assert np.array_equal(hid.cpu().numpy(), hid_o) and nh == len(halos.id)
