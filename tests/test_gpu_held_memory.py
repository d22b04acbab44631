"""rs_workspace_bytes counts what the context holds: its workspace, and a freed
tree's memory as long as the pool keeps it."""
import numpy as np
import pytest

from paper_1110_4372_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_a_freed_trees_memory_is_counted():
    from paper_1110_4372_gb300 import rsgpu as rs
    rng = np.random.default_rng(8)
    n, box = 100_000, 20.0
    pos = torch.from_numpy(synth.wrap(rng.standard_normal((n, 3)) * 0.15, box)).cuda()
    vel = torch.from_numpy((rng.standard_normal((n, 3)) * 60.0).astype(np.float32)).cuda()
    perm = torch.arange(n, dtype=torch.int32, device="cuda")
    off = torch.tensor([0, n], dtype=torch.int64, device="cuda")
    ctx = rs.Context()
    tree = rs.rs_refine6d(ctx, pos, vel, box, perm, off)
    held = rs.rs_workspace_bytes(ctx)
    tree.free()
    freed = rs.rs_workspace_bytes(ctx)
    assert freed >= held + 4 * n  # the member list alone
    tree = rs.rs_refine6d(ctx, pos, vel, box, perm, off)
    assert rs.rs_workspace_bytes(ctx) == held
    tree.free()
    assert rs.rs_workspace_bytes(ctx) == freed
