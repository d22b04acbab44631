"""The one-pass scans and sorts behind the calls, at the edges of their tiles
(2048 sorted keys, 4096 scanned words, 16,384 counted particles) and of the
one-block variants (8192 keys, 16,384 words): 3D labels and group lists of
random boxes against plain NumPy on the oracle's labels."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [2047, 2048, 2049, 4096, 4097, 8191, 8192, 8193, 16_384, 16_385, 40_961])
@pytest.mark.parametrize("b", [0.28, 0.9])
def test_fof_and_groups_at_tile_edges(n, b):
    from paper_1110_4372_gb300 import rsgpu
    ctx = rsgpu.Context()
    c = synth.uniform(n, 20.0, n)
    lab, ng, _ = rsgpu.rs_fof3d(ctx, torch.from_numpy(c.pos).cuda(), c.box, b, want_groups=True)
    ref, _, _ = oracle.fof3d(c.pos, c.box, b)
    assert np.array_equal(lab.cpu().numpy(), ref) and ng == len(np.unique(ref))
    for min_n in (1, 2, 10):
        perm, off = rsgpu.rs_group_sort(ctx, lab, min_n)
        m, o = oracle.groups_from_labels(ref, min_n)
        assert np.array_equal(perm.cpu().numpy(), m) and np.array_equal(off.cpu().numpy(), o), min_n


def test_labels_of_a_clustered_box_are_roots():
    """Every label is the smallest index of its group, in a box whose groups span many cells (the labels read the
    cells' parents directly): against the oracle, and the same labels in repeated calls."""
    from paper_1110_4372_gb300 import rsgpu
    n = 400_001
    c = synth.generate("c2", seed=5, n=n, box=10.0 * (n / 32768) ** (1 / 3), n_halos=480)
    ref, _, _ = oracle.fof3d(c.pos, c.box, 0.28)
    ctx, pos = rsgpu.Context(), torch.from_numpy(c.pos).cuda()
    for _ in range(20):
        lab, _, _ = rsgpu.rs_fof3d(ctx, pos, c.box, 0.28)
        assert np.array_equal(lab.cpu().numpy(), ref)


@pytest.mark.parametrize("n,groups", [(300_001, 1), (300_001, 3), (1_000_003, 70_000), (2_500_000, 2_500_000)])
def test_group_sort_of_synthetic_labels(n, groups):
    """Labels drawn directly: one huge group, a few, many, and singletons only."""
    from paper_1110_4372_gb300 import rsgpu
    rng = np.random.default_rng(groups)
    g = rng.integers(0, groups, n) if groups < n else np.arange(n)
    first = np.full(groups, n, np.int64)
    np.minimum.at(first, g, np.arange(n))
    lab = first[g].astype(np.int32)
    ctx = rsgpu.Context()
    for min_n in (1, 12):
        perm, off = rsgpu.rs_group_sort(ctx, torch.from_numpy(lab).cuda(), min_n)
        m, o = oracle.groups_from_labels(lab, min_n)
        assert np.array_equal(perm.cpu().numpy(), m) and np.array_equal(off.cpu().numpy(), o), min_n
