"""The refinement screens pairs by half-precision products: big nodes leaf
against leaf (32 members a leaf), small ones by tiles of 16 x 8 pairs in one
block.  Node sizes at the edges of leaves, tiles and tiers, and inputs that
leave the screen's range (boxes far larger than the linking length, a zero
linking length) or that the clique boxes serve (dense cores, copies).  Trees
and tie counts must equal the float64 oracle's exactly."""
import numpy as np
import pytest

from paper_1110_4372_gb300 import synth

from gpu_util import gpu_tree_dict, oracle_tree_dict, run_gpu_path, run_oracle_path

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _members(kind, n, rng):
    """Positions around 0 (spread about 0.15, one 3D group at l = 0.4 or more) and velocities of one group."""
    if kind == "blob":
        return rng.standard_normal((n, 3)) * 0.15, rng.standard_normal((n, 3)) * 60.0
    if kind == "pairs":  # close pairs: boxes of thousands of linking lengths
        p, v = np.repeat(rng.standard_normal((n // 2 + 1, 3)) * 0.15, 2, 0), np.repeat(
            rng.standard_normal((n // 2 + 1, 3)) * 60.0, 2, 0)
        p[1::2] += rng.standard_normal((n // 2 + 1, 3)) * 1e-6
        return p[:n], v[:n]
    if kind == "copies":  # most members on a few points: l = 0
        p, v = rng.standard_normal((n, 3)) * 0.15, rng.standard_normal((n, 3)) * 60.0
        at = rng.integers(0, 5, n)
        few = rng.random(n) < 0.8
        p[few], v[few] = p[:5][at[few]], v[:5][at[few]]
        return p, v
    if kind == "core":  # a core far denser than the linking length
        p, v = rng.standard_normal((n, 3)) * 0.15, rng.standard_normal((n, 3)) * 60.0
        c = rng.random(n) < 0.5
        p[c] *= 1e-3
        v[c] *= 1e-3
        return p, v
    if kind == "still":  # no velocity dispersion: its term is dropped
        return rng.standard_normal((n, 3)) * 0.15, np.full((n, 3), 7.0)
    raise ValueError(kind)


@pytest.mark.parametrize("kind,n,f", [
    ("blob", 1025, 0.7), ("blob", 1055, 0.7), ("blob", 1057, 0.5), ("blob", 2049, 0.9), ("blob", 4097, 0.7),
    ("blob", 33_000, 0.7), ("pairs", 1500, 0.7), ("pairs", 5001, 0.9), ("copies", 1500, 0.7), ("copies", 6000, 0.5),
    ("core", 3000, 0.7), ("core", 6001, 0.9), ("still", 1100, 0.7), ("still", 5000, 0.7)])
def test_leaf_searches_match_oracle(kind, n, f):
    rng = np.random.default_rng([n, len(kind)])
    box = 20.0
    p, v = _members(kind, n, rng)
    # one corner of the box, so that the group wraps
    cat = synth.Catalogue(pos=synth.wrap(p, box), vel=v.astype(np.float32), box=box, truth=np.zeros(n, np.int32),
                          comp_parent=np.zeros(0, np.int32), comp_n=np.zeros(0))
    o = _check(cat, f)
    assert np.diff(o["offsets"]).max() > 1024


@pytest.mark.parametrize("kind", ["blob", "pairs", "copies", "core", "still"])
@pytest.mark.parametrize("f", [0.5, 0.7])
def test_subtree_tiers_match_oracle(kind, f):
    rng = np.random.default_rng([7, len(kind)])
    sizes = [10, 11, 31, 32, 33, 34, 47, 48, 49, 63, 65, 127, 128, 129, 255, 256, 257, 258, 272, 273, 500, 511, 513,
             777, 1008, 1009, 1023, 1024]
    box = 40.0
    parts = [_members(kind, k, rng) for k in sizes]
    at = np.stack(np.meshgrid(*[np.arange(4) * 10.0] * 3), -1).reshape(-1, 3)[:len(sizes)]
    p = np.vstack([q[0] + c for q, c in zip(parts, at)])
    v = np.vstack([q[1] for q in parts])
    mix = rng.permutation(len(p))
    cat = synth.Catalogue(pos=synth.wrap(p[mix], box), vel=v[mix].astype(np.float32), box=box,
                          truth=np.zeros(len(p), np.int32), comp_parent=np.zeros(0, np.int32), comp_n=np.zeros(0))
    o = _check(cat, f)
    assert o["tree"].n_nodes >= 20


def _check(cat, f):
    from paper_1110_4372_gb300 import rsgpu
    b = 0.4 * cat.n ** (1 / 3) / cat.box
    g = run_gpu_path(rsgpu.Context(), rsgpu, cat, f=f, b=b, assign=False)
    o = run_oracle_path(cat, f=f, b=b, assign=False)
    # what the searches decide (the moments of a core of 1e-4 Mpc/h reach the
    # fixed-point sums' resolution, 2^-32)
    gd, od = gpu_tree_dict(g["tree"]), oracle_tree_dict(o["tree"])
    assert set(gd) == set(od)
    for k, a in gd.items():
        for q in ("members", "parent_key", "nchild", "tie"):
            assert a[q] == od[k][q], (k, q)
        assert abs(a["lnk"] - od[k]["lnk"]) <= 1e-6 * od[k]["lnk"], k
    return o
