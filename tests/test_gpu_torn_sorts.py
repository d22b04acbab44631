"""A one-pass sort or scan whose waits for earlier tiles run out leaves part of
its result unwritten.  The injected faults RS_FAULT=wait_<tag> make every wait
of one sort or scan run out at once: the call that holds it reports
RS_ERR_TIMEOUT, nothing uses the incomplete result as an index, and the same
context then gives the results of before."""
import numpy as np
import pytest

from paper_1110_4372_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RS_ERR_TIMEOUT = 4
SIDE = 27      # groups per axis: more of them than a one-block scan or sort takes
LATTICE = 22   # members per axis of the one large group, a single seed of 10,648


def _catalogue():
    rng = np.random.default_rng(11)
    box = 2.0 * SIDE
    at = 2.0 * np.stack(np.meshgrid(*[np.arange(SIDE)] * 3), -1).reshape(-1, 1, 3) + 1.0
    pos = at[1:] + rng.standard_normal((SIDE ** 3 - 1, 12, 3)) * 0.03
    vel = rng.standard_normal(pos.shape) * 30.0
    grid = np.stack(np.meshgrid(*[np.arange(LATTICE)] * 3), -1).reshape(-1, 3) / 32.0 + 0.5
    pos = np.concatenate([grid, pos.reshape(-1, 3)])
    vel = np.concatenate([np.zeros_like(grid), vel.reshape(-1, 3)])
    mix = rng.permutation(len(pos))
    return synth.wrap(pos[mix], box), vel[mix].astype(np.float32), box


@pytest.fixture(scope="module")
def state():
    from paper_1110_4372_gb300 import rsgpu as rs
    pos, vel, box = _catalogue()
    s = dict(rs=rs, ctx=rs.Context(), box=box, p=torch.from_numpy(pos).cuda(), v=torch.from_numpy(vel).cuda())
    s["params"] = rs.params()
    s["labels"] = _fof(s)[0]
    s["perm"], s["off"] = _groups(s)
    s["tree"] = rs.rs_refine6d(s["ctx"], s["p"], s["v"], box, s["perm"], s["off"])
    s["hid"], s["halos"] = rs.rs_assign_ex(s["ctx"], s["tree"], s["p"], s["v"], box, s["params"])
    s["host"] = _props(s)[-1]
    assert s["halos"].n > 16_384 and s["tree"].info().n_nodes > 16_384
    nd = s["tree"].nodes()
    assert int(nd["count"][nd["nchild"] == 0].max()) == LATTICE ** 3
    return s


def _fof(s):
    return [s["rs"].rs_fof3d(s["ctx"], s["p"], s["box"], 0.28, want_groups=True)[0]]


def _accel(s):
    return [s["rs"].rs_fof3d_accel(s["ctx"], s["p"], s["box"], 0.28, 8)[0]]


def _find(s):
    return [s["rs"].rs_find_halos(s["ctx"], s["p"], s["v"], s["box"])[0]]


def _groups(s):
    return list(s["rs"].rs_group_sort(s["ctx"], s["labels"], 10))


def _refine(s):
    t = s["rs"].rs_refine6d(s["ctx"], s["p"], s["v"], s["box"], s["perm"], s["off"])
    return [t.level_labels(k) for k in range(3)]


def _assign(s):
    hid, halos = s["rs"].rs_assign_ex(s["ctx"], s["tree"], s["p"], s["v"], s["box"], s["params"])
    s["rs"].rs_halo_props(s["ctx"], s["tree"], halos, hid)  # synchronises
    return [hid] + [halos.arrays()[k] for k in ("id", "rdyn2")]


def _props(s):
    hp = s["rs"].rs_halo_props(s["ctx"], s["tree"], s["halos"], s["hid"])
    return [hp["n_assigned"], hp["host"]]


def _unbind(s):
    out = s["rs"].rs_unbind(s["ctx"], s["tree"], s["halos"], s["hid"], s["host"], s["p"], s["v"], 1e-3, 0.0, 0.04)
    return [out[k] for k in ("n_part", "n_bound", "bound_own")]


CASES = [(c, t) for c, tags in [
    (_fof, ["sort_fof", "fof_cells"]),
    (_accel, ["sort_fof", "fof_cells"]),
    (_find, ["sort_fof", "fof_cells", "gs_select", "sort_gs", "scan_gs", "sort_kd", "sort_child", "scan_leaf",
             "sort_as", "scan_cand"]),
    (_groups, ["gs_select", "sort_gs", "scan_gs"]),
    (_refine, ["sort_kd", "sort_child"]),
    (_assign, ["scan_leaf", "sort_as", "scan_root", "scan_halo", "scan_large", "sort_rdyn", "scan_tile", "scan_cand"]),
    (_props, ["sort_ids", "sort_hosts"]),
    (_unbind, ["sort_ids", "sort_sets", "scan_tile", "scan_box", "scan_job", "sort_morton"]),
] for t in tags]


@pytest.mark.parametrize("call,tag", CASES, ids=[f"{c.__name__[1:]}-{t}" for c, t in CASES])
def test_incomplete_sorts_and_scans_are_reported(state, monkeypatch, call, tag):
    rs = state["rs"]
    before = call(state)
    monkeypatch.setenv("RS_FAULT", "wait_" + tag)
    with pytest.raises(rs.RsError) as e:
        call(state)
    assert e.value.status == RS_ERR_TIMEOUT
    monkeypatch.delenv("RS_FAULT")
    for a, b in zip(before, call(state)):
        assert torch.equal(a, b)
