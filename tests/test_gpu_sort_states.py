"""The one-pass sort above 8192 keys at the edges of its tiles of 4096 keys,
with 32-bit tile states and with the 64-bit ones that 2^30 keys and more take
(RS_FAULT=sort64: at any size): 64-bit keys through the 3D labels, 32-bit ones
through the group list."""
import numpy as np
import pytest

import oracle
from paper_1110_4372_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [8193, 12_287, 12_288, 12_289, 65_536, 300_007])
@pytest.mark.parametrize("fault", ["", "sort64"])
def test_sorts_match_oracle(monkeypatch, n, fault):
    from paper_1110_4372_gb300 import rsgpu
    monkeypatch.setenv("RS_FAULT", fault)
    ctx = rsgpu.Context()
    c = synth.uniform(n, 20.0, n)
    lab, ng, _ = rsgpu.rs_fof3d(ctx, torch.from_numpy(c.pos).cuda(), c.box, 0.28, want_groups=True)
    ref, _, _ = oracle.fof3d(c.pos, c.box, 0.28)
    assert np.array_equal(lab.cpu().numpy(), ref) and ng == len(np.unique(ref))
    perm, off = rsgpu.rs_group_sort(ctx, lab, 1)
    m, o = oracle.groups_from_labels(ref, 1)
    assert np.array_equal(perm.cpu().numpy(), m) and np.array_equal(off.cpu().numpy(), o)


def test_whole_path_with_64_bit_states(monkeypatch):
    from paper_1110_4372_gb300 import rsgpu
    n = 100_003
    c = synth.generate("c1", seed=9, n=n, box=10.0 * (n / 32768) ** (1 / 3), n_halos=60)
    monkeypatch.setenv("RS_FAULT", "sort64")
    hid, _, _ = rsgpu.rs_find_halos(rsgpu.Context(), *(torch.from_numpy(a).cuda() for a in (c.pos, c.vel)), c.box)
    assert np.array_equal(hid.cpu().numpy(), oracle.run_all(c.pos, c.vel, c.box)["halo_id"])


def test_torn_64_bit_states_are_reported(monkeypatch):
    from paper_1110_4372_gb300 import rsgpu
    c = synth.uniform(20_000, 20.0, 1)
    pos = torch.from_numpy(c.pos).cuda()
    ctx = rsgpu.Context()
    monkeypatch.setenv("RS_FAULT", "sort64,wait_sort_fof")
    with pytest.raises(rsgpu.RsError) as e:
        rsgpu.rs_fof3d(ctx, pos, c.box, 0.28, want_groups=True)
    assert e.value.status == 4  # RS_ERR_TIMEOUT
