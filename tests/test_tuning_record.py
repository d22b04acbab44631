"""A tuner record made when a launch choice meant something else does not set
that choice; a record of today sets every one."""
import json

import pytest

pytest.importorskip("torch")

TUNED = dict(link_blocks_per_sm=6, nn_blocks_per_sm=5, kd_levels=2, bracket_min=8192, mid_max=192, tiny_max=24,
             small_ctas_per_sm=1, mid_ctas_per_sm=6, tiny_ctas_per_sm=12, fof_link_ctas_per_sm=16)


@pytest.mark.parametrize("meaning,left", [(None, {"link_blocks_per_sm", "bracket_min"}), (2, set())])
def test_records_set_what_they_mean(monkeypatch, tmp_path, meaning, left):
    from paper_1110_4372_gb300 import rsgpu
    got = {}
    monkeypatch.setattr(rsgpu, "rs_set_tuning", lambda ctx, **fields: got.update(fields))
    rec = dict(tuned=TUNED) if meaning is None else dict(meaning=meaning, tuned=TUNED)
    path = tmp_path / "record.json"
    path.write_text(json.dumps(rec))
    rsgpu.apply_tuning(None, str(path))
    assert got == {k: v for k, v in TUNED.items() if k not in left}


def test_the_tuner_writes_todays_meaning():
    from paper_1110_4372_gb300 import rsgpu
    assert rsgpu.TUNING_MEANING not in rsgpu.TUNING_CHANGED
    assert set(f for c in rsgpu.TUNING_CHANGED.values() for f in c) <= set(rsgpu.rs_tuning_default())
