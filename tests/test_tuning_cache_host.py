"""Host side of the tuning cache (no GPU): an entry is taken only for the sweeps that it was timed on."""
import json

import torch

from paper_1204_2088_gb300 import dscf, inputs


def test_entries_of_earlier_sweeps_are_not_taken(tmp_path, monkeypatch):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda device=None: "a GPU")
    cfgs = [inputs.melt((64, 64, 64), 64, 0.5, 20.0)]
    path = tmp_path / "tuning.json"
    old = json.dumps(["a GPU", dscf.FP32, [[[64, 64, 64], 2, 64]]])    # a key without a revision
    path.write_text(json.dumps({old: [16, 0]}))
    key = dscf._tuning_key(cfgs, dscf.FP32, None)
    assert dscf._tuning_cache_read(str(path)).get(key) is None
    dscf._tuning_cache_write(str(path), key, (8, 1))
    assert dscf._tuning_cache_read(str(path)) == {old: (16, 0), key: (8, 1)}
    monkeypatch.setattr(dscf, "SWEEPS_REVISION", dscf.SWEEPS_REVISION + 1)
    assert dscf._tuning_cache_read(str(path)).get(dscf._tuning_key(cfgs, dscf.FP32, None)) is None
