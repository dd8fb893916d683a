"""The autotuner leaves the configuration alone for batches whose products do not use one."""
import json
import os
import re

from paper_1510_04686_gb300 import autotune, negf as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_large_batches_neither_tune_nor_apply_a_record(monkeypatch, tmp_path):
    calls = []

    def tc_config(idx=None):
        calls.append(idx)
        return 20

    monkeypatch.setattr(B, "tc_config", tc_config)
    monkeypatch.setattr(B, "tc_config_count", lambda: 26)
    monkeypatch.setattr(autotune, "_key", lambda b, n: str(tmp_path / f"{b}_{n}.json"))
    for n in (B.RESIDUE_ITEMS, 256):
        # a record of an earlier run, when such batches were tuned too
        (tmp_path / f"400_{n}.json").write_text(json.dumps(
            {"b": 400, "batch": n, "config": 4, "n_configs": 26}))
        assert autotune.tune_tc(400, n)["config"] == 20
    assert set(calls) == {None}
    n = B.RESIDUE_ITEMS - 1
    (tmp_path / f"400_{n}.json").write_text(json.dumps(
        {"b": 400, "batch": n, "config": 4, "n_configs": 26}))
    assert autotune.tune_tc(400, n)["config"] == 4
    assert calls[-1] == 4


def test_the_batch_is_the_librarys():
    with open(os.path.join(ROOT, "include", "negf.h")) as fh:
        assert re.search(rf"#define NEGF_RESIDUE_ITEMS {B.RESIDUE_ITEMS}\b", fh.read())
