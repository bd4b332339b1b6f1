"""The autotuner's cache: a record is used for the kernels it was measured on
and no others."""
import json
import os
import shutil

import pytest

torch = pytest.importorskip("torch")

from paper_1808_03801_gb300 import autotune, build, workloads as W


def test_records_of_other_kernels_are_not_used(monkeypatch, tmp_path):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "GPU")
    monkeypatch.setattr(autotune, "CACHE", str(tmp_path / "cache.json"))
    w = W.cavity(n=200, ppc=100)
    w["params"]["pipeline"] = "fused"
    src = tmp_path / "csrc"
    shutil.copytree(build.CSRC, src)
    monkeypatch.setattr(build, "CSRC", str(src))
    record = {"fused_R": 8, "grid_per_sm": 8, "s_per_step": 1.0, "tried": []}
    before = autotune._key(w, "GPU")
    without_source = before.rsplit("|", 1)[0]
    with open(autotune.CACHE, "w") as f:
        json.dump({before: record, "batch:3:" + before: record, without_source: dict(record, fused_R=12)}, f)
    assert autotune.tune(w) == record and autotune.tune_batch([w] * 3) == record
    with open(os.path.join(src, "usp_fused.cu"), "a") as f:
        f.write("\n")

    def measured(*a, **k):
        raise LookupError("measured again")

    from paper_1808_03801_gb300 import usp as U
    monkeypatch.setattr(U, "Simulation", measured)
    for call in (lambda: autotune.tune(w), lambda: autotune.tune_batch([w] * 3)):
        with pytest.raises(LookupError):
            call()
