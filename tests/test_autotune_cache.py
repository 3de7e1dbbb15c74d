"""A tuning entry counts only for the kernels and the GPU that it was measured on."""
import json
from types import SimpleNamespace

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2202_12567_gb300 import autotune


@pytest.fixture
def R(monkeypatch):
    r = SimpleNamespace(smp=SimpleNamespace(ncol=torch.tensor([500, 600])), frame=SimpleNamespace(sizes=np.array([1024, 1100])),
                        cfg=dict(rank=16), ctx=None, dev=0, tuned=0, applied=[])

    def tune(R, **_):
        R.tuned += 1
        return dict(values=dict(als_form=R.tuned), stage_ms={})

    monkeypatch.setattr(autotune, "tune", tune)
    monkeypatch.setattr(autotune.lt, "lt_set_tuning", lambda ctx, **v: r.applied.append(v))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev: "one GPU")
    return r


def test_other_kernels_or_gpu_are_tuned_again(R, tmp_path, monkeypatch):
    path = str(tmp_path / "cache.json")
    key, values, cached = autotune.apply(R, "w", path)
    assert not cached and values == dict(als_form=1)
    assert autotune.apply(R, "w", path) == (key, dict(als_form=1), True) and R.tuned == 1
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev: "another GPU")
    assert autotune.apply(R, "w", path) == (key, dict(als_form=2), False)
    monkeypatch.setattr(autotune, "HERE", str(tmp_path))
    (tmp_path / "csrc").mkdir()
    (tmp_path / "csrc" / "a.cu").write_text("one kernel")
    assert not autotune.apply(R, "w", path)[2]
    assert autotune.apply(R, "w", path)[2]
    (tmp_path / "csrc" / "a.cu").write_text("a kernel changed since")
    assert not autotune.apply(R, "w", path)[2]


def test_an_entry_that_names_neither_is_not_used(R, tmp_path):
    path = tmp_path / "cache.json"
    key = autotune.workload_key("w", 16, R.frame.sizes, [500, 600])
    path.write_text(json.dumps({key: dict(values=dict(als_form=9), stage_ms={})}))
    assert autotune.apply(R, "w", str(path)) == (key, dict(als_form=1), False) and not R.applied
    assert json.loads(path.read_text())[key]["made_for"]["gpu"] == "one GPU"
