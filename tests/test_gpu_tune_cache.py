"""Choices that the tuner saved when the forward shape (1, 4) stood for the library's choice are not
taken up as that shape: the plan is tuned again and the new choice saved beside them."""
import json

import pytest

pytestmark = pytest.mark.gpu


def test_choices_of_another_meaning_are_tuned_again(tmp_path, monkeypatch):
    import torch
    from paper_1810_03275_gb300 import autotune
    from paper_1810_03275_gb300 import ctrecon as ct
    path = tmp_path / "tune.json"
    monkeypatch.setenv("CTR_TUNE_CACHE", str(path))
    device = torch.cuda.get_device_name().replace(" ", "_")
    old = f"plan/{device}/f32/n256/N180/M363"
    plan = ct.Plan(256, 180, 363)
    assert plan.dtype == "f32"
    path.write_text(json.dumps({old: {"bp_groups": 1, "fwd_shape": [1, 4]}}))
    autotune.tune_plan(plan, reps=2)
    saved = json.loads(path.read_text())
    new = [v for k, v in saved.items() if k != old]
    assert len(new) == 1 and tuple(new[0]["fwd_shape"]) == plan.fwd_shape and new[0]["bp_groups"] == plan.bp_groups
