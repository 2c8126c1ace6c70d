"""The autotuner's answers belong to a form of the step: the sweeps have knobs,
a step of one launch has none."""
import pytest

from paper_2006_10142_gb300 import autotune


def test_keys_tell_the_forms_apart():
    plan = dict(form="patches", fp64_x=0, fp64_y=0)
    weak = dict(form="sweeps", fp64_x=0, fp64_y=1)
    forms = [autotune._form(plan, 0), autotune._form(plan, 10), autotune._form(weak, 0)]
    assert forms == ["one launch", "sweeps fp32 fp32", "sweeps fp32 fp64"]
    assert autotune._form(weak, 10) == forms[2]
    keys = {autotune._key("GB300", 700, 500, "auto", f) for f in forms}
    assert len(keys) == 3
    # what an earlier version stored for the shape is not among them
    assert autotune._key("GB300", 700, 500, "auto") not in keys


@pytest.mark.gpu
def test_apply_follows_the_handle(tmp_path, monkeypatch):
    import torch
    from paper_2006_10142_gb300 import api
    monkeypatch.setenv("ADIWAVE_TUNE_CACHE", str(tmp_path / "tune.json"))
    dev = torch.device("cuda:0")
    nx, ny = 700, 500
    knobs = dict(solver=2, chunk_x=32, chunk_y=32)
    name = torch.cuda.get_device_name(dev)
    autotune._store_cache({autotune._key(name, nx, ny, "auto"): dict(tuning=knobs, x_ms=1.0, y_ms=1.0)})
    asked = []

    def candidates(*shape):
        asked.append(shape)
        return [dict(solver=1)], [dict(chunk_x=8), dict(chunk_x=16)], [dict(chunk_y=8), dict(chunk_y=16)]
    monkeypatch.setattr(autotune, "candidates", candidates)
    m = torch.ones(ny, nx, device=dev)

    def handle(cfl):
        return api.AdiWave(m, torch.zeros_like(m), cfl / (nx + 1))

    h = handle(0.5)
    assert h.plan()["form"] == "small_patches" and h.plan()["halo"] == 12
    assert autotune.apply(h)["tuning"] == {}
    assert not asked and h.plan()["form"] == "small_patches"
    h.set_checkpointing(5)  # its runs take the sweeps
    res = autotune.apply(h, steps=2)
    assert len(asked) == 1 and res["x_ms"] > 0 and res["y_ms"] > 0
    h.close()
    h = handle(2.0)
    assert h.plan()["form"] == "sweeps"
    again = autotune.apply(h)  # the same sweeps: from the cache
    assert len(asked) == 1 and again == res
    h.close()
    h = handle(20.0)
    assert h.plan()["fp64_x"] and h.plan()["fp64_y"]
    autotune.apply(h, steps=2)
    assert len(asked) == 2
    h.close()
