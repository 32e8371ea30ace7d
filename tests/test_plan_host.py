"""Host-side checks of the plan's settings and kernel queries that need no device."""
import os
import re

import pytest

import paper_2405_04253_gb300 as fnt

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_internal_routes_of_a_null_plan():
    L = fnt.lib()
    assert L.fnt_internal_aeq_route(None, 1, 100, 100) == 0 and L.fnt_internal_cdc_route(None, 1) == 0


@pytest.mark.parametrize("setter,needs", [("set_launch", "set_aeq_kernel"), ("set_launch", "set_cdc_kernel"),
                                          ("set_aeq_occupancy", "set_aeq_kernel"),
                                          ("set_cdc_items", "set_cdc_kernel"),
                                          ("set_tensor_gradient", "set_aeq_kernel")])
def test_transform_settings_say_which_kernel_they_need(setter, needs):
    """A setting that the default kernels do not have names, in its own entry of the
    header and in its docstring, the setter that picks a kernel which does."""
    with open(os.path.join(ROOT, "include", "fnt.h")) as fh:
        text = fh.read()
    entry = re.search(r"/\*(?:(?!\*/).)*\*/\s*FNT_API fnt_status fnt_plan_%s\(" % setter, text, re.S).group(0)
    assert "fnt_plan_" + needs in entry and "direct form" in entry
    doc = getattr(fnt.Plan, setter).__doc__ or ""
    assert needs in doc and "direct" in doc


class _FakePlan:
    """The calls of a plan that the autotuner makes, without a device."""

    def __init__(self, cdc, aeq):
        from types import SimpleNamespace
        self.desc = SimpleNamespace(n_aeq=32, aeq_segment=0, aeq_warmup=0, aeq_update_period=1)
        self.routes, self.calls = (cdc, aeq), []

    def cdc_route(self, n_items=1):
        return self.routes[0]

    def aeq_route(self, n_chains, total, longest):
        return self.routes[1]

    def set_launch(self, cdc_warps=0, aeq_warps=0):
        self.calls.append(("launch", cdc_warps, aeq_warps))

    def set_aeq_occupancy(self, warps):
        self.calls.append(("occupancy", warps))


@pytest.mark.parametrize("cdc", ["cdc_direct_kernel", "cdc_kernel", "cdc_split_kernel"])
@pytest.mark.parametrize("aeq", ["aeq_duo_kernel", "aeq_split_kernel", "aeq_kernel", "aeq_serial_kernel"])
@pytest.mark.parametrize("op", [fnt.OP_CDC, fnt.OP_AEQ, fnt.OP_CHAIN])
def test_autotune_tunes_only_kernels_with_launch_settings(monkeypatch, tmp_path, cdc, aeq, op):
    """Stages in direct form are timed once and nothing is set, kept or called tuned
    for them; stages in the tunable transform kernels try their candidates."""
    import torch
    from types import SimpleNamespace
    from paper_2405_04253_gb300 import autotune
    timed = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: None)
    monkeypatch.setattr(autotune, "Batch", lambda *a, **k: SimpleNamespace(close=lambda: None))
    monkeypatch.setattr(autotune, "_time_stage", lambda b, stage, reps, s: timed.append(stage) or 1.0 / len(timed))
    plan, cache = _FakePlan(cdc, aeq), str(tmp_path / "shapes.json")
    frames = [SimpleNamespace(n=5000)]
    best = autotune.tune(plan, frames, op, cache=cache)
    tunes = [s for s, name, has in (("cdc", cdc, op != fnt.OP_AEQ), ("aeq", aeq, op != fnt.OP_CDC))
             if has and name in ("cdc_kernel", "aeq_kernel")]
    assert best["tuned"] == tunes
    assert timed.count(0) == (0 if op == fnt.OP_AEQ else 4 if "cdc" in tunes else 1)
    assert timed.count(1) == (0 if op == fnt.OP_CDC else 16 if "aeq" in tunes else 1)
    assert bool(plan.calls) == bool(tunes) == os.path.exists(cache)
    assert all(c[1] == 0 for c in plan.calls if c[0] == "launch") or "cdc" in tunes
    assert all(c[0] == "launch" and c[2] == 0 for c in plan.calls) or "aeq" in tunes
    # the second call takes the stages' shapes from the cache and sets the same
    timed.clear()
    again = _FakePlan(cdc, aeq)
    second = autotune.tune(again, frames, op, cache=cache)
    if tunes:
        assert second == best and not timed
        assert again.calls == plan.calls[-len(again.calls):]
    else:
        assert not again.calls
