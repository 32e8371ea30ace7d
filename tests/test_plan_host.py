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
