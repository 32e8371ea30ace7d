"""Host-side checks of the plan's kernel queries that need no device."""
import paper_2405_04253_gb300 as fnt


def test_internal_routes_of_a_null_plan():
    L = fnt.lib()
    assert L.fnt_internal_aeq_route(None, 1, 100, 100) == 0 and L.fnt_internal_cdc_route(None, 1) == 0
