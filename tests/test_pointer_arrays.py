"""The binding's pointer-array parameters take any ctypes array of addresses."""
import ctypes

import pytest

from paper_2311_15429_gb300 import rp


@pytest.mark.parametrize("item", [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_int64, ctypes.c_size_t,
                                  ctypes.POINTER(ctypes.c_float)])
def test_arrays_of_addresses_reach_the_library(item):
    ctx = rp.rp_create(137.0, 0.05, flags=rp.RP_FLAG_PLAN_ONLY)
    try:
        rp.rp_add_domain(ctx, (0.0, 0.0, 0.0), (4, 4, 4), 0.3)
        rp.rp_finalize(ctx)
        for call in (rp.rp_push_all, rp.rp_evaluate, rp.rp_push_all_host, rp.rp_evaluate_host):
            with pytest.raises(rp.RPError) as e:     # past the binding: the context only plans
                call(ctx, (item * 1)(), (item * 1)())
            assert e.value.status == rp.RP_ERR_STATE
    finally:
        rp.rp_destroy(ctx)


def test_arrays_of_other_things_are_refused():
    with pytest.raises(ValueError):
        rp.rp_push_all(None, (ctypes.c_float * 2)(), (ctypes.c_float * 2)())
