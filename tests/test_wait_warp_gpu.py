"""A warp whose lanes see different ends of a bounded wait gives up as one (the kernel that checks it
runs no warp-wide instruction behind the wait, so a split would be reported, not waited for)."""
import pytest

from paper_2501_07047_gb300 import hefx, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lanes", [0xffffffff, 0, 1, 0xfffffffe, 0xffff0000, 0x55555555])
def test_lanes_decide_together(lanes):
    ctx = hefx.hefx_create(0)
    p = hefx.hefx_params_create(ctx, 5, inputs.source_primes(1))
    try:
        hefx.hefx_wait_check_warp(ctx, p, 1_000_000, lanes)
        if lanes == 0xffffffff:
            hefx.hefx_stream_check(ctx, p)
        else:
            with pytest.raises(hefx.HefxError, match=r"code 32\)") as e:
                hefx.hefx_stream_check(ctx, p)
            assert e.value.status == hefx.HEFX_ETIMEOUT
        hefx.hefx_stream_check(ctx, p)  # read and cleared
    finally:
        hefx.hefx_params_destroy(p)
        hefx.hefx_destroy(ctx)
