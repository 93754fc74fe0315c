"""HeMult.check on the device: clean after runs, an expired wait of one of its parameter sets is reported once."""
import pytest
import torch

from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bconv", ["auto", "tensor", "cudacore"])
def test_check(bconv):
    ctx = hefx.hefx_create(0)
    logn, L, K, alpha = 8, 6, 4, 4
    hm = HeMult(ctx, logn, inputs.source_primes(L), inputs.special_primes(K), alpha, bconv_path=bconv)
    try:
        ins = [torch.zeros((L, 1 << logn), dtype=torch.int32, device="cuda") for _ in range(4)]
        evk = torch.zeros((hm.dnum, 2, L + K, 1 << logn), dtype=torch.int32, device="cuda")
        hm.run(*ins, evk, torch.zeros((2, L - 1, 1 << logn), dtype=torch.int32, device="cuda"))
        hm.check()
        hefx.hefx_wait_check(ctx, hm.pQP, 1_000_000, arrive=False)  # nothing arrives: gives up after 1 ms
        with pytest.raises(hefx.HefxError) as e:
            hm.check()
        assert e.value.status == hefx.HEFX_ETIMEOUT
        hm.check()
    finally:
        hm.close()
        hefx.hefx_destroy(ctx)
