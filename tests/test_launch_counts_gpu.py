"""The launch counts of HE-Mult and of a batch plan equal the kernel nodes of the captured call."""
import pytest
import torch

from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult

from graph_util import kernel_blocks

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


def buffer(*shape):
    return torch.zeros(shape, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("logn,L,K,alpha,bconv", [(8, 6, 4, 4, "auto"), (12, 9, 3, 3, "tensor"), (14, 6, 2, 2, "auto"),
                                                  (15, 6, 2, 2, "cudacore"), (16, 12, 4, 4, "auto")])
def test_he_mult(ctx, logn, L, K, alpha, bconv):
    n = 1 << logn
    hm = HeMult(ctx, logn, inputs.source_primes(L), inputs.special_primes(K), alpha, bconv_path=bconv)
    try:
        ins, evk = [buffer(L, n) for _ in range(4)], buffer(hm.dnum, 2, L + K, n)
        c, out = buffer(2, L, n), buffer(2, L - 1, n)
        assert len(kernel_blocks(lambda s: hm.run(*ins, evk, out, s))) == hm.launches(captured=True)
        assert len(kernel_blocks(lambda s: hm.run(*ins, evk, c, s, rescale=False))) == hm.launches(False, captured=True)
        assert len(kernel_blocks(lambda s: hm.rescale(c, out, s))) == hm.rescale_launches(captured=True)
        few = logn == 15 and hm.dnum * (L + K) <= 32  # the only form that differs outside a graph
        assert hm.launches() == hm.launches(captured=True) - (1 if few else 0)
    finally:
        hm.close()


@pytest.mark.parametrize("jobs", [[(28, 12, 3), (28, 16, 2)], [(30, 9, 2), (28, 14, 3), (30, 15, 1), (30, 14, 2), (28, 17, 1)]])
@pytest.mark.parametrize("squares", [False, True])
def test_batch_plan(ctx, jobs, squares):
    held, entries = [], []
    for bits, logn, L in jobs:
        p = hefx.hefx_params_create(ctx, logn, inputs.ntt_primes(L, bits, 2 << logn))
        a, b, c = (buffer(L, 1 << logn) for _ in range(3))
        held.append((p, a, b, c))
        entries.append((p, L, a, a if squares else b, c))
    plan = hefx.hefx_batch_plan_create(ctx, entries)
    try:
        assert len(kernel_blocks(lambda s: hefx.hefx_batch_polymul(ctx, plan, s))) == hefx.hefx_batch_plan_launches(plan)
    finally:
        hefx.hefx_batch_plan_destroy(plan)
        for p, *_ in held:
            hefx.hefx_params_destroy(p)
