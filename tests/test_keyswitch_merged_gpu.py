"""The inner product that scales and adds, and the ModDown of scaled limbs: together with the
inverse transform between them they equal ModDown(INTT(sum)) + INTT(add) bit for bit, on the tensor-core
conversion and on the CUDA-core one (few special limbs, one tile and less)."""
import numpy as np
import pytest

import oracle
from paper_2501_07047_gb300 import hefx, inputs

from hefx_testutil import to_dev as dev, to_host as host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn,L,K,dnum,batch", [(5, 2, 1, 1, 1), (7, 9, 4, 3, 2), (9, 3, 2, 2, 3), (12, 17, 5, 4, 1)])
def test_scaled_and_added(logn, L, K, dnum, batch):
    ctx = hefx.hefx_create(0)
    n = 1 << logn
    qs, ps = list(inputs.source_primes(L)), list(inputs.special_primes(K))
    qp = qs + ps
    p = hefx.hefx_params_create(ctx, logn, qp)
    plan = hefx.hefx_bconv_plan_create(ctx, logn, ps, qs)
    try:
        dig, evk = (np.stack([inputs.residue_tensor(inputs.derive_seed(81, k, b), m, qp, n) for b in range(c)])
                    for k, m, c in ((0, dnum, batch), (1, 2, dnum)))
        add = np.stack([inputs.residue_tensor(inputs.derive_seed(82, b), 2, qs, n) for b in range(batch)])
        dig[..., 0], evk[..., 0] = (np.asarray(qp, dtype=np.uint32) - 1,) * 2
        add[..., 0] = np.asarray(qs, dtype=np.uint32) - 1
        dout = dev(np.full((batch, 2, L + K, n), 0xFFFFFFFF, dtype=np.uint32))
        dc = dev(np.full((2 * batch, L, n), 0xFFFFFFFF, dtype=np.uint32))
        hefx.hefx_key_inner_product_add(ctx, p, plan, dev(dig), dev(evk), dev(add), dout, dnum, batch)
        hefx.hefx_ntt_inv(ctx, p, dout, 2 * batch)
        hefx.hefx_mod_down_scaled(ctx, plan, dout, dc, 2 * batch)
        hefx.hefx_bconv_check(ctx, plan)
        got = host(dc).reshape(batch, 2, L, n)
        q = np.asarray(qs, dtype=np.uint64)[None, :, None]
        for b in range(batch):
            acc = oracle.ntt_batch(oracle.key_inner_product(dig[b], evk, qp), qp, inverse=True)
            want = oracle.moddown(acc, qs, ps).astype(np.uint64) + oracle.ntt_batch(add[b], qs, inverse=True)
            assert np.array_equal(got[b], (want % q).astype(np.uint32))
        other = hefx.hefx_bconv_plan_create(ctx, logn, qs, ps)  # the wrong way round
        assert hefx.raw_status("hefx_key_inner_product_add", ctx, p, other, dout.data_ptr(), dout.data_ptr(),
                               dout.data_ptr(), dc.data_ptr(), 1, 0, 0) == hefx.HEFX_EINVAL
        hefx.hefx_bconv_plan_destroy(other)
    finally:
        hefx.hefx_bconv_plan_destroy(plan)
        hefx.hefx_params_destroy(p)
        hefx.hefx_destroy(ctx)
