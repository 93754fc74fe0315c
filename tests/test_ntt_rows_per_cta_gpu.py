"""Launches whose rows per CTA, register budget or number of launches depend on the row count: every
transform and product equals the same call on one polynomial at a time (one row per CTA), the
product also its three separate steps and, on the first and last polynomial, the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_07047_gb300 import hefx, inputs

from hefx_testutil import to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


@pytest.mark.parametrize("bits,logn,L,batch", [
    (28, 3, 1, 1), (28, 3, 3, 53), (30, 5, 1, 155), (28, 8, 5, 61), (28, 10, 1, 152), (28, 10, 2, 77), (30, 10, 7, 180),
    (28, 11, 3, 1), (28, 11, 1, 153), (30, 11, 1, 609), (28, 11, 1, 1217), (28, 12, 1, 1), (28, 12, 1, 153),
    (28, 12, 1, 336), (30, 12, 1, 609), (28, 13, 1, 1), (30, 13, 5, 61), (28, 14, 1, 1), (30, 14, 1, 128),
    (28, 14, 1, 129), (28, 15, 2, 3), (28, 16, 1, 3), (30, 16, 3, 1), (28, 17, 2, 2)])
def test_rows(ctx, bits, logn, L, batch):
    n = 1 << logn
    primes = inputs.ntt_primes(L, bits, 2 << logn)
    p = hefx.hefx_params_create(ctx, logn, primes)
    try:
        g = torch.Generator(device="cuda").manual_seed(logn * 4096 + batch)
        q = torch.tensor(primes, device="cuda").view(1, L, 1)
        x, y = ((torch.randint(0, 1 << 30, (batch, L, n), generator=g, device="cuda") % q).int() for _ in range(2))
        x[..., 0], y[..., 0] = (q[..., 0] - 1).int(), (q[..., 0] - 1).int()

        def mul(a, b, c):
            hefx.hefx_poly_mul(ctx, p, a, b, c, c.shape[0])
            return c

        fx, fy, ix = x.clone(), y.clone(), x.clone()
        hefx.hefx_ntt_fwd(ctx, p, fx, batch)
        hefx.hefx_ntt_fwd(ctx, p, fy, batch)
        hefx.hefx_ntt_inv(ctx, p, ix, batch)
        steps = torch.empty_like(x)
        hefx.hefx_ntt_inv_hadamard(ctx, p, fx, fy, steps, batch)
        assert torch.equal(mul(x, y, torch.empty_like(x)), steps)
        xa, yb = x.clone(), y.clone()
        assert torch.equal(mul(xa, y, xa), steps) and torch.equal(mul(x, yb, yb), steps)
        for b in sorted({0, 1, batch // 2, batch - 2, batch - 1} & set(range(batch))):
            one, inv = x[b:b + 1].clone(), x[b:b + 1].clone()
            hefx.hefx_ntt_fwd(ctx, p, one, 1)
            hefx.hefx_ntt_inv(ctx, p, inv, 1)
            assert torch.equal(one[0], fx[b]) and torch.equal(inv[0], ix[b])
            assert torch.equal(mul(x[b:b + 1].clone(), y[b:b + 1].clone(), one)[0], steps[b])
        for b in {0, batch - 1}:
            hx, hy = to_host(x[b:b + 1].contiguous()), to_host(y[b:b + 1].contiguous())
            assert np.array_equal(to_host(fx[b]), oracle.ntt_batch(hx, primes)[0])
            assert np.array_equal(to_host(ix[b]), oracle.ntt_batch(hx, primes, inverse=True)[0])
            assert np.array_equal(to_host(steps[b]), oracle.polymul_batch(hx, hy, primes)[0])
        hefx.hefx_stream_check(ctx, p)
    finally:
        hefx.hefx_params_destroy(p)
