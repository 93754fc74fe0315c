"""The two-pass schedule where AUTO takes it (N = 2^14 .. 2^17): equal to the cluster schedule, word for
word, for every form of the call (forward, inverse, inverse of a Hadamard product,
rescaling forward), at one row, ragged counts and both sides of AUTO's lines; and
to the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_07047_gb300 import hefx, inputs

from hefx_testutil import empty_dev, to_dev, to_host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


def forms(ctx, p, x, y, L, batch, n):
    """Every non-plan form on device copies of x, y: a list of device results."""
    f, i = x.clone(), x.clone()
    hefx.hefx_ntt_fwd(ctx, p, f, batch)
    hefx.hefx_ntt_inv(ctx, p, i, batch)
    h = torch.empty_like(x)
    hefx.hefx_ntt_inv_hadamard(ctx, p, x, y, h, batch)
    out = [f, i, h]
    if L > 1:
        r = empty_dev((batch, L - 1, n))
        hefx.hefx_rescale_ntt(ctx, p, x, r, batch)
        out.append(r)
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("bits", [28, 30])
@pytest.mark.parametrize("logn,L,batch", [(14, 1, 1), (14, 3, 5), (15, 1, 1), (15, 5, 3), (16, 1, 1), (16, 3, 3),
                                          (17, 1, 1), (17, 2, 3)])
def test_forms_against_cluster_and_oracle(ctx, bits, logn, L, batch):
    n = 1 << logn
    primes = inputs.ntt_primes(L, bits, 2 << logn)
    p = hefx.hefx_params_create(ctx, logn, primes)
    try:
        data, other = (np.stack([inputs.residue_tensor(inputs.derive_seed(91, k, bits, b), 1, primes, n)[0]
                                 for b in range(batch)]) for k in (0, 1))
        data[..., :2] = (np.asarray(primes, dtype=np.uint32) - 1)[:, None]
        other[..., 0], data[..., 2] = (np.asarray(primes, dtype=np.uint32) - 1), 0
        x, y = to_dev(data), to_dev(other)
        got = forms(ctx, p, x, y, L, batch, n)
        hefx.hefx_params_set_cc_schedule(ctx, p, "cluster")
        for k, (a, b) in enumerate(zip(got, forms(ctx, p, x, y, L, batch, n))):
            assert torch.equal(a, b), f"form {k}"
        assert np.array_equal(to_host(got[0]).reshape(data.shape), oracle.ntt_batch(data, primes))
        assert np.array_equal(to_host(got[1]).reshape(data.shape), oracle.ntt_batch(data, primes, inverse=True))
        prod = data.astype(np.uint64) * other % np.asarray(primes, dtype=np.uint64)[:, None]
        assert np.array_equal(to_host(got[2]).reshape(data.shape),
                              oracle.ntt_batch(prod.astype(np.uint32), primes, inverse=True))
        hefx.hefx_stream_check(ctx, p)
    finally:
        hefx.hefx_params_destroy(p)


@pytest.mark.parametrize("logn,L,batch", [(14, 9, 20), (15, 1, 89), (16, 1, 44), (16, 3, 15), (16, 2, 72), (16, 1, 145),
                                          (15, 2, 257), (14, 2, 641), (16, 1, 257), (17, 1, 23), (17, 3, 50)])
def test_both_sides_of_the_lines(ctx, logn, L, batch):
    """Rows around 44, 144, 256 and 320 rows of 2^16 elements (each rounded to whole rows)."""
    n = 1 << logn
    primes = inputs.ntt_primes(L, 28, 2 << logn)
    p = hefx.hefx_params_create(ctx, logn, primes)
    try:
        g = torch.Generator(device="cuda").manual_seed(logn * 1000 + L)
        q = torch.tensor(primes, device="cuda").view(1, L, 1)
        x, y = ((torch.randint(0, 1 << 28, (batch, L, n), generator=g, device="cuda") % q).int() for _ in range(2))
        got = forms(ctx, p, x, y, L, batch, n)
        hefx.hefx_params_set_cc_schedule(ctx, p, "cluster")
        for k, (a, b) in enumerate(zip(got, forms(ctx, p, x, y, L, batch, n))):
            assert torch.equal(a, b), f"form {k}"
        hefx.hefx_stream_check(ctx, p)
    finally:
        hefx.hefx_params_destroy(p)
