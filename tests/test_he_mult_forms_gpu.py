"""Every composed form of HE-Mult against the oracle: without the Rescale, followed by rescale(), with it; on
the CUDA-core and the tensor-core transforms; the stages of the forms that compute them directly; and
rescale=False captured as a graph.  The shapes are small ones and the ones that the benchmark times."""
import numpy as np
import pytest
import torch

import oracle
from oracle import keyswitch as oks
from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult

from hefx_testutil import to_dev as dev, to_host as host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


def residues(seed, rows, primes, n):
    a = inputs.residue_tensor(inputs.derive_seed(*seed), rows, primes, n)
    a[..., 0] = np.asarray(primes, dtype=np.uint32) - 1
    return a


@pytest.mark.parametrize("logn,L,K,alpha,ntt,bconv", [
    (6, 2, 1, 1, "cudacore", "auto"), (8, 5, 2, 2, "cudacore", "tensor"), (10, 6, 3, 3, "cudacore", "cudacore"),
    (12, 7, 4, 4, "tensor", "auto"), (15, 9, 4, 4, "tensor", "tensor"), (14, 9, 4, 4, "cudacore", "auto"),
    (14, 6, 3, 3, "tensor", "cudacore"), (16, 24, 8, 8, "cudacore", "auto"), (16, 24, 8, 8, "tensor", "auto"),
    (16, 48, 16, 16, "cudacore", "auto")])
def test_forms(ctx, logn, L, K, alpha, ntt, bconv):
    n, qs, ps = 1 << logn, inputs.source_primes(L), inputs.special_primes(K)
    qp = list(qs) + list(ps)
    hm = HeMult(ctx, logn, qs, ps, alpha, ntt_path=ntt, bconv_path=bconv)
    try:
        ins = [residues((87, logn, c), 1, qs, n)[0] for c in range(4)]
        evk = np.stack([residues((88, logn, j), 2, qp, n) for j in range(hm.dnum)])
        want = oks.he_mult(*ins, evk, qs, ps, alpha)
        dins, devk = [dev(a) for a in ins], dev(evk)
        c, out, again = (dev(np.full((2, r, n), 0xFFFFFFFF, dtype=np.uint32)) for r in (L, L - 1, L - 1))

        hm.run(*dins, devk, c, rescale=False)
        got = host(c)
        assert np.array_equal(got[0], want["c0"]) and np.array_equal(got[1], want["c1"])
        st = {k: host(v) for k, v in hm.stages().items()}
        q = np.asarray(qs, dtype=np.uint64)[:, None]
        a0, a1, b0, b1 = (x.astype(np.uint64) for x in ins)
        assert np.array_equal(st["d0"], (a0 * b0 % q).astype(np.uint32))
        assert np.array_equal(st["d1"], ((a0 * b1 % q + a1 * b0 % q) % q).astype(np.uint32))
        assert np.array_equal(st["d2_coeff"], oracle.ntt_batch(want["d2"][None], qs, inverse=True)[0])
        assert np.array_equal(st["modup_eval"], oracle.ntt_batch(want["modup"], qp))
        assert np.array_equal(st["acc_coeff"], oracle.ntt_batch(want["acc"], qp, inverse=True))
        assert np.array_equal(st["ks_eval"], oracle.ntt_batch(want["ks"], qs))

        cw = c.clone()
        hm.rescale(cw, out)
        got = host(out)
        assert np.array_equal(got[0], want["c0r"]) and np.array_equal(got[1], want["c1r"])
        hm.run(*dins, devk, again)
        assert torch.equal(again, out)
        assert np.array_equal(host(hm.stages()["c_coeff"]),
                              oracle.ntt_batch(np.stack([want["c0"], want["c1"]]), qs, inverse=True))

        g = hm.capture(*dins, devk, cw, rescale=False)
        cw.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(cw, c)
        del g
        hm.check()
    finally:
        hm.close()
