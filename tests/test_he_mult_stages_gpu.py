"""HeMult.stages after a replayed graph whose form is not the last eager run's: told the form, it returns
that form's stages."""
import numpy as np
import pytest
import torch

import oracle
from oracle import keyswitch as oks
from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult

from hefx_testutil import to_dev as dev, to_host as host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ntt", ["cudacore", "tensor"])
@pytest.mark.parametrize("replayed", [True, False])
def test_stages_of_a_replay(ntt, replayed):
    ctx = hefx.hefx_create(0)
    logn, L, K, alpha = 12, 6, 3, 3
    n, qs, ps = 1 << logn, inputs.source_primes(L), inputs.special_primes(K)
    qp = list(qs) + list(ps)
    hm = HeMult(ctx, logn, qs, ps, alpha, ntt_path=ntt)
    try:
        ins = [inputs.residue_tensor(inputs.derive_seed(89, c), 1, qs, n)[0] for c in range(4)]
        evk = np.stack([inputs.residue_tensor(inputs.derive_seed(90, j), 2, qp, n) for j in range(hm.dnum)])
        want = oks.he_mult(*ins, evk, qs, ps, alpha)
        dins, devk = [dev(a) for a in ins], dev(evk)
        out = {r: dev(np.zeros((2, L - r, n), dtype=np.uint32)) for r in (True, False)}
        g = hm.capture(*dins, devk, out[replayed], rescale=replayed)
        hm.run(*dins, devk, out[not replayed], rescale=not replayed)
        g.replay()
        torch.cuda.synchronize()
        st = {k: host(v) for k, v in hm.stages(rescale=replayed).items()}
        assert np.array_equal(st["acc_coeff"], oracle.ntt_batch(want["acc"], qp, inverse=True))
        assert np.array_equal(st["ks_eval"], oracle.ntt_batch(want["ks"], qs))
        del g
    finally:
        hm.close()
        hefx.hefx_destroy(ctx)
