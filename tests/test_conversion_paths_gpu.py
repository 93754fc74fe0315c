"""ModUp, ModDown and the ModDown of scaled limbs on the CUDA cores, asked for and where the
tensor-core kernel does not apply (fewer than 4 sources, N < 2^7), with many targets and several full groups
of sources: equal to the oracle on sampled coefficients, and run by the kernel that was asked for (256
threads a block; the tensor-core kernel has 704)."""
import numpy as np
import pytest
import torch

import oracle
from oracle import keyswitch as oks
from paper_2501_07047_gb300 import hefx, inputs
from paper_2501_07047_gb300.hemult import HeMult

from graph_util import kernel_blocks
from hefx_testutil import to_dev as dev, to_host as host

pytestmark = pytest.mark.gpu
TENSOR, CUDACORE = 704, 256


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


def residues(seed, batch, primes, n):
    a = inputs.residue_tensor(inputs.derive_seed(*seed), batch, primes, n)
    a[..., 0] = np.asarray(primes, dtype=np.uint32) - 1
    a[..., 1] = 0
    return a


SHAPES = [(16, 48, 16, 16, 1, "cudacore"), (13, 33, 17, 17, 2, "cudacore"), (7, 30, 9, 4, 3, "cudacore"),
          (9, 30, 3, 2, 2, "auto"), (12, 12, 1, 1, 1, "auto"), (10, 23, 3, 3, 1, "auto"), (6, 20, 12, 8, 2, "auto")]


@pytest.mark.parametrize("logn,L,K,alpha,batch,path", SHAPES)
def test_cuda_core_forms(ctx, logn, L, K, alpha, batch, path):
    n, qs, ps = 1 << logn, inputs.source_primes(L), inputs.special_primes(K)
    qp = list(qs) + list(ps)
    cols = np.arange(n) if n <= 4096 else np.r_[0, 1, np.sort(np.random.default_rng(3).choice(n, 510, replace=False))]
    up, pq = hefx.hefx_modup_plan_create(ctx, logn, qs, ps, alpha), hefx.hefx_bconv_plan_create(ctx, logn, ps, qs)
    try:
        hefx.hefx_modup_plan_set_path(ctx, up, path)
        hefx.hefx_bconv_plan_set_mod_down_path(ctx, pq, path)
        dnum = hefx.hefx_modup_plan_dnum(up)
        c, x = residues((83, logn, L), batch, qs, n), residues((84, logn, L), batch, qp, n)
        dc, dx = dev(c), dev(x)
        dU = dev(np.full((batch, dnum, L + K, n), 0xFFFFFFFF, dtype=np.uint32))
        down, scaled = (dev(np.full((batch, L, n), 0xFFFFFFFF, dtype=np.uint32)) for _ in range(2))
        assert kernel_blocks(lambda s: hefx.hefx_mod_up(ctx, up, dc, dU, batch, s)) == [CUDACORE]
        assert kernel_blocks(lambda s: hefx.hefx_mod_down(ctx, pq, dx, down, batch, s)) == [CUDACORE]
        assert kernel_blocks(lambda s: hefx.hefx_mod_down_scaled(ctx, pq, dx, scaled, batch, s)) == [CUDACORE]
        got = host(dU)
        for b in range(batch):
            assert np.array_equal(got[b][..., cols], oks.modup(c[b][:, cols], qs, ps, alpha))
        xc = np.ascontiguousarray(x[..., cols])
        assert np.array_equal(host(down)[..., cols], oracle.moddown(xc, qs, ps))
        zero = xc.copy()
        zero[:, :L] = 0  # -BConv P^-1
        q = np.asarray(qs, dtype=np.uint64)[None, :, None]
        want = (xc[:, :L].astype(np.uint64) + oracle.moddown(zero, qs, ps)) % q
        assert np.array_equal(host(scaled)[..., cols], want.astype(np.uint32))
    finally:
        hefx.hefx_modup_plan_destroy(up)
        hefx.hefx_bconv_plan_destroy(pq)


def test_paths_of_the_plans(ctx):
    """AUTO undoes the request; a path that the fused forms do not offer is refused and changes nothing."""
    logn, L, K = 8, 12, 6
    n, qs, ps = 1 << logn, inputs.source_primes(L), inputs.special_primes(K)
    up, pq = hefx.hefx_modup_plan_create(ctx, logn, qs, ps, 6), hefx.hefx_bconv_plan_create(ctx, logn, ps, qs)
    c, x = (torch.zeros((r, n), dtype=torch.int32, device="cuda") for r in (L, L + K))
    U, out = (torch.zeros((r, n), dtype=torch.int32, device="cuda") for r in (2 * (L + K), L))
    try:
        def blocks():
            return (kernel_blocks(lambda s: hefx.hefx_mod_up(ctx, up, c, U, 1, s)) +
                    kernel_blocks(lambda s: hefx.hefx_mod_down(ctx, pq, x, out, 1, s)))

        assert blocks() == [TENSOR, TENSOR]
        for path, want in (("cudacore", CUDACORE), ("auto", TENSOR)):
            hefx.hefx_modup_plan_set_path(ctx, up, path)
            hefx.hefx_bconv_plan_set_mod_down_path(ctx, pq, path)
            for call, plan in ((hefx.hefx_modup_plan_set_path, up), (hefx.hefx_bconv_plan_set_mod_down_path, pq)):
                with pytest.raises(hefx.HefxError) as e:
                    call(ctx, plan, "tensor")
                assert e.value.status == hefx.HEFX_EINVAL
            assert blocks() == [want, want]
        assert hefx.raw_status("hefx_modup_plan_set_path", 0, 0) == hefx.HEFX_EINVAL
        assert hefx.raw_status("hefx_bconv_plan_set_mod_down_path", 0, 0) == hefx.HEFX_EINVAL
    finally:
        hefx.hefx_modup_plan_destroy(up)
        hefx.hefx_bconv_plan_destroy(pq)


@pytest.mark.parametrize("path", ["cudacore", "auto"])
def test_he_mult_keeps_the_path(ctx, path):
    logn, L, K, alpha = 10, 9, 4, 4
    n, qs, ps = 1 << logn, inputs.source_primes(L), inputs.special_primes(K)
    qp = list(qs) + list(ps)
    hm = HeMult(ctx, logn, qs, ps, alpha, bconv_path=path)
    try:
        ins = [residues((85, c), 1, qs, n)[0] for c in range(4)]
        evk = np.stack([residues((86, j), 2, qp, n) for j in range(hm.dnum)])
        dins, devk, out = [dev(a) for a in ins], dev(evk), dev(np.zeros((2, L - 1, n), dtype=np.uint32))
        blocks = kernel_blocks(lambda s: hm.run(*dins, devk, out, s))
        assert blocks.count(TENSOR) == (0 if path == "cudacore" else 2)
        want = oks.he_mult(*ins, evk, qs, ps, alpha)
        got = host(out)
        assert np.array_equal(got[0], want["c0r"]) and np.array_equal(got[1], want["c1r"])
    finally:
        hm.close()
