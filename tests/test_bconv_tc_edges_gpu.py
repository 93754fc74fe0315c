"""The tensor-core conversion at the edges of its tiles, bit for bit against the oracle: source
counts around the 16-source chunks of its A operand and the places of its constant columns, target
counts around its groups of eight and its accumulator widths, one tile and odd numbers of tiles,
28- and 30-bit sources, targets below 2^18 (the 64-bit reduction), extreme residues; the plain
conversion, ModDown, ModUp with a ragged last digit, and the bounded-wait flags.  Outputs are
whole numbers: equal."""
import numpy as np
import pytest

import oracle
from oracle import keyswitch as oks
from paper_2501_07047_gb300 import hefx, inputs

from hefx_testutil import to_dev as dev, to_host as host

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = hefx.hefx_create(0)
    yield c
    hefx.hefx_destroy(c)


def residues(seed, batch, primes, n):
    a = inputs.residue_tensor(inputs.derive_seed(*seed), batch, primes, n)
    a[..., 0] = np.asarray(primes, dtype=np.uint32) - 1  # every digit at its largest
    a[..., 1] = 0
    return a


def converted(ctx, src, dst, a, path):
    batch, _, n = a.shape
    plan = hefx.hefx_bconv_plan_create(ctx, n.bit_length() - 1, src, dst)
    try:
        out = dev(np.full((batch, len(dst), n), 0xFFFFFFFF, dtype=np.uint32))
        hefx.hefx_basis_convert(ctx, plan, dev(a), out, batch, path)
        hefx.hefx_bconv_check(ctx, plan)
        return host(out)
    finally:
        hefx.hefx_bconv_plan_destroy(plan)


@pytest.mark.parametrize("L,Lp", [(1, 1), (2, 4), (3, 5), (4, 8), (12, 9), (13, 16), (15, 17), (16, 32), (16, 48),
                                  (17, 33), (28, 40), (31, 31), (32, 64), (33, 12), (44, 7), (48, 20)])
def test_tensor_source_and_target_counts(ctx, L, Lp):
    src, dst = inputs.source_primes(L), inputs.special_primes(Lp)
    a = residues((71, L, Lp), 3, src, 128)
    assert np.array_equal(converted(ctx, src, dst, a, "tensor"), oracle.bconv(a, src, dst))


@pytest.mark.parametrize("logn,batch", [(7, 1), (8, 5), (10, 33), (13, 7)])
def test_tensor_tile_counts(ctx, logn, batch):
    """From one tile to several rounds of every ring of buffers, some CTAs one tile short."""
    src, dst = inputs.source_primes(20), inputs.special_primes(12)
    a = residues((72, logn), batch, src, 1 << logn)
    assert np.array_equal(converted(ctx, src, dst, a, "tensor"), oracle.bconv(a, src, dst))


@pytest.mark.parametrize("dst", [[3], [65537, 3, 262139, 262147, 1073479681], [257, 786433]])
def test_tensor_small_targets(ctx, dst):
    src = inputs.source_primes(9)
    a = residues((73, len(dst)), 2, src, 256)
    assert np.array_equal(converted(ctx, src, dst, a, "tensor"), oracle.bconv(a, src, dst))


@pytest.mark.parametrize("L,Lp", [(4, 9), (16, 48), (24, 11), (15, 40)])
def test_auto_with_30_bit_sources(ctx, L, Lp):
    """30-bit sources (AUTO only: HEFX_PATH_TENSOR stays refused for them), mixed with 28-bit ones."""
    src = list(inputs.special_primes(L - 1)) + list(inputs.source_primes(Lp + 1)[Lp:])
    dst = inputs.source_primes(Lp)
    a = residues((74, L, Lp), 3, src, 512)
    assert np.array_equal(converted(ctx, src, dst, a, "auto"), oracle.bconv(a, src, dst))
    with pytest.raises(hefx.HefxError) as e:
        converted(ctx, src, dst, a, "tensor")
    assert e.value.status == hefx.HEFX_EUNSUPPORTED


@pytest.mark.parametrize("logn,L,K,alpha,batch", [(7, 9, 4, 4, 3), (9, 23, 12, 8, 2), (8, 33, 17, 17, 1),
                                                  (7, 48, 16, 16, 1)])
def test_mod_up_and_down_tiles(ctx, logn, L, K, alpha, batch):
    n = 1 << logn
    qs, ps = inputs.source_primes(L), inputs.special_primes(K)
    c = residues((75, logn, L), batch, qs, n)
    plan = hefx.hefx_modup_plan_create(ctx, logn, qs, ps, alpha)
    dnum = hefx.hefx_modup_plan_dnum(plan)
    dU = dev(np.full((batch, dnum, L + K, n), 0xFFFFFFFF, dtype=np.uint32))
    hefx.hefx_mod_up(ctx, plan, dev(c), dU, batch)
    hefx.hefx_modup_check(ctx, plan)
    got = host(dU)
    for b in range(batch):
        assert np.array_equal(got[b], oks.modup(c[b], qs, ps, alpha))
    hefx.hefx_modup_plan_destroy(plan)
    x = residues((76, logn, L), batch, list(qs) + list(ps), n)
    plan = hefx.hefx_bconv_plan_create(ctx, logn, ps, qs)
    out = dev(np.full((batch, L, n), 0xFFFFFFFF, dtype=np.uint32))
    hefx.hefx_mod_down(ctx, plan, dev(x), out, batch)
    hefx.hefx_bconv_check(ctx, plan)
    assert np.array_equal(host(out), oracle.moddown(x, qs, ps))
    hefx.hefx_bconv_plan_destroy(plan)
