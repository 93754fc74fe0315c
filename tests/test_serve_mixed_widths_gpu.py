"""A group of serving requests whose ciphertext primes are of different widths (28 bits, 30 bits, and a
set of both) equals each request on its own, in every order: what a row's arithmetic may assume
follows from the largest prime of the whole group, not from the first request's."""
import itertools

import pytest
import torch

from paper_2501_07047_gb300 import hefx, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("logn", [10, 12, 13, 14, 15, 16])
def test_group_of_mixed_widths(logn):
    n, K = 1 << logn, 3
    wide = inputs.special_primes(K + 5)
    ps, sets = wide[:K], [inputs.source_primes(4), wide[K:], inputs.source_primes(2) + wide[-2:]]
    ctx = hefx.hefx_create(0)
    pp = hefx.hefx_params_create(ctx, logn, ps)
    slots = hefx.hefx_mult_batch_create(ctx, 4, 8)
    gen = torch.Generator(device="cuda").manual_seed(logn)

    def residues(primes):
        q = torch.tensor(primes, device="cuda")[:, None]
        x = (torch.randint(0, 1 << 62, (len(primes), n), generator=gen, device="cuda") % q).int()
        x[:, :4] = (q - 1).int()
        return x

    made, keep = [], []
    try:
        for qs in sets:
            L = len(qs)
            pq, bc = hefx.hefx_params_create(ctx, logn, qs), hefx.hefx_bconv_plan_create(ctx, logn, qs, ps)
            keys = [residues(p) for p in (qs, qs, ps, ps)]
            made.append((hefx.hefx_mult_plan_create(ctx, pq, pp, bc, *keys), pq, bc))
            ct = torch.cat([residues(qs) for _ in range(4)])
            out, work = (torch.zeros((r, n), dtype=torch.int32, device="cuda") for r in (4 * L + 2 * K, 2 * L + K))
            hefx.hefx_mult_front(ctx, made[-1][0], ct, out, work)
            keep.append((L, ct, out, keys))
        torch.cuda.synchronize()
        for order in itertools.permutations(range(len(sets))):
            outs = [torch.full_like(keep[k][2], -1) for k in order]
            works = [torch.zeros((2 * keep[k][0] + K, n), dtype=torch.int32, device="cuda") for k in order]
            operands = [[keep[k][1][i * keep[k][0]:(i + 1) * keep[k][0]] for k in order] for i in range(4)]
            hefx.hefx_mult_front_batch(ctx, slots, [made[k][0] for k in order], *operands, outs, works)
            torch.cuda.synchronize()
            for k, got in zip(order, outs):
                assert torch.equal(got, keep[k][2]), (order, k)
    finally:
        for plan, pq, bc in made:
            hefx.hefx_mult_plan_destroy(plan)
            hefx.hefx_bconv_plan_destroy(bc)
            hefx.hefx_params_destroy(pq)
        hefx.hefx_mult_batch_destroy(slots)
        hefx.hefx_params_destroy(pp)
        hefx.hefx_destroy(ctx)
