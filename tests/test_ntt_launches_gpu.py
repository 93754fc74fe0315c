"""Launches of a transform: the library's count equals the kernel nodes of the same call captured into a
graph, and a lone forward call of few rows of 2^15 is one launch (equal to the captured form's two
and to the oracle)."""
import ctypes

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


def captured_nodes(call):
    """Nodes of the graph of call(stream) and the graph, already run once."""
    call(torch.cuda.current_stream())
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        call(torch.cuda.current_stream())
    count = ctypes.c_size_t(0)
    cudart = ctypes.CDLL("libcudart.so.13")
    assert cudart.cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None, ctypes.byref(count)) == 0
    return count.value


@pytest.mark.parametrize("logn,L,batch", [(5, 2, 3), (12, 3, 1), (13, 2, 70), (14, 2, 2), (14, 3, 43), (15, 4, 8), (15, 3, 11),
                                          (15, 2, 257), (16, 3, 1), (16, 3, 87), (17, 2, 1)])
def test_counts_equal_the_graph(ctx, logn, L, batch):
    n = 1 << logn
    p = hefx.hefx_params_create(ctx, logn, inputs.ntt_primes(L, 28, 2 << logn))
    x, y, z = (torch.zeros((batch, L, n), dtype=torch.int32, device="cuda") for _ in range(3))
    try:
        calls = {"fwd": lambda s: hefx.hefx_ntt_fwd(ctx, p, x, batch, stream=s),
                 "inv": lambda s: hefx.hefx_ntt_inv(ctx, p, x, batch, stream=s),
                 "inv_hadamard": lambda s: hefx.hefx_ntt_inv_hadamard(ctx, p, x, y, z, batch, stream=s),
                 "rescale_fwd": lambda s: hefx.hefx_rescale_ntt(ctx, p, x, z, batch, stream=s),
                 "poly_mul": lambda s: hefx.hefx_poly_mul(ctx, p, x, y, z, batch, stream=s)}
        for schedule in ("auto", "cluster"):
            hefx.hefx_params_set_cc_schedule(ctx, p, schedule)
            for form, call in calls.items():
                assert captured_nodes(call) == hefx.hefx_ntt_launches(p, form, batch, captured=True), (schedule, form)
    finally:
        hefx.hefx_params_destroy(p)


@pytest.mark.parametrize("bits", [28, 30])
@pytest.mark.parametrize("L,batch", [(1, 1), (5, 3), (16, 2), (11, 3)])
def test_lone_forward_of_few_rows(ctx, bits, L, batch):
    logn, n = 15, 1 << 15
    primes = inputs.ntt_primes(L, bits, 2 << logn)
    p = hefx.hefx_params_create(ctx, logn, primes)
    try:
        few = L * batch <= 32
        assert hefx.hefx_ntt_launches(p, "fwd", batch) == (1 if few else 2)
        assert hefx.hefx_ntt_launches(p, "fwd", batch, captured=True) == 2
        data = np.stack([inputs.residue_tensor(inputs.derive_seed(95, bits, b), 1, primes, n)[0] for b in range(batch)])
        data[..., 0] = np.asarray(primes, dtype=np.uint32) - 1
        want = oracle.ntt_batch(data, primes)
        lone, held = to_dev(data), empty_dev(data.shape)
        hefx.hefx_ntt_fwd(ctx, p, lone, batch)
        assert np.array_equal(to_host(lone).reshape(data.shape), want)
        src = to_dev(data)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            held.copy_(src)
            hefx.hefx_ntt_fwd(ctx, p, held, batch, stream=torch.cuda.current_stream())
        g.replay()
        assert np.array_equal(to_host(held).reshape(data.shape), want)
        hefx.hefx_stream_check(ctx, p)
    finally:
        hefx.hefx_params_destroy(p)
