"""Tickets after a wait that ran out in some of the CTAs: they are zero again, so the calls that follow on the stream, whose tickets
are the same words, add up all parts, whether the status is cleared or not.
"""

import numpy as np
import pytest
import torch

import paper_2510_19482_b200 as elutq
import workloads
from oracle import hlq
from workloads import synth

pytestmark = pytest.mark.gpu

from gpu_util import gemm_f32, pack_layer, x_dev  # noqa: E402

HALF = 0x80000000          # every other CTA gives up


# the fragment kernel with output tiles in clusters, which take no tickets, and with several chunks per CTA; the tensor-memory kernel with tiles of two parts
# (and with more output tiles than clusters take, with one and with several batch blocks)
@pytest.mark.parametrize("q,G,N,K,M", [(3, 64, 1000, 1984, 20), (2, 64, 9000, 2240, 9), (4, 128, 20480, 2048, 16), (3, 64, 20000, 2688, 9), (2, 64, 10000, 2240, 20)])
def test_tickets_are_zero_after_some_ctas_gave_up(q, G, N, K, M):
    layer = workloads.hlq_layer(64, f"tickets/{q}/{G}/{N}/{K}", q, G, N, K)
    X = synth.activations(64, f"tickets/x/{M}/{K}", M, K)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    elutq.elutq_release_scratch()
    Y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    for limit in (300, 20000):
        elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, HALF | limit)
        assert elutq.elutq_device_status() == 0x7C05
        for m in (1, M):                                 # the decode kernel and the same kernel again
            y = gemm_f32(X[:m], packed, N, K)
            assert hlq.rel_fro_error(y, ref[:m]) <= 1e-3
    elutq.elutq_release_scratch()
    assert np.array_equal(gemm_f32(X, packed, N, K), y)
    assert elutq.elutq_device_status() == 0


def test_tickets_of_one_chunk_per_cta():
    # (more chunks than a cluster has CTAs, so their parts meet in the workspace)
    from test_frag_gpu import parts_meet_in_the_workspace
    q, G, N, K, M = 3, 64, 1500, 4672, 9
    X = synth.activations(64, f"tickets/x/{M}/{K}", M, K)
    assert parts_meet_in_the_workspace(X, pack_layer(workloads.hlq_layer(64, f"tickets/{q}/{G}/{N}/{K}", q, G, N, K)), N, K)
    test_tickets_are_zero_after_some_ctas_gave_up(q, G, N, K, M)
