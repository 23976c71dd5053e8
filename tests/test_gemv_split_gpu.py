"""The two reductions of the decode kernel's K split: the last CTA of a row range (elutq_lut_gemm), the finalize kernel
(elutq_lut_gemm_static, and elutq_lut_gemm for long ranges).  Both add the chunks in the same order, so their bits are equal.

Tolerance against the oracle: K fp32 sums, each rounded by at most 2^-24 of the magnitudes added: K * 2^-24 * A per element.
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

# (q, G, N, K): 1, 2, 8, 9, 32 and 33 chunks of 512 columns; at 8 and 9 chunks the longest ranges of 1024 rows and the next
CASES = [(2, 128, 100, 512), (3, 64, 17, 544 + 32), (2, 128, 16384, 4096), (2, 128, 16400, 4096), (1, 128, 14336, 4224), (1, 128, 14352, 4224),
         (4, 32, 1000, 16384), (2, 128, 333, 16512), (2, 128, 1, 1024)]


@pytest.mark.parametrize("q,G,N,K", CASES)
def test_both_reductions_agree(q, G, N, K):
    layer = workloads.hlq_layer(62, f"split/{q}/{G}/{N}/{K}", q, G, N, K)
    X = synth.activations(62, f"split/x/{K}", 1, K, outliers=True)
    packed, x = pack_layer(layer), x_dev(X)
    ys = [torch.empty((1, N), dtype=torch.float16, device="cuda") for _ in range(4)]
    for y in ys[:3]:                                     # the tickets are zero again after every call
        elutq.elutq_lut_gemm(x, packed, y, 1, N, K)
    elutq.elutq_lut_gemm_static(x, packed, ys[3], 1, N, K)
    assert elutq.elutq_device_status() == 0
    bits = [y.cpu().numpy().view(np.uint16) for y in ys]
    assert all(np.array_equal(bits[0], b) for b in bits[1:])
    y = gemm_f32(X, packed, N, K)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    assert np.all(np.abs(y - ref) <= K * 2.0 ** -24 * hlq.magnitude_bound(X, layer.scales, layer.offsets, G))


@pytest.mark.parametrize("q,G,N,K", [(2, 128, 2048, 2048), (1, 128, 1000, 8192), (3, 64, 14336, 4096), (2, 128, 4096, 4096)])
def test_calls_in_a_graph_give_the_same_bits(q, G, N, K):
    layer = workloads.hlq_layer(63, f"split/graph/{q}/{G}/{N}/{K}", q, G, N, K)
    X = synth.activations(63, f"split/graph/x/{K}", 1, K)
    packed, x = pack_layer(layer), x_dev(X)
    plain, replayed = (torch.empty((1, N), dtype=torch.float16, device="cuda") for _ in range(2))
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        elutq.elutq_lut_gemm(x, packed, plain, 1, N, K)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            for _ in range(3):
                elutq.elutq_lut_gemm(x, packed, replayed, 1, N, K)
        for _ in range(2):
            graph.replay()
        elutq.elutq_lut_gemm(x, packed, plain, 1, N, K)
        stream.synchronize()
    assert torch.equal(plain.view(torch.int16), replayed.view(torch.int16))
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    assert hlq.rel_fro_error(plain.cpu().numpy(), ref) <= 1e-3
