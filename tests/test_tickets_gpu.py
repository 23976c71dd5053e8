"""Tickets that an expired wait left half counted: whoever they name as the last CTA (or warp) of a shared tile writes nothing, and a
workspace that is initialised again is as good as new.  The control area is prepared by hand: word 0 the status, tickets from word
64 on, each counted once already.
"""

import numpy as np
import pytest
import torch

import paper_2510_19482_b200 as elutq
import workloads
from oracle import hlq
from workloads import synth

pytestmark = pytest.mark.gpu

from gpu_util import pack_layer, x_dev  # noqa: E402

# (q, G, N, K, M, tickets): the decode kernel, the fragment kernel, the tensor-memory kernel with tiles of two or three parts
CASES = [(2, 128, 4096, 4096, 1, 256), (3, 64, 1000, 1024, 1, 256), (2, 128, 1000, 1024, 4, 8), (3, 64, 1000, 1984, 20, 8),
         (4, 128, 20480, 2048, 16, 4096)]
SENTINEL = -77.0


@pytest.mark.parametrize("q,G,N,K,M,tickets", CASES)
def test_half_counted_tickets_name_nobody(q, G, N, K, M, tickets):
    layer = workloads.hlq_layer(64, f"tickets/{q}/{G}/{N}/{K}", q, G, N, K)
    X = synth.activations(64, f"tickets/x/{M}/{K}", M, K)
    packed, x = pack_layer(layer), x_dev(X)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    ws = torch.empty(elutq.elutq_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    words = ws.view(torch.int32)
    elutq.elutq_workspace_init(ws)
    words[0] = 0x7C05
    words[64:64 + tickets] = 1
    Y = torch.full((M, N), SENTINEL, dtype=torch.float32, device="cuda")
    for _ in range(2):
        elutq.elutq_lut_gemm_ws(x, packed, Y, M, N, K, elutq.FLAG_OUT_F32, ws)
    y = Y.cpu().numpy()
    left = y == SENTINEL
    tol = 2e-2 * np.sqrt(np.mean(ref ** 2))              # far below a missing part, far above any rounding
    assert np.all(left | (np.abs(y - ref) <= tol))       # a tile that one CTA has to itself needs no ticket
    assert left.mean() > 0.5
    elutq.elutq_workspace_init(ws)
    elutq.elutq_lut_gemm_ws(x, packed, Y, M, N, K, elutq.FLAG_OUT_F32, ws)
    assert np.all(np.abs(Y.cpu().numpy() - ref) <= tol)
    assert int(words[0]) == 0
