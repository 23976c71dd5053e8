"""GPU parity of the kernel that rebuilds weights in tensor memory (batches of more than 8 rows at G = 128 with enough weight rows).

Tolerance: W_hat = z + sum_j b_j s_j is formed with one fp16 fma per plane (exact products, each sum rounded at 2^-11 relative; above 32
rows weight 7 of a byte starts from z^ = z + (1/2) sum_j s_j, rounded once, and adds +-s_j / 2), products are exact and the sums fp32.  The
weights' rounding errors are independent across k: a relative error of about 2^-12 .. 2^-11 in norm, bar 1e-3; per element
the worst-case bound of gpu_util.assert_elementwise.
"""

import numpy as np
import pytest
import torch

import paper_2510_19482_b200 as elutq
import workloads
from oracle import hlq
from workloads import synth

pytestmark = pytest.mark.gpu

from gpu_util import assert_elementwise, gemm_f32, pack_layer, x_dev  # noqa: E402

G, TOL = 128, 1e-3

# (q, N, K, M): one step of K, a K that ends inside a 512-k chunk, ragged rows and tokens, one and several token tiles (9 -> 16 tokens,
# 200 -> 2 x 112); whole tiles per CTA, shared tiles of two or three parts, of many parts, clusters of two CTAs and more (with K steps and
# tokens that they do not divide evenly, and N no multiple of the stores' four), whole rounds with the rest by clusters
CASES = [(2, 4621, 128, 9), (1, 4480, 1152, 128), (3, 4600, 640, 200), (4, 5000, 2944, 100), (4, 12800, 2048, 384), (2, 38000, 256, 33),
         (3, 10240, 1024, 130), (2, 11776, 7680, 16), (2, 16000, 1024, 100), (2, 3001, 4096, 20), (3, 1100, 1152, 90), (1, 300, 256, 33), (2, 13000, 2560, 384),
         # few tokens, whose activations the kernel puts in another order: the last sizes on that path and the first beyond it, loaders of one, two and
         # three steps, clusters, shared tiles, whole rounds with a rest
         (1, 4480, 128, 12), (2, 4621, 256, 10), (4, 1100, 384, 15), (3, 4600, 1152, 17), (3, 12800, 640, 32), (4, 38000, 512, 25), (4, 3001, 4096, 33),
         (2, 16000, 1024, 17), (4, 10240, 1024, 32), (3, 38000, 256, 16),
         # few tokens in equal shares instead of whole tiles: in one round, in two
         (4, 21500, 2048, 9), (4, 43001, 1024, 16)]


@pytest.mark.parametrize("q,N,K,M", CASES)
def test_tensor_memory_kernel_matches_oracle(q, N, K, M):
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    layer = workloads.hlq_layer(70, f"tmem/{q}/{N}/{K}", q, G, N, K, signed_scales=(q == 3))
    X = synth.activations(70, f"tmem/x/{M}/{K}", M, K, outliers=True)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert max(hlq.rel_fro_error(y[m], ref[m]) for m in range(M)) <= TOL
    assert_elementwise(y, ref, hlq.magnitude_bound(X, layer.scales, layer.offsets, G), q, K, True, False, "fp32 out")
    assert np.array_equal(y.view(np.uint32), gemm_f32(X, packed, N, K).view(np.uint32))       # and the tickets are zero again
    ys = gemm_f32(X, packed, N, K, elutq.FLAG_SKIP_OFFSET)
    yb = gemm_f32(X, packed, N, K, elutq.FLAG_OFFSET_ONLY)
    assert hlq.rel_fro_error(ys, hlq.scale_term(X, layer.planes, layer.scales, G)) <= TOL
    assert hlq.rel_fro_error(yb, hlq.offset_term(X, layer.offsets, G)) <= TOL
    Y = torch.full((M, N), 1.5, dtype=torch.float32, device="cuda")
    elutq.elutq_lut_gemm_f32(x_dev(X), packed, Y, M, N, K, elutq.FLAG_ACCUMULATE)
    np.testing.assert_allclose(Y.cpu().numpy(), y + 1.5, rtol=0, atol=1e-5 * np.abs(y).max())


# Two rounds of tiles less a part: the equal shares' own cost is below that of whole rounds and the rest by clusters, which are two launches
@pytest.mark.parametrize("q,N,K,M", [(4, 42703, 1280, 24), (4, 43008, 2048, 16)])
def test_equal_shares_of_few_tokens_are_one_launch(q, N, K, M):
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    gen = torch.Generator(device="cuda").manual_seed(74)
    planes = torch.randint(0, 2, (q, N, K), generator=gen, device="cuda", dtype=torch.uint8)
    scales = (torch.randn((N, K // G, q), generator=gen, device="cuda") * 0.02).abs().half()
    offsets = (torch.randn((N, K // G), generator=gen, device="cuda") * 0.01).half()
    packed = elutq.elutq_pack(planes, scales, offsets, q, G, N, K)
    X = synth.activations(74, f"tmem/shares/{M}/{K}", M, K)
    gemm_f32(X, packed, N, K)
    before = elutq.elutq_launch_count()
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_launch_count() == before + 1
    assert hlq.rel_fro_error(y, gemm_f32(X, packed, N, K, elutq.FLAG_LUT_ONLY)) <= TOL


# 17 to 32 tokens, half of them each loader's, with two steps on their way: one step, two, three, tokens that end in either half, a run that begins inside
# a tile, more steps than places in the ring
@pytest.mark.parametrize("q,N,K,M", [(1, 4480, 128, 17), (2, 4621, 256, 24), (3, 5000, 384, 25), (4, 3001, 1152, 31), (1, 21500, 2048, 32), (4, 300, 4096, 18), (2, 38000, 640, 23)])
def test_few_tokens_in_two_halves(q, N, K, M):
    test_tensor_memory_kernel_matches_oracle(q, N, K, M)


@pytest.mark.parametrize("q", [1, 2, 4])
def test_scales_of_one_and_more(q, M=40):
    N, K = 4700, 256
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    layer = workloads.hlq_layer(71, f"tmem/scales/{q}", q, G, N, K)
    s = layer.scales.astype(np.float32)
    s[1::4] *= 64.0                                      # around 1: only some groups of a row
    s[2::4] *= 8192.0
    s[3::4, :, 0] = 30000.0 + 2000.0 * np.arange(s[3::4].shape[0])[:, None] % 10000.0         # the largest exponent
    layer.scales[...] = s.astype(np.float16)
    X = synth.activations(71, "tmem/scales/x", M, K)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    for first in range(4):
        assert hlq.rel_fro_error(y[:, first::4], ref[:, first::4]) <= TOL


@pytest.mark.parametrize("q,M", [(1, 12), (2, 16), (3, 9), (4, 17)])
def test_scales_of_one_and_more_with_few_tokens(q, M):
    test_scales_of_one_and_more(q, M)


def test_a_wait_that_runs_out_is_reported():
    q, N, K, M = 2, 8192, 2048, 64
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    layer = workloads.hlq_layer(72, "tmem/expiry", q, G, N, K)
    X = synth.activations(72, "tmem/expiry/x", M, K)
    packed = pack_layer(layer)
    elutq.elutq_release_scratch()
    Y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, 4096)
    assert elutq.elutq_device_status() == 0x7C05
    elutq.elutq_release_scratch()
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert hlq.rel_fro_error(y, hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)) <= TOL


@pytest.mark.parametrize("q,N,K,M", [(2, 512, 2048, 64), (1, 4096, 512, 9), (4, 40000, 384, 128)])
def test_waits_that_run_out_behind_loaders_that_are_done(q, N, K, M):
    # Clusters and whole tiles with so few steps of K that the loaders have requested everything when the other warps give up: they
    # still wait for their copies.  The calls that follow at once get the shared memory.
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    layer = workloads.hlq_layer(73, f"tmem/drain/{N}", q, G, N, K)
    X = synth.activations(73, f"tmem/drain/x/{M}/{K}", M, K)
    packed = pack_layer(layer)
    Y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    ws = torch.empty(elutq.elutq_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    elutq.elutq_workspace_init(ws)
    y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    x = x_dev(X)
    elutq.elutq_release_scratch()
    elutq.elutq_test_wait_expiry(x, packed, Y, M, N, K, 64)
    elutq.elutq_lut_gemm_ws(x, packed, y, M, N, K, elutq.FLAG_OUT_F32, ws)
    assert elutq.elutq_device_status() == 0x7C05
    assert int(ws.view(torch.int32)[0]) == 0
    assert hlq.rel_fro_error(y.cpu().numpy(), ref) <= TOL
    elutq.elutq_release_scratch()


# few tokens, whose activations two warps bring in another order: clusters, whole tiles, equal shares, and (1000 rows) the order of more tokens
@pytest.mark.parametrize("q,N,K,M", [(2, 4096, 4096, 16), (3, 28672, 2048, 9), (4, 21500, 2048, 27), (1, 4500, 1152, 32), (2, 1000, 1024, 17)])
def test_activations_that_are_not_finite(q, N, K, M):
    """An infinity makes its row's results infinite by the signs of its weights, a NaN or opposite infinities NaN; the other rows keep their bits."""
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_TENSOR_MEMORY
    layer = workloads.hlq_layer(77, f"tmem/inf/{q}/{N}/{K}", q, G, N, K, signed_scales=True)
    X = synth.activations(77, f"tmem/inf/x/{M}/{K}", M, K)
    packed = pack_layer(layer)
    y = gemm_f32(X, packed, N, K)
    X[0, 3] = np.inf
    X[2, K - 1] = -np.inf
    X[M - 2, K // 2 + 17] = np.nan
    X[M - 1, 40], X[M - 1, K - 30] = np.inf, np.inf
    z = gemm_f32(X, packed, N, K)
    keep = np.ones(M, dtype=bool)
    keep[[0, 2, M - 2, M - 1]] = False
    assert np.array_equal(z[keep], y[keep])
    assert np.isnan(z[M - 2]).all()

    def column(k):                                           # W_hat[:, k], and how far the rebuilt one may be from it
        w = hlq.reconstruct(layer.planes[:, :, k // G * G: (k // G + 1) * G], layer.scales[:, k // G: k // G + 1], layer.offsets[:, k // G: k // G + 1], G)[:, k % G]
        size = np.abs(layer.offsets[:, k // G].astype(np.float64)) + np.abs(layer.scales[:, k // G].astype(np.float64)).sum(1)
        return w, np.abs(w) > (q + 1) * 2.0 ** -11 * size

    for row, k, sign in ((0, 3, 1.0), (2, K - 1, -1.0)):
        w, sure = column(k)
        assert np.array_equal(z[row][sure], np.where(sign * w > 0, np.inf, -np.inf)[sure])
        assert not np.isfinite(z[row]).any()
    (w0, sure0), (w1, sure1) = column(40), column(K - 30)
    sure = sure0 & sure1
    same = np.sign(w0) == np.sign(w1)
    assert np.array_equal(z[M - 1][sure & same], np.where(w0 > 0, np.inf, -np.inf)[sure & same])
    assert np.isnan(z[M - 1][sure & ~same]).all()


# the fragment kernel's clusters (digits, halves at G = 64) and the rebuild of few tokens (clusters, whole tiles, equal shares)
@pytest.mark.parametrize("q,g,N,K,M", [(3, 128, 4096, 4096, 4), (2, 64, 1300, 3648, 20), (2, 128, 4096, 4096, 16), (2, 128, 28672, 1024, 9), (4, 128, 21500, 2048, 32)])
def test_captured_batches_read_what_is_there_at_replay(q, g, N, K, M):
    layer = workloads.hlq_layer(78, f"tmem/graph/{q}/{g}/{N}/{K}", q, g, N, K)
    packed = pack_layer(layer)
    Xs = [synth.activations(78, f"tmem/graph/x/{i}/{M}/{K}", M, K) for i in range(3)]
    eager = [gemm_f32(X, packed, N, K) for X in Xs]
    x = x_dev(Xs[0])
    Y = torch.zeros((2, M, N), dtype=torch.float32, device="cuda")
    stream = torch.cuda.Stream()
    elutq.elutq_reserve(M, N, K, stream)
    stream.synchronize()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for i in range(2):                                   # twice: the second begins while the first is still running
            elutq.elutq_lut_gemm_f32(x, packed, Y[i], M, N, K, 0)
    for X, want in zip(Xs, eager):
        x.copy_(x_dev(X))
        Y.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(Y[0].cpu().numpy(), want) and np.array_equal(Y[1].cpu().numpy(), want)
    graph.reset()
    assert elutq.elutq_device_status(stream) == 0
