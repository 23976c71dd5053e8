"""GPU parity of the fragment kernel (batches of 3 to 8 rows and two rows of some sizes at G = 128, any from 3 rows on at G = 64): bit-planes
contracted on the tensor cores as they are, scales applied to fp32 sums.

Tolerance.  As halves, activations are scaled by powers of two (exact but for 2^-33 of the row's largest), products are exact, the
MMAs' fp32 sums run over one group and are truncated (at most 2^-23 per step of 16 k), the groups are added in fp32: the same
order as the look-up kernels' K * 2^-24 * A per element, doubled for the truncation, and 5e-6 in norm.  As bytes (up to four rows at
G = 128 but for three and four at q = 1) activations and group sums are exact; the same bound, and a closer one where it matters.
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

# (q, G, N, K, M): edges of the 8- and 16-row blocks and of the 128-row tile, K ending inside a 512-k chunk and
# a 64-k half step, one tile and one chunk, row tiles shared by several CTAs, every q
CASES = [(2, 128, 128, 512, 3), (1, 128, 17, 128, 8), (3, 128, 129, 640, 7), (4, 128, 1000, 1408, 8), (2, 128, 4096, 4096, 5),
         (4, 128, 300, 4224, 8), (2, 64, 129, 640, 9), (3, 64, 127, 64, 3), (2, 64, 256, 1088, 16), (4, 64, 333, 2880, 17), (3, 64, 1000, 1984, 33),
         (1, 64, 2048, 4096, 32)]


@pytest.mark.parametrize("q,G,N,K,M", CASES)
def test_fragment_kernel_matches_oracle(q, G, N, K, M):
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_FRAGMENT
    layer = workloads.hlq_layer(60, f"frag/{q}/{G}/{N}/{K}", q, G, N, K, signed_scales=(q % 2 == 1))
    X = synth.activations(60, f"frag/x/{M}/{K}", M, K, outliers=True)
    X[0] *= np.float16(2.0 ** -12)                       # rows of very different size: each has its own exponent
    X[-1] *= np.float16(100.0)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert max(hlq.rel_fro_error(y[m], ref[m]) for m in range(M)) <= 5e-6
    A = hlq.magnitude_bound(X, layer.scales, layer.offsets, G)
    assert np.all(np.abs(y - ref) <= 2 * K * 2.0 ** -24 * A)
    assert np.array_equal(y.view(np.uint32), gemm_f32(X, packed, N, K).view(np.uint32))       # and the tickets are zero again
    ys = gemm_f32(X, packed, N, K, elutq.FLAG_SKIP_OFFSET)
    yb = gemm_f32(X, packed, N, K, elutq.FLAG_OFFSET_ONLY)
    assert max(hlq.rel_fro_error(ys[m], hlq.scale_term(X, layer.planes, layer.scales, G)[m]) for m in range(M)) <= 5e-6
    assert max(hlq.rel_fro_error(yb[m], hlq.offset_term(X, layer.offsets, G)[m]) for m in range(M)) <= 5e-6


# Up to four rows as digits of 8 bits: edges of the row tile, K of one step and inside a chunk, tiles of one and of many parts, two rows
@pytest.mark.parametrize("q,N,K,M", [(1, 17, 128, 4), (3, 129, 640, 4), (4, 1000, 1408, 3), (2, 4100, 4224, 2), (3, 5003, 3456, 2), (4, 300, 14336, 4)])
def test_rows_as_digits(q, N, K, M):
    test_fragment_kernel_matches_oracle(q, 128, N, K, M)
    # one element of every step much larger than the rest, against the bound of the whole sum (results without it: the next test)
    layer = workloads.hlq_layer(68, f"frag/digits/{q}/{N}/{K}", q, 128, N, K)
    X = synth.activations(68, f"frag/digits/x/{M}/{K}", M, K)
    X[:, 5::128] = np.float16(2.0 ** 13)
    y, ref = gemm_f32(X, pack_layer(layer), N, K), hlq.matmul(X, layer.planes, layer.scales, layer.offsets, 128)
    assert np.all(np.abs(y - ref) <= 2 * K * 2.0 ** -24 * hlq.magnitude_bound(X, layer.scales, layer.offsets, 128))


def clear_of_large_values(seed, q, N, K, M, large, size):
    """A layer and activations of the given size with one large value in every 128 k, whose bits are clear and whose group has no offset:
    no result depends on it.  Returns also the activations without it."""
    layer = workloads.hlq_layer(seed, f"frag/large/{q}/{N}/{K}", q, 128, N, K)
    at = 128 * np.arange(K // 128) + 37 * np.arange(K // 128) % 128
    layer.planes[:, :, at] = 0
    layer.offsets[:] = 0
    X = (synth.activations(seed, f"frag/large/x/{M}/{K}", M, K).astype(np.float32) * size).astype(np.float16)
    X[:, at] = 0
    with_large = X.copy()
    with_large[:, at] = np.float16(large)
    return layer, with_large, X


# Digits hold every value exactly, also next to one of another size.  Bound: a result is a sum of K / 128 groups of q products, each exact up to
# one rounding in its lower and one in its upper digits' part (together at most 3 |x|), added over a step, the chunks, the four steps of a chunk and
# the parts of a tile: at most q + K / 512 + 11 roundings.  Without its lowest digit a value would be off by 2^-21 of the large one.
@pytest.mark.parametrize("q,N,K,M", [(1, 4100, 4224, 2), (2, 4100, 4224, 2), (4, 4100, 4224, 2), (2, 300, 1408, 4), (3, 129, 640, 3), (4, 300, 4224, 4)])
@pytest.mark.parametrize("large,size", [(2.0 ** 10, 0.02), (2.0 ** 13, 1.0), (-65504.0, 1.0), (65504.0, 2.0 ** -18)])
def test_values_next_to_a_large_one_keep_every_bit(q, N, K, M, large, size):
    assert elutq.elutq_gemm_kernel(M, N, K, q, 128) == elutq.KERNEL_FRAGMENT
    layer, X, small = clear_of_large_values(69, q, N, K, M, large, size)
    packed = pack_layer(layer)
    ref = hlq.matmul(small, layer.planes, layer.scales, layer.offsets, 128)
    A = hlq.magnitude_bound(small, layer.scales, layer.offsets, 128)
    for flags in (0, elutq.FLAG_SKIP_OFFSET):
        y = gemm_f32(X, packed, N, K, flags)
        assert np.all(np.abs(y - ref) <= 3 * (q + K / 512 + 11) * 2.0 ** -24 * A)
        assert hlq.rel_fro_error(y, ref) <= 4e-7           # (about 1e-7)


@pytest.mark.parametrize("q,N,K,M", [(2, 4100, 4224, 2), (3, 300, 1408, 4)])
def test_group_sums_are_fp32_sums(q, N, K, M):
    # many values of one sign that are small next to one: a sum of 128 in pairs has 7 roundings, and the groups' products and sums as above
    layer = workloads.hlq_layer(70, f"frag/sums/{q}/{N}/{K}", q, 128, N, K)
    X = np.full((M, K), np.float16(0.49 * 2.0 ** -11))
    X[:, 77::128] = np.float16(2.0 ** 13)
    y, ref = gemm_f32(X, pack_layer(layer), N, K, elutq.FLAG_OFFSET_ONLY), hlq.offset_term(X, layer.offsets, 128)
    A = hlq.offset_term(np.abs(X), np.abs(layer.offsets), 128)
    assert np.all(np.abs(y - ref) <= (7 + K / 512 + 11) * 2.0 ** -24 * A)
    assert hlq.rel_fro_error(y, ref) <= 7 * 2.0 ** -24


def test_fragment_kernel_reports_a_wait_that_runs_out():
    q, G, N, K, M = 2, 64, 512, 2048, 12
    layer = workloads.hlq_layer(61, "frag/expiry", q, G, N, K)
    X = synth.activations(61, "frag/expiry/x", M, K)
    packed = pack_layer(layer)
    elutq.elutq_release_scratch()
    Y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, 4096)
    assert elutq.elutq_device_status() == 0x7C05
    elutq.elutq_release_scratch()
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert hlq.rel_fro_error(y, hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)) <= 5e-6


def test_warps_that_give_up_leave_together():
    # K in one chunk and four row tiles per CTA: no barrier but the compute warps' own lies between two runs of units
    q, G, N, K, M = 2, 64, 128 * 148 * 4 - 5, 448, 9
    layer = workloads.hlq_layer(63, "frag/expiry/runs", q, G, N, K)
    X = synth.activations(63, "frag/expiry/runs/x", M, K)
    packed = pack_layer(layer)
    Y = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    for limit in (64, 1000, 4096):
        elutq.elutq_release_scratch()
        elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, limit)
        assert elutq.elutq_device_status() == 0x7C05
    elutq.elutq_release_scratch()
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert hlq.rel_fro_error(y, hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)) <= 5e-6


@pytest.mark.parametrize("G,N,M", [(64, 1024, 8), (64, 2900, 16), (64, 2900, 32), (128, 1024, 4), (128, 12800, 8)])
def test_long_sums_are_as_exact_as_the_look_up_kernels(G, N, M):
    # Many chunks and planes: fp32 roundings of one long chain would show.  The error in norm over N * M >= 4096 results varies by
    # about 1 / sqrt(2 N M) (1 %) from sample to sample: 5 % leaves room for that and for nothing else.
    q, K = 4, 14336 if N < 10000 else 4096
    layer = workloads.hlq_layer(65, f"frag/exact/{G}/{N}", q, G, N, K)
    X = synth.activations(65, f"frag/exact/x/{M}", M, K)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    lut = hlq.rel_fro_error(gemm_f32(X, packed, N, K, elutq.FLAG_LUT_ONLY), ref)
    assert hlq.rel_fro_error(gemm_f32(X, packed, N, K), ref) <= 1.05 * lut


@pytest.mark.parametrize("G,M", [(128, 3), (128, 8), (64, 5), (64, 20)])
@pytest.mark.parametrize("values", [(np.inf,), (-np.inf,), (np.inf, np.inf), (np.inf, -np.inf), (np.nan,), (np.inf, np.nan)])
def test_activations_that_are_not_finite(G, M, values):
    # the same kind of result as from the decode kernel row by row, and no other row changes
    q, N, K = 2, 300, 1024
    layer = workloads.hlq_layer(66, f"frag/inf/{G}", q, G, N, K)
    layer.offsets[::7] = 0
    X = synth.activations(66, f"frag/inf/x/{M}", M, K)
    packed = pack_layer(layer)
    clean = gemm_f32(X, packed, N, K)
    X[1, 200:200 + 3 * len(values):3] = values
    y = gemm_f32(X, packed, N, K)
    one = gemm_f32(X[1:2], packed, N, K)[0]
    for kind in (np.isnan, np.isposinf, np.isneginf):
        assert np.array_equal(kind(y[1]), kind(one))
    keep = np.arange(M) != 1
    assert np.array_equal(y[keep], clean[keep])


def plain_row(x, layer, G, flags):
    """One row of the product in 64 bits, element by element: what is not selected is not there (0 * infinity does not come up)."""
    x, groups = x.astype(np.float64), (layer.N, layer.K // G, G)
    with np.errstate(invalid="ignore", over="ignore"):
        y = np.zeros(layer.N)
        if flags != elutq.FLAG_OFFSET_ONLY:
            for j in range(layer.q):
                y += (layer.scales[:, :, j].astype(np.float64) * np.where(layer.planes[j] != 0, x, 0.0).reshape(groups).sum(-1)).sum(-1)
        if flags != elutq.FLAG_SKIP_OFFSET:
            y += (layer.offsets.astype(np.float64) * x.reshape(groups[1:]).sum(-1)).sum(-1)
    return y


@pytest.mark.parametrize("q,N,K,M", [(1, 4100, 4224, 2), (2, 4100, 4224, 2), (3, 300, 1024, 4), (4, 300, 1408, 3), (2, 300, 14336, 4)])
@pytest.mark.parametrize("where", ["activation", "activations", "nan", "scale", "offset"])
def test_infinities_up_to_four_rows(q, N, K, M, where):
    # every result is of the kind that the sum of its terms has, finite ones have their value, and no other row or output changes
    layer = workloads.hlq_layer(71, f"frag/inf/{q}/{N}/{K}", q, 128, N, K)
    layer.offsets[::7] = 0
    X = synth.activations(71, f"frag/inf/x/{M}/{K}", M, K)
    clean, rows = gemm_f32(X, pack_layer(layer), N, K), np.arange(M)
    if where in ("activation", "activations", "nan"):
        X[1, 200] = np.nan if where == "nan" else np.inf
        if where == "activations":
            X[1, K - 3] = -np.inf
        touched = np.broadcast_to((rows == 1)[:, None], (M, N))
    else:
        (layer.scales[:, :, 0] if where == "scale" else layer.offsets)[5:40, 1] = np.inf
        touched = np.broadcast_to((np.arange(N) >= 5) & (np.arange(N) < 40), (M, N))
    packed = pack_layer(layer)
    for flags in (0, elutq.FLAG_SKIP_OFFSET, elutq.FLAG_OFFSET_ONLY):
        y = gemm_f32(X, packed, N, K, flags)
        ref = np.stack([plain_row(x, layer, 128, flags) for x in X])
        for kind in (np.isnan, np.isposinf, np.isneginf):
            assert np.array_equal(kind(y), kind(ref))
        finite = np.isfinite(ref)
        A = hlq.magnitude_bound(np.nan_to_num(X, posinf=0.0, neginf=0.0), np.nan_to_num(layer.scales, posinf=0.0), np.nan_to_num(layer.offsets, posinf=0.0), 128)
        assert np.all(np.abs(np.where(finite, y, 0) - np.where(finite, ref, 0)) <= 2 * K * 2.0 ** -24 * A)
        if flags == 0:
            assert np.array_equal(y[~touched], clean[~touched])
    assert elutq.elutq_device_status() == 0


@pytest.mark.parametrize("q,N,K,M", [(1, 129, 64, 257), (2, 1000, 1024, 33), (2, 2048, 4096, 130), (3, 4000, 2880, 57), (4, 300, 4160, 100)])
def test_batch_blocks_of_one_launch(q, N, K, M):
    # blocks of 8 and 16 rows with a remainder, several to a row tile, output tiles shared by CTAs; one launch, no call slower for its rows
    layer = workloads.hlq_layer(67, f"frag/blocks/{q}/{N}/{K}", q, 64, N, K)
    X = synth.activations(67, f"frag/blocks/x/{M}/{K}", M, K, outliers=True)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, 64)
    y = gemm_f32(X, packed, N, K)
    before = elutq.elutq_launch_count()
    again = gemm_f32(X, packed, N, K)
    assert elutq.elutq_launch_count() == before + 1
    assert max(hlq.rel_fro_error(y[m], ref[m]) for m in range(M)) <= 5e-6
    assert np.array_equal(y, again)
    assert elutq.elutq_device_status() == 0


# Few output tiles, most of them shared by a cluster of CTAs (1500 x 4736, 200 x 7680 and 257 x 5184 have more chunks than a cluster has CTAs: tickets), shares of
# unequal length, a last chunk of one step, ragged rows, several batch blocks; the widest call that clusters of two take, and one tile more
@pytest.mark.parametrize("q,G,N,K,M", [(3, 128, 1500, 4736, 4), (1, 128, 130, 1024, 4), (2, 128, 4100, 4224, 2), (4, 128, 3000, 2688, 8), (1, 128, 200, 7680, 3),
                                       (2, 64, 1300, 3648, 7), (3, 64, 257, 5184, 16), (4, 64, 1000, 2112, 40), (2, 128, 74 * 128, 1152, 6), (2, 128, 74 * 128 + 1, 1152, 6)])
def test_output_tiles_of_clusters(q, G, N, K, M):
    layer = workloads.hlq_layer(72, f"frag/clusters/{q}/{G}/{N}/{K}", q, G, N, K)
    X = synth.activations(72, f"frag/clusters/x/{M}/{K}", M, K, outliers=True)
    packed = pack_layer(layer)
    assert elutq.elutq_gemm_kernel(M, N, K, q, G) == elutq.KERNEL_FRAGMENT
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    y = gemm_f32(X, packed, N, K)
    assert elutq.elutq_device_status() == 0
    assert max(hlq.rel_fro_error(y[m], ref[m]) for m in range(M)) <= 5e-6
    assert np.all(np.abs(y - ref) <= 2 * K * 2.0 ** -24 * hlq.magnitude_bound(X, layer.scales, layer.offsets, G))
    assert np.array_equal(y, gemm_f32(X, packed, N, K))
    Y = torch.full((M, N), 1.5, dtype=torch.float32, device="cuda")
    elutq.elutq_lut_gemm_f32(x_dev(X), packed, Y, M, N, K, elutq.FLAG_ACCUMULATE)
    np.testing.assert_allclose(Y.cpu().numpy(), y + 1.5, rtol=0, atol=1e-5 * np.abs(y).max())
    # a value that is not finite in the share of a later CTA
    X[1, K - 5] = np.inf
    z = gemm_f32(X, packed, N, K)
    keep = np.arange(M) != 1
    assert np.array_equal(z[keep], y[keep]) and not np.isfinite(z[1]).any()


@pytest.mark.parametrize("M,half", [(9, 0), (20, 0), (9, 0x80000000), (20, 0x80000000)])
def test_clusters_report_a_wait_that_runs_out(M, half):
    # in all CTAs, or in every other one: nothing is written where a part is missing, and the next call is whole (ten chunks: tickets, no clusters)
    q, G, N, K = 3, 64, 1500, 4672
    layer = workloads.hlq_layer(73, "frag/clusters/expiry", q, G, N, K)
    X = synth.activations(73, f"frag/clusters/expiry/x/{M}", M, K)
    packed = pack_layer(layer)
    ref = hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)
    for limit in (300, 20000):
        elutq.elutq_release_scratch()
        Y = torch.full((M, N), 7.5, dtype=torch.float32, device="cuda")
        elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, half | limit)
        assert elutq.elutq_device_status() == 0x7C05
        assert torch.all(Y == 7.5)
    elutq.elutq_release_scratch()
    assert hlq.rel_fro_error(gemm_f32(X, packed, N, K), ref) <= 5e-6
    assert elutq.elutq_device_status() == 0


@pytest.mark.parametrize("chunks,tiles,more", [(27, 45, 48), (17, 45, 49), (29, 26, 30), (13, 26, 30)])
def test_fewer_output_tiles_take_no_longer(chunks, tiles, more):
    """As many clusters of three or five CTAs as the device counts as resident do not all find a place behind the call before (a third more time)."""
    q, G, M, K = 4, 64, 4, 512 * chunks - 128
    gen = torch.Generator(device="cuda").manual_seed(75)
    X = torch.randn((M, K), generator=gen, device="cuda").half()

    def us(N):
        planes = torch.randint(0, 2, (q, N, K), generator=gen, device="cuda", dtype=torch.uint8)
        scales = (torch.randn((N, K // G, q), generator=gen, device="cuda") * 0.02).abs().half()
        packed = elutq.elutq_pack(planes, scales, torch.zeros((N, K // G), dtype=torch.float16, device="cuda"), q, G, N, K)
        Y = torch.empty((M, N), dtype=torch.float16, device="cuda")
        times = []
        for _ in range(9):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                elutq.elutq_lut_gemm(X, packed, Y, M, N, K)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 50)
        return sorted(times)[4]

    assert us(128 * tiles) <= 1.1 * us(128 * more)


def parts_meet_in_the_workspace(X, packed, N, K):
    """Whether the call leaves parts of its output tiles in the workspace (tickets).  With fewer output tiles than SMs every tile is shared: if not there, in a cluster."""
    M = X.shape[0]
    assert -(-N // 128) * -(-M // 8) < torch.cuda.get_device_properties(0).multi_processor_count
    ws = torch.zeros(elutq.elutq_workspace_bytes(M, N, K), dtype=torch.uint8, device="cuda")
    elutq.elutq_workspace_init(ws)
    before = ws.clone()
    Y = torch.empty((M, N), dtype=torch.float32, device="cuda")
    elutq.elutq_lut_gemm_ws(x_dev(X), packed, Y, M, N, K, elutq.FLAG_OUT_F32, ws)
    return not torch.equal(ws, before)


# Digits of four rows in shares of two units; halves of three rows, of 16 and of 7 in clusters of eight; blocks of 16 rows in clusters of three
@pytest.mark.parametrize("q,G,N,K,M", [(3, 128, 3700, 4096, 4), (1, 128, 200, 3712, 3), (3, 64, 257, 3904, 16), (4, 64, 1500, 3648, 7), (2, 64, 4400, 2880, 16)])
def test_clusters_of_every_form(q, G, N, K, M):
    X = synth.activations(72, f"frag/clusters/x/{M}/{K}", M, K, outliers=True)
    packed = pack_layer(workloads.hlq_layer(72, f"frag/clusters/{q}/{G}/{N}/{K}", q, G, N, K))
    assert not parts_meet_in_the_workspace(X, packed, N, K)
    test_output_tiles_of_clusters(q, G, N, K, M)


# clusters of 4, of 8, of 5 (whose first CTA is sometimes the one that gives up), and shares of several units
@pytest.mark.parametrize("N,K,M", [(1000, 1984, 20), (1500, 3648, 9), (890, 2496, 9), (800, 4608, 40)])
@pytest.mark.parametrize("half", [0, 0x80000000])
def test_clusters_write_nothing_where_a_part_is_missing(N, K, M, half):
    q, G = 3, 64
    layer = workloads.hlq_layer(76, "frag/clusters/missing", q, G, N, K)
    X = synth.activations(76, f"frag/clusters/missing/x/{M}", M, K)
    packed = pack_layer(layer)
    assert not parts_meet_in_the_workspace(X, packed, N, K)
    for limit in (300, 20000):
        elutq.elutq_release_scratch()
        Y = torch.full((M, N), 7.5, dtype=torch.float32, device="cuda")
        elutq.elutq_test_wait_expiry(x_dev(X), packed, Y, M, N, K, half | limit)
        assert elutq.elutq_device_status() == 0x7C05
        assert torch.all(Y == 7.5)
    elutq.elutq_release_scratch()
    assert hlq.rel_fro_error(gemm_f32(X, packed, N, K), hlq.matmul(X, layer.planes, layer.scales, layer.offsets, G)) <= 5e-6
    assert elutq.elutq_device_status() == 0
