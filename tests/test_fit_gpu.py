"""GPU parity of elutq_hlq_fit (Algorithm 1) against the fp64 oracle: planes and fp16 parameters bit for bit."""
import numpy as np
import pytest
import torch

import paper_2510_19482_b200 as elutq
import workloads
from oracle import fit as ofit
from oracle import hlq
from tests.gpu_util import gemm_f32, to_dev

pytestmark = pytest.mark.gpu

SORTED_MIN_GROUPS = 24576        # from this many groups on elutq_hlq_fit sorts the groups for every q and G at ten rounds (without a trace)


def _fit_gpu(W, q, G, t_max=10, trace=False):
    Wd = to_dev(W.view(np.int16)).view(torch.float16)
    out = elutq.elutq_hlq_fit(Wd, q, G, t_max, trace)
    torch.cuda.synchronize()
    planes = out[0].cpu().numpy()
    scales = out[1].cpu().view(torch.int16).numpy().view(np.float16)
    offsets = out[2].cpu().view(torch.int16).numpy().view(np.float16)
    if trace:
        return planes, scales, offsets, out[3].cpu().numpy()
    return planes, scales, offsets


def _same_bits(a, b):
    return np.array_equal(np.ascontiguousarray(a).view(np.uint16), np.ascontiguousarray(b).view(np.uint16))


@pytest.mark.parametrize("q", [1, 2, 3, 4])
@pytest.mark.parametrize("G", [32, 64, 128])
def test_fit_matches_oracle_bit_for_bit(q, G):
    N, K = 37, 1024                       # 37 rows: the last CTA of 8 groups is ragged for every G
    W = workloads.dense_weights(23, f"fit{q}{G}", N, K)
    p_ref, s_ref, z_ref, tr_ref = ofit.fit(W, q, G, 10, trace=True)
    p, s, z, tr = _fit_gpu(W, q, G, 10, trace=True)
    assert np.array_equal(p, p_ref)
    assert _same_bits(s, s_ref) and _same_bits(z, z_ref)
    assert np.allclose(tr, tr_ref, rtol=1e-10, atol=1e-20)
    assert np.all(tr[1:] <= tr[:-1] * (1 + 1e-12) + 1e-18)


@pytest.mark.parametrize("t_max", [1, 3])
def test_fit_short_runs(t_max):
    W = workloads.dense_weights(29, "fit-short", 16, 512)
    p_ref, s_ref, z_ref = ofit.fit(W, 3, 128, t_max)
    p, s, z = _fit_gpu(W, 3, 128, t_max)
    assert np.array_equal(p, p_ref) and _same_bits(s, s_ref) and _same_bits(z, z_ref)


def test_fit_degenerate_groups():
    """Constant groups (singular from the first round), two-valued groups (higher planes dependent), grid weights."""
    q, G = 3, 32
    rng = np.random.default_rng(4)
    W = workloads.dense_weights(31, "fit-deg", 8, 256)
    W[0, :32] = np.float16(0.0625)                                            # constant
    W[1, 32:64] = np.where(rng.integers(0, 2, 32) == 1, np.float16(0.5), np.float16(-0.25))   # two values
    c = rng.integers(0, 8, 32)
    c[:8] = np.arange(8)
    W[2, 64:96] = (-0.125 + 2.0 ** -6 * c).astype(np.float16)                 # exactly on a uniform grid
    p_ref, s_ref, z_ref = ofit.fit(W, q, G, 10)
    p, s, z = _fit_gpu(W, q, G, 10)
    assert np.array_equal(p, p_ref) and _same_bits(s, s_ref) and _same_bits(z, z_ref)
    rec = hlq.reconstruct(p, s, z, G)
    assert np.array_equal(rec[0, :32], W[0, :32].astype(np.float64))
    assert np.allclose(rec[1, 32:64], W[1, 32:64].astype(np.float64), atol=1e-3)
    assert np.allclose(rec[2, 64:96], W[2, 64:96].astype(np.float64), atol=2e-4)


def test_fit_then_pack_then_product():
    """The offline chain on the device: fit -> pack -> GEMV equals the oracle product of the oracle's fit."""
    q, G, N, K = 2, 128, 64, 1024
    W = workloads.dense_weights(37, "fit-chain", N, K)
    Wd = to_dev(W.view(np.int16)).view(torch.float16)
    planes, scales, offsets = elutq.elutq_hlq_fit(Wd, q, G)
    packed = elutq.elutq_pack(planes, scales, offsets, q, G, N, K)
    X = workloads.activations(37, "fit-chain", 1, K)
    Y = gemm_f32(X, packed, N, K)
    p_ref, s_ref, z_ref = ofit.fit(W, q, G)
    Y_ref = hlq.matmul(X, p_ref, s_ref, z_ref, G)
    assert hlq.rel_fro_error(Y, Y_ref) <= 5e-6
    # and the fitted layer approximates the dense product far better than its energy
    Y_dense = X.astype(np.float64) @ W.astype(np.float64).T
    assert hlq.rel_fro_error(Y_ref, Y_dense) < 0.5


# (q, G, N, K): the last warp of 32 groups ragged, fewer than 32 groups, a block of 128 weights cut in two by the end
@pytest.mark.parametrize("q,G,N,K", [(1, 128, 37, 1024), (2, 128, 1, 384), (2, 64, 33, 320), (3, 32, 7, 160), (3, 128, 65, 512), (4, 64, 50, 1088),
                                     (4, 32, 129, 96), (4, 128, 64, 2048)])
@pytest.mark.parametrize("shift", [0, 1])
def test_fit_of_sorted_groups_matches_oracle_bit_for_bit(q, G, N, K, shift):
    """Without a trace the groups' sorted form runs (from a number of groups on: tiled here to reach it); `shift` = an input that
    starts two bytes after an aligned address.  Groups on a grid, with few values, with equal or very different magnitudes."""
    rng = np.random.default_rng(41)
    W = workloads.dense_weights(41, f"fit-sorted{q}{G}{N}", N, K)
    flat = W.reshape(-1, G)
    n = flat.shape[0]
    flat[0] = np.float16(0.25)
    flat[n // 2] = rng.choice(np.array([-3.0, 0.0, -0.0, 5.0], dtype=np.float16), G)
    flat[n // 3] = (0.5 * rng.integers(-2 ** (q - 1), 2 ** (q - 1), G)).astype(np.float16)
    flat[n - 1] = (flat[n - 1].astype(np.float64) * 1e4).astype(np.float16)
    flat[n // 4] = (flat[n // 4].astype(np.float64) * 2.0 ** -13).astype(np.float16)      # subnormal values
    copies = -(-SORTED_MIN_GROUPS // n)
    Wall = np.concatenate([W] * copies)
    buf = torch.zeros(Wall.size + 8, dtype=torch.int16, device="cuda")
    Wd = buf[shift: shift + Wall.size].view(Wall.shape)
    Wd.copy_(to_dev(Wall.view(np.int16)))
    p, s, z = elutq.elutq_hlq_fit(Wd.view(torch.float16), q, G, 10)
    p = p.cpu().numpy()
    s, z = (t.cpu().view(torch.int16).numpy().view(np.float16) for t in (s, z))
    p_ref, s_ref, z_ref = ofit.fit(W, q, G, 10)
    for c in range(copies):
        rows = slice(c * N, (c + 1) * N)
        assert np.array_equal(p[:, rows], p_ref)
        assert _same_bits(s[rows], s_ref) and _same_bits(z[rows], z_ref)


# N rows of 1024 weights: the first number of groups that is sorted
@pytest.mark.parametrize("q,G,N,t_max", [(1, 64, 2048, 1), (2, 64, 768, 2), (3, 128, 1536, 2), (4, 32, 384, 1), (2, 128, 4096, 1), (2, 128, 1536, 7)])
def test_fit_on_both_sides_of_the_sorted_form_s_lower_end(q, G, N, t_max):
    """The same bits as with a trace, which takes the direct form at any size."""
    W = workloads.dense_weights(42, f"fit-ends{q}{G}", N, 1024)
    Wd = to_dev(W.view(np.int16)).view(torch.float16)
    for rows in (N - 1, N):
        a = elutq.elutq_hlq_fit(Wd[:rows], q, G, t_max)
        b = elutq.elutq_hlq_fit(Wd[:rows], q, G, t_max, trace=True)
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))


# the same with fewer groups, which are the direct form's with and without a trace, and weights that begin 8 bytes after a 16-byte boundary
@pytest.mark.parametrize("q,G,N,t_max", [(1, 64, 640, 1), (2, 64, 256, 2), (3, 128, 512, 2), (4, 32, 192, 1), (2, 128, 1280, 1), (2, 128, 512, 7), (4, 128, 384, 10)])
@pytest.mark.parametrize("shift", [0, 4])
def test_fit_on_both_sides_of_the_lane_sort_s_lower_end(q, G, N, t_max, shift):
    W = workloads.dense_weights(43, f"fit-lanes{q}{G}", N, 1024)
    buf = torch.zeros(W.size + 8, dtype=torch.int16, device="cuda")
    Wd = buf[shift: shift + W.size].view(W.shape)
    Wd.copy_(to_dev(W.view(np.int16)))
    Wd = Wd.view(torch.float16)
    for rows in (N - 1, N):
        a = elutq.elutq_hlq_fit(Wd[:rows], q, G, t_max)
        b = elutq.elutq_hlq_fit(Wd[:rows], q, G, t_max, trace=True)
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))


def test_fit_of_weights_next_to_a_place():
    """Weights at, and an ulp or two beside, the middle of two candidates: the exact choice decides, with the lower code where both are equally far."""
    rng = np.random.default_rng(44)
    q, G, n = 2, 128, 4096 + 32
    mid = np.array([0.5, 1.5, 2.5], dtype=np.float16)
    near = np.concatenate([mid, np.nextafter(mid, np.float16(9)), np.nextafter(mid, np.float16(-9)), np.nextafter(np.nextafter(mid, np.float16(9)), np.float16(9))])
    W = rng.choice(np.concatenate([near, np.arange(4, dtype=np.float16)]), (n, G)).astype(np.float16)
    W[:, 0], W[:, 1] = 0.0, 3.0                          # the first round's candidates are 0, 1, 2, 3
    W *= np.float16(2.0) ** rng.integers(-12, 8, (n, 1)).astype(np.float16)
    Wd = to_dev(W.view(np.int16)).view(torch.float16)
    for t_max in (2, 5):
        a, b = elutq.elutq_hlq_fit(Wd, q, G, t_max), elutq.elutq_hlq_fit(Wd, q, G, t_max, trace=True)
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))


@pytest.mark.parametrize("q,G,groups", [(2, 128, 4096), (2, 128, 12000), (4, 128, 8192), (2, 64, 8192), (3, 32, 8192)])
def test_groups_that_settle_at_once_take_no_longer_than_their_rounds(q, G, groups):
    """Groups of one value are done after two rounds, whatever number is asked for: below the sorted form's lower end they cost what the direct form costs (the
    call with a trace, which writes more), not a sort and a warp's groups in turn (three to seven times as much)."""
    W = torch.full((groups, G), 0.25, dtype=torch.float16, device="cuda")

    def us(trace):
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(10):
                elutq.elutq_hlq_fit(W, q, G, 10, trace)
            b.record()
            b.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return sorted(times)[3]

    us(False), us(True)
    assert us(False) <= 1.5 * us(True)


# The sorted form's lower ends again, with weights that begin 8 and 2 bytes after a 16-byte boundary (loads of 2 bytes instead of 16; of the output's weights, too)
@pytest.mark.parametrize("q,G,N,t_max", [(1, 64, 2048, 1), (2, 64, 768, 2), (3, 128, 1536, 2), (4, 32, 384, 1), (2, 128, 1536, 7), (4, 128, 768, 10)])
@pytest.mark.parametrize("shift", [1, 4])
def test_sorted_form_of_weights_off_the_boundary(q, G, N, t_max, shift):
    test_fit_on_both_sides_of_the_lane_sort_s_lower_end(q, G, N, t_max, shift)


@pytest.mark.parametrize("q,G", [(1, 128), (2, 128), (3, 64), (4, 32), (4, 128)])
def test_first_choice_next_to_a_place(q, G):
    """Weights at, and an ulp or two beside, the middle of two candidates, in so many groups that all q and G are sorted from one round on.  After one round the
    planes are the first choice itself, so that a wrong one cannot have been mended by a later round."""
    rng = np.random.default_rng(45)
    top, n = 2 ** q - 1, 4128
    grid = np.arange(top + 1).astype(np.float16)
    mid = (grid[:-1].astype(np.float32) + 0.5).astype(np.float16)
    up = np.nextafter(mid, np.float16(99))
    near = np.concatenate([mid, up, np.nextafter(mid, np.float16(-9)), np.nextafter(up, np.float16(99))])
    W = rng.choice(np.concatenate([near, grid]), (n, G)).astype(np.float16)
    W[:, 0], W[:, 1] = 0.0, top                          # the first round's candidates are 0 .. top
    W *= np.float16(2.0) ** rng.integers(-12, 8, (n, 1)).astype(np.float16)
    Wd = to_dev(W.view(np.int16)).view(torch.float16).repeat(32, 1)
    for t_max in (1, 2, 5):
        a, b = elutq.elutq_hlq_fit(Wd, q, G, t_max), elutq.elutq_hlq_fit(Wd, q, G, t_max, trace=True)
        for x, y in zip(a[:3], b[:3]):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8))
