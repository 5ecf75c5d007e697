"""K1 parity: SSC score + lowest-c selection on the GPU is bit-exact with the
oracle (Sec. 4.1-4.2 Eq. ssc / Eq. normalize; Algorithm 1 SSC) on the
selection-only workload (16^3 tokens x 8 channels, batch 1-64, quotas
10-90%), on ties, constant fields, NaN / Inf, edge quotas and other grids."""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_clean, dev_i32, dev_u16, handle_for
from paper_2511_22533_gb300 import synth

pytestmark = pytest.mark.gpu


def _shape(grid):
    return synth.ModelShape(grid, 8, 128, 1, 4, 4, 64, 128, 25, 64)


@pytest.fixture(scope="module")
def h16():
    h, _, _ = handle_for(_shape(16), max_batch=64)
    yield h
    h.close()


def _run(h, hist, quotas):
    B, N = hist.shape[1], hist.shape[2]
    v1, v2 = dev_u16(hist[2]), dev_u16(hist[1])
    q = dev_i32(quotas)
    idx = torch.full((B, N), -7, dtype=torch.int32, device="cuda")
    na = torch.zeros(B, dtype=torch.int32, device="cuda")
    mask = torch.full((B, N), 9, dtype=torch.uint8, device="cuda")
    h.ssc_select(v1, v2, B, q, idx, na, mask)
    torch.cuda.synchronize()
    assert_clean(h)
    return idx.cpu().numpy(), na.cpu().numpy(), mask.cpu().numpy()


def _check(orc, hist, quotas, idx, na, mask, omega=0.7):
    N = hist.shape[2]
    for b in range(hist.shape[1]):
        s = orc.ssc_score(hist[2, b], hist[1, b], omega)
        cached, aidx = orc.select(s, int(quotas[b]))
        assert na[b] == len(aidx) == N - min(max(int(quotas[b]), 0), N)
        np.testing.assert_array_equal(mask[b], cached, err_msg=f"sample {b}")
        np.testing.assert_array_equal(idx[b, :na[b]], aidx, err_msg=f"sample {b}")


@pytest.mark.parametrize("B", [1, 8, 64])
def test_selection_sweep_drift(orc, h16, B):
    hist = synth.velocity_history(16, 8, B, seed=B, kind="drift")
    N = 4096
    qs = np.array([int(np.floor(q * N)) for q in np.tile([0.1, 0.3, 0.5, 0.7, 0.9], 13)[:B]], np.int32)
    idx, na, mask = _run(h16, hist, qs)
    _check(orc, hist, qs, idx, na, mask)


@pytest.mark.parametrize("kind", ["ties", "constant"])
def test_selection_ties_and_constant(orc, h16, kind):
    hist = synth.velocity_history(16, 8, 6, seed=3, kind=kind)
    qs = np.array([1, 409, 2048, 2867, 4000, 4095], np.int32)
    idx, na, mask = _run(h16, hist, qs)
    _check(orc, hist, qs, idx, na, mask)


def test_selection_edge_quotas(orc, h16):
    hist = synth.velocity_history(16, 8, 6, seed=4)
    qs = np.array([0, 4096, -5, 9999, 1, 4095], np.int32)
    idx, na, mask = _run(h16, hist, qs)
    _check(orc, hist, qs, idx, na, mask)
    np.testing.assert_array_equal(idx[0], np.arange(4096))
    assert na.tolist() == [4096, 0, 4096, 0, 4095, 1]


def test_selection_nan_inf(orc, h16):
    hist = synth.velocity_history(16, 8, 2, seed=5)
    f = synth.bf16_bits_to_f32(hist).copy()
    f[2, 0, 17, 3] = np.nan          # NaN velocity: never cached
    f[2, 0, 99, 0] = np.inf          # an infinite magnitude
    f[1, 1, 5, :] = f[2, 1, 5, :]    # a token with zero acceleration
    hist = synth.f32_to_bf16_bits(f)
    qs = np.array([3000, 2000], np.int32)
    idx, na, mask = _run(h16, hist, qs)
    _check(orc, hist, qs, idx, na, mask)
    assert mask[0, 17] == 0


@pytest.mark.parametrize("omega", [0.0, 0.3, 1.0])
def test_selection_omega(orc, omega):
    h, _, _ = handle_for(_shape(16), max_batch=4, omega=omega)
    hist = synth.velocity_history(16, 8, 4, seed=6)
    qs = np.array([500, 1500, 2500, 3500], np.int32)
    idx, na, mask = _run(h, hist, qs)
    _check(orc, hist, qs, idx, na, mask, omega=omega)
    h.close()


@pytest.mark.parametrize("grid,B", [(8, 3), (32, 2)])
def test_selection_other_grids(orc, grid, B):
    h, _, _ = handle_for(_shape(grid), max_batch=B)
    hist = synth.velocity_history(grid, 8, B, seed=grid)
    N = grid ** 3
    qs = np.array([N // 2, int(0.7 * N), N // 10][:B], np.int32)
    idx, na, mask = _run(h, hist, qs)
    _check(orc, hist, qs, idx, na, mask)
    h.close()


def test_selection_batch64_32cubed(orc):
    # the largest selection workload: 64 samples of 32768 tokens (the 32^3
    # grid), quotas 10-90 %, bit-exact on every sample
    h, _, _ = handle_for(_shape(32), max_batch=64)
    hist = synth.velocity_history(32, 8, 64, seed=32)
    N = 32768
    qs = np.array([int(np.floor(q * N)) for q in np.tile([0.1, 0.3, 0.5, 0.7, 0.9], 13)[:64]], np.int32)
    idx, na, mask = _run(h, hist, qs)
    _check(orc, hist, qs, idx, na, mask)
    h.close()


@pytest.mark.parametrize("log2_scale", [25, -40, -70])
def test_selection_at_scaled_velocities(orc, h16, log2_scale):
    # the shared-reciprocal division serves ranges in [2^-98, 2^20]: above it
    # (2^25) the general one runs; at 2^-70 the squares' sums are subnormal
    hist = synth.velocity_history(16, 8, 2, seed=11)
    scaled = synth.f32_to_bf16_bits(np.ldexp(synth.bf16_bits_to_f32(hist), log2_scale))
    qs = np.array([1500, 3001], np.int32)
    idx, na, mask = _run(h16, scaled, qs)
    _check(orc, scaled, qs, idx, na, mask)


def test_selection_mask_at_any_address(orc, h16):
    hist = synth.velocity_history(16, 8, 1, seed=12)
    N = 4096
    idx = torch.full((1, N), -1, dtype=torch.int32, device="cuda")
    na = torch.zeros(1, dtype=torch.int32, device="cuda")
    buf = torch.full((N + 8,), 9, dtype=torch.uint8, device="cuda")
    v1, v2 = dev_u16(hist[2]), dev_u16(hist[1])
    h16.ssc_select(v1, v2, 1, dev_i32([1234]), idx, na, buf[3:])
    torch.cuda.synchronize()
    got = buf.cpu().numpy()
    assert np.all(got[:3] == 9) and np.all(got[3 + N:] == 9)
    _check(orc, hist, np.array([1234]), idx.cpu().numpy(), na.cpu().numpy(), got[None, 3:3 + N])


@pytest.mark.parametrize("case", ["one_digit", "ties_across_ctas", "both_sides_of_the_knee"])
def test_selection_where_the_radix_search_ends(orc, h16, case):
    # the search ends at the first digit whose keys are all cached: after one
    # pass, after all four (ties that must be broken by index), and with scores
    # on both sides of 2^-6, where the keys' spacing changes
    N = 4096
    v = np.zeros((3, 1, N, 8), np.float32)
    if case == "one_digit":
        v[2, 0, :, 0] = np.where(np.arange(N) % 3 == 0, 1.0, 2.0)
        q = np.count_nonzero(np.arange(N) % 3 == 0)
    elif case == "ties_across_ctas":
        v[2, 0, :, 0] = np.where(np.arange(N) % 5 == 0, 1.0, 2.0)
        v[2, 0, 7, 0] = 0.0
        q = 1 + 300
    else:
        v[2, 0, :, 0] = np.exp2(np.random.default_rng(3).uniform(-14, 0, N))
        q = 2500
    hist = synth.f32_to_bf16_bits(v)
    qs = np.array([q], np.int32)
    idx, na, mask = _run(h16, hist, qs)
    _check(orc, hist, qs, idx, na, mask)


def _norm(x):
    s = np.zeros(x.shape[:-1], np.float32)
    for c in range(x.shape[-1]):
        s = s + x[..., c] * x[..., c]
    return np.sqrt(s)


def _vector_of_norm(target, g):
    # bf16 channels whose fp32 norm is `target` to the bit: a greedy expansion of
    # its square from a random first channel
    def floor_bf16(x):
        return (np.asarray(x, np.float32).view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)

    x = np.zeros((4000, 8), np.float32)
    rest = np.full(4000, float(target) ** 2)
    x[:, 0] = floor_bf16(target * g.uniform(0.3, 0.95, 4000))
    for c in range(1, 5):
        rest = rest - x[:, c - 1].astype(np.float64) ** 2
        x[:, c] = floor_bf16(np.sqrt(np.maximum(rest, 0)))
    return x[np.flatnonzero(_norm(x) == target)[0]]


def test_selection_where_one_ulp_of_a_quotient_decides(orc):
    # 510 tokens of an 8^3 grid whose norms lie within 300 neighbouring floats, so
    # that a quotient norm / range off by one ulp changes which are cached for some
    # of the 511 quotas; ranges next to a power of two, with all ones, and others.
    # For two of the ranges the product with the reciprocal alone is that far off
    # (the rest of the score is 0 there), which shows that the quotas can tell.
    N, omega = 512, 0.7
    quotas = np.arange(1, N, dtype=np.int32)
    told = 0
    h, _, _ = handle_for(_shape(8), max_batch=64)
    for mant in (1, 2, 3, 2 ** 23 - 1, 2 ** 23 - 2, 2 ** 22 - 1, 2 ** 22, 0x2AAAAB):
        g = np.random.default_rng(mant)
        top = np.uint32(127 << 23 | mant).view(np.float32)
        base = np.float32(0.37 + 0.6 * g.random()) * top
        v1 = np.zeros((N, 8), np.float32)  # token N - 2 stays 0: the range is `top`
        for i in range(N - 2):
            v1[i] = _vector_of_norm((base.view(np.uint32) + np.uint32(g.integers(0, 300))).view(np.float32), g)
        v1[N - 1] = _vector_of_norm(top, g)
        v2 = v1.copy()
        v2[0, 7] = -1.0  # A is 1 for this token and 0 for the others
        perm = g.permutation(N)
        b1, b2 = (synth.f32_to_bf16_bits(x[perm]) for x in (v1, v2))
        score = orc.ssc_score(b1, b2, omega)
        rough = np.where(perm == 0, score, (np.float32(1) - np.float32(omega)) * (_norm(v1[perm]) * (np.float32(1) / top)))
        for q0 in range(0, len(quotas), 64):
            qs = quotas[q0:q0 + 64]
            hist = np.stack([b2 * 0, b2, b1])[:, None].repeat(len(qs), 1)
            idx, na, mask = _run(h, hist, qs)
            for b, c in enumerate(qs):
                cached, aidx = orc.select(score, int(c))
                np.testing.assert_array_equal(mask[b], cached, err_msg=f"range {mant:#x}, quota {c}")
                np.testing.assert_array_equal(idx[b, :na[b]], aidx)
                told += not np.array_equal(orc.select(rough.astype(np.float32), int(c))[0], cached)
    assert told > 100
    h.close()
