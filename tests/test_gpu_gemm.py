"""K4 parity: the tcgen05 GEMM with its fused epilogues against the oracle's
fp64-accumulated nn.Linear (Supp. Sec. F projections), on sampled output
rows at the transformer's shapes (active-token counts 1229 / 4096, widths
1024 / 3072 / 4096, K 1024 / 4096) and on ragged small cases."""
import ctypes

import numpy as np
import pytest
import torch

from gpu_helpers import dev_bf16, dev_f32, rel_l2
from paper_2511_22533_gb300 import f3dc, synth

pytestmark = pytest.mark.gpu

SHAPES = [(1229, 1024, 1024), (4096, 3072, 1024), (1000, 4096, 1024), (1229, 1024, 4096), (100, 256, 128),
          (1, 64, 64), (257, 384, 128), (300, 128, 256)]
# few row tiles.  On CTA pairs (N a multiple of 256, K of 128): whole sums of K
# 1024, sums in pieces of K 4096.  Otherwise, and beyond K 8192, single CTAs split
# K and reduce the partials in split order (workspace + per-tile arrival counters):
# tiles of 128, 64 and 256 columns, 3 to 16 splits.
SPLIT_SHAPES = [(955, 1024, 1024), (300, 1024, 4096), (128, 256, 1024), (640, 3072, 1024), (413, 1024, 4096),
                (300, 384, 4096), (413, 192, 2048), (128, 64, 4096), (1100, 640, 2112), (300, 256, 2112), (5, 512, 8448)]


def _inputs(M, N, K, seed):
    g = np.random.default_rng(seed)
    A = synth.f32_to_bf16_bits(g.standard_normal((M, K)).astype(np.float32))
    Bw = synth.f32_to_bf16_bits((g.standard_normal((N, K)) / np.sqrt(K)).astype(np.float32))
    bias = synth.f32_to_bf16_bits((0.02 * g.standard_normal(N)).astype(np.float32))
    gate = g.standard_normal(N).astype(np.float32)
    rows = np.unique(np.concatenate([[0, M - 1], g.integers(0, M, 64)]))
    return A, Bw, bias, gate, rows


def _ref(orc, A, Bw, bias, rows):
    a = synth.bf16_bits_to_f32(A[rows])
    w = synth.bf16_bits_to_f32(Bw)
    return orc.linear(a, w, synth.bf16_bits_to_f32(bias)).astype(np.float64)


@pytest.mark.parametrize("M,N,K", SHAPES + SPLIT_SHAPES)
def test_gemm_bias(orc, M, N, K):
    A, Bw, bias, _, rows = _inputs(M, N, K, M + N + K)
    out = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    f3dc.gemm(dev_bf16(A), dev_bf16(Bw), dev_bf16(bias), None, out, M, N, K, f3dc.EPI_BIAS)
    torch.cuda.synchronize()
    got = out.float().cpu().numpy()[rows]
    ref = _ref(orc, A, Bw, bias, rows)
    assert rel_l2(got, ref) < 4e-3
    # bf16 output: within one rounding step of the fp64 result
    assert np.all(np.abs(got - ref) <= 2.0 ** -7 * np.abs(ref) + 1e-3)


@pytest.mark.parametrize("M,N,K", SHAPES[:4] + SPLIT_SHAPES[:2] + SPLIT_SHAPES[5:])
def test_gemm_gelu(orc, M, N, K):
    A, Bw, bias, _, rows = _inputs(M, N, K, 7 + M)
    out = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    f3dc.gemm(dev_bf16(A), dev_bf16(Bw), dev_bf16(bias), None, out, M, N, K, f3dc.EPI_GELU)
    torch.cuda.synchronize()
    got = out.float().cpu().numpy()[rows]
    pre = _ref(orc, A, Bw, bias, rows)
    ref = np.vectorize(orc.gelu)(pre.astype(np.float32)).astype(np.float64)
    assert rel_l2(got, ref) < 5e-3
    assert np.max(np.abs(got - ref)) < 2e-2 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("M,N,K", SHAPES[:4] + SHAPES[6:] + SPLIT_SHAPES)
@pytest.mark.parametrize("with_gate", [True, False])
def test_gemm_residual(orc, M, N, K, with_gate):
    A, Bw, bias, gate, rows = _inputs(M, N, K, 11 + N)
    x0 = np.random.default_rng(1).standard_normal((M, N)).astype(np.float32)
    x = dev_f32(x0)
    f3dc.gemm(dev_bf16(A), dev_bf16(Bw), dev_bf16(bias), dev_f32(gate) if with_gate else None, x, M, N, K,
              f3dc.EPI_RESID)
    torch.cuda.synchronize()
    got = x.cpu().numpy().astype(np.float64)
    y = _ref(orc, A, Bw, bias, rows)
    ref = x0[rows].astype(np.float64) + (gate[None, :] * y if with_gate else y)
    assert np.max(np.abs(got[rows] - ref)) < 1e-3 * max(1.0, np.abs(ref).max())
    # untouched rows beyond M do not exist; every row of x was updated exactly once
    others = np.setdiff1d(np.arange(M), rows)[:8]
    if len(others):
        y2 = _ref(orc, A, Bw, bias, others)
        r2 = x0[others] + (gate[None, :] * y2 if with_gate else y2)
        assert np.max(np.abs(got[others] - r2)) < 1e-3 * max(1.0, np.abs(r2).max())


def test_gemm_no_bias_and_repeat_is_deterministic(orc):
    M, N, K = 777, 1024, 1024
    A, Bw, _, _, rows = _inputs(M, N, K, 5)
    outs = []
    for _ in range(2):
        out = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
        f3dc.gemm(dev_bf16(A), dev_bf16(Bw), None, None, out, M, N, K, f3dc.EPI_BIAS)
        outs.append(out)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])
    ref = orc.linear(synth.bf16_bits_to_f32(A[rows]), synth.bf16_bits_to_f32(Bw))
    assert rel_l2(outs[0].float().cpu().numpy()[rows], ref) < 4e-3


@pytest.mark.parametrize("M,N,K", [(300, 1024, 4096), (300, 384, 4096), (300, 256, 2112)])
def test_gemm_split_k_repeat_is_deterministic(orc, M, N, K):
    # pieces are summed in order, split partials in split order by whichever
    # CTA arrives last, so repeated launches agree bit for bit
    A, Bw, bias, gate, rows = _inputs(M, N, K, 21)
    outs = []
    for _ in range(3):
        x = torch.zeros((M, N), dtype=torch.float32, device="cuda")
        f3dc.gemm(dev_bf16(A), dev_bf16(Bw), dev_bf16(bias), dev_f32(gate), x, M, N, K, f3dc.EPI_RESID)
        outs.append(x)
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.parametrize("M,N,K", [(63, 1024, 2048), (64, 1024, 2048), (257, 256, 128), (1229, 1024, 4096),
                                   (1229, 4096, 128), (1300, 4096, 256), (2400, 1024, 2048), (4096, 4096, 128),
                                   (5000, 1024, 384)])
@pytest.mark.parametrize("epi", [f3dc.EPI_BIAS, f3dc.EPI_RESID])
def test_gemm_pair_units(M, N, K, epi):
    # the CTA-pair kernel's work units, every element against 64 bits: last
    # waves of 64-, 128- and 256-column units (63 and 64 rows lie on either
    # side of the row limit of the narrowest), full waves with a rest (80, 96,
    # 256 and 80 tiles on 76 clusters), odd row tiles, and sums in several
    # accumulators (K >= 2048 on few tiles; 2400 rows: two of 256 columns)
    A, Bw, bias, gate, _ = _inputs(M, N, K, M + N + K + epi)
    Ad, Bd, bd, gd = dev_bf16(A), dev_bf16(Bw), dev_bf16(bias), dev_f32(gate)
    y = Ad.double() @ Bd.double().T + bd.double()
    if epi == f3dc.EPI_BIAS:
        out = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
        f3dc.gemm(Ad, Bd, bd, None, out, M, N, K, epi)
        # one bf16 rounding (2^-9 of the value) and the fp32 sum
        assert torch.all((out.double() - y).abs() <= 2.0 ** -8 * y.abs() + 1e-4)
    else:
        x0 = dev_f32(np.random.default_rng(M).standard_normal((M, N)).astype(np.float32))
        out = x0.clone()
        f3dc.gemm(Ad, Bd, bd, gd, out, M, N, K, epi)
        ref = x0.double() + gd.double() * y
        # the tensor core's sums are off by at most ~8e-10 K relative (truncation),
        # with pieces of at most 1024 for K > 2048; the rest rounds at 2^-24
        assert ((out.double() - ref).norm() / ref.norm()).item() < 2e-6
        assert (out.double() - ref).abs().max().item() < 1e-4
    assert f3dc.gemm_status() == 0


def _split_length(M, N, K):
    """K per partial sum where the library splits K over CTAs (its rule, restated)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bn = 256 if N % 256 == 0 else (128 if N % 128 == 0 else 64)
    tiles, kb = -(-M // 128) * (N // bn), K // 64
    sp = min(sms // tiles, kb // 4, 16) if 2 * tiles <= sms and kb >= 32 else 1
    return 64 * -(-kb // max(sp, 1))


@pytest.mark.parametrize("M,N,K", [(1, 1024, 4096), (64, 1024, 4096), (128, 1024, 2048), (77, 512, 5120),
                                   (300, 1024, 4096), (500, 2048, 2176), (384, 6400, 2048), (129, 256, 8192),
                                   (100, 12800, 4096)])
@pytest.mark.parametrize("epi", [f3dc.EPI_BIAS, f3dc.EPI_GELU, f3dc.EPI_RESID])
def test_gemm_long_sums_in_pieces(M, N, K, epi):
    # few tiles and a long K: sums in pieces no longer than split K's, in units of
    # 64, 128 and 256 columns, with fewer and more pieces than TMEM holds
    # accumulators (2 to 16; the last shape three in two), and a last piece that
    # is shorter.  Positive
    # products, so that truncation adds up: a step of 16 K loses 2^-24 of the sum
    # so far on average (up to 2^-23), a piece of L (L / 32) 2^-24 = 1.9e-9 L of
    # itself, the fp32 sum of the pieces about 1e-7.  A bias close to -sum shows
    # the same in a bf16 result.
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    A = torch.randn(M, K, generator=g, device="cuda").abs().bfloat16()
    Bw = torch.randn(N, K, generator=g, device="cuda").abs().bfloat16()
    y = A.double() @ Bw.double().T
    rel = 2.2e-9 * _split_length(M, N, K) + 1.5e-7
    if epi == f3dc.EPI_RESID:
        out = torch.zeros((M, N), dtype=torch.float32, device="cuda")
        f3dc.gemm(A, Bw, None, None, out, M, N, K, epi)
        assert ((out.double() - y).norm() / y.norm()).item() <= rel
        assert ((out.double() - y) / y).abs().max().item() <= 2 * rel
    else:
        bias = (-y.mean(0)).bfloat16()
        out = torch.full((M, N), 7.0, dtype=torch.bfloat16, device="cuda")
        f3dc.gemm(A, Bw, bias, None, out, M, N, K, epi)
        ref = y + bias.double()
        slack = 2 * rel * y.max()
        if epi == f3dc.EPI_GELU:
            # slope up to 1.13; tanh.approx is off by 2^-11, times |x| / 2 where that matters (|x| < 4)
            ref, slack = torch.nn.functional.gelu(ref, approximate="tanh"), 1.13 * slack + 1e-3
        assert torch.all((out.double() - ref).abs() <= 2.0 ** -8 * ref.abs() + slack)
    assert f3dc.gemm_status() == 0


@pytest.mark.parametrize("M,N,K,nodes", [
    (1, 256, 6144, 1), (128, 256, 6272, 2), (129, 256, 8192, 1), (129, 256, 8320, 2), (4, 256, 65536, 2),  # few tiles
    (9800, 256, 8320, 1),                                       # more tiles than half of the SMs: nothing to split
    (300, 384, 2048, 2), (300, 192, 2112, 2), (300, 256, 2112, 2),  # widths and K that the pairs do not take
    (300, 384, 1984, 1)])
def test_gemm_kernel_by_shape(M, N, K, nodes):
    # a captured call is one kernel on CTA pairs or on single CTAs without a
    # split, and split K clears its arrival counters before: very long sums of
    # few tiles go there (on a pair 4 x 256 x 65536 takes 158 us, split 42)
    cuda = ctypes.CDLL("libcuda.so.1")
    A, Bw = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda"), torch.zeros((N, K), dtype=torch.bfloat16, device="cuda")
    out = torch.zeros((M, N), dtype=torch.bfloat16, device="cuda")
    f3dc.gemm(A, Bw, None, None, out, M, N, K, f3dc.EPI_BIAS)  # the workspace is allocated on first use
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    graph, n = ctypes.c_void_p(), ctypes.c_size_t()
    assert cuda.cuStreamBeginCapture_v2(ctypes.c_void_p(s.cuda_stream), 2) == 0  # relaxed
    f3dc.gemm(A, Bw, None, None, out, M, N, K, f3dc.EPI_BIAS, stream=s.cuda_stream)
    assert cuda.cuStreamEndCapture(ctypes.c_void_p(s.cuda_stream), ctypes.byref(graph)) == 0
    assert cuda.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    assert cuda.cuGraphDestroy(graph) == 0
    assert n.value == nodes


@pytest.mark.parametrize("M", [1, 300, 2500])
def test_gemm_rows_first(M):
    # 67 MB of weights and fewer rows than columns: units run row-fastest.  1, 2
    # and 10 row pairs of 32 column tiles on 76 clusters: narrow units, full units
    # only, and full waves with a rest.
    N, K = 8192, 4096
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, K, generator=g, device="cuda").bfloat16()
    Bw = (torch.randn(N, K, generator=g, device="cuda") / K ** 0.5).bfloat16()
    out = torch.zeros((M, N), dtype=torch.float32, device="cuda")
    f3dc.gemm(A, Bw, None, None, out, M, N, K, f3dc.EPI_RESID)
    y = A.double() @ Bw.double().T
    # K / 16 steps, each truncating 2^-24 of the sum so far on average: at most
    # half of them, with a sum that grows to its final size (4.4e-6 measured, with
    # column-fastest units too)
    assert ((out.double() - y).norm() / y.norm()).item() < K / 32 * 2.0 ** -24
    assert (out.double() - y).abs().max().item() < 1e-4
    assert f3dc.gemm_status() == 0
