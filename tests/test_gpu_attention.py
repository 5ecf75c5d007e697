"""K5 / K6 parity: the tcgen05 flash attention against the oracle's fp64
softmax attention (Supp. Sec. F self- and cross-attention) on sampled query
rows: active-token sequences (ragged, 1229, 4096), the 1374-token condition,
head dims 32 and 64, a single key and odd tails.  f3dc_attention runs the
one-tile kernel (k_attn_one.cu) when every (query tile, head) item gets an
SM of its own and the pair kernel (k_attn.cu) otherwise: on a 152-SM GB300
the cases with more than 152 items (1229 x 16 heads, 4096 x 16, 2600 x 8,
whose odd tile count leaves the last pair half empty) take the pair kernel,
the others the one-tile kernel."""
import numpy as np
import pytest
import torch

from gpu_helpers import dev_bf16, rel_l2
from paper_2511_22533_gb300 import f3dc, synth

pytestmark = pytest.mark.gpu

CASES = [(300, 300, 4, 32), (1229, 1229, 16, 64), (4096, 4096, 16, 64), (1229, 1374, 16, 64), (5, 1, 2, 64),
         (130, 129, 2, 32), (128, 256, 1, 64), (700, 77, 4, 32), (256, 256, 1, 64), (128, 384, 1, 64),
         (1, 200, 1, 32), (128, 129, 1, 64), (2600, 700, 8, 32), (955, 1374, 16, 64)]


@pytest.mark.parametrize("nq,nk,H,dh", CASES)
def test_attention(orc, nq, nk, H, dh):
    g = np.random.default_rng(nq * 7 + nk)
    W = H * dh
    q = synth.f32_to_bf16_bits(g.standard_normal((nq, W)).astype(np.float32))
    kv = synth.f32_to_bf16_bits(g.standard_normal((nk, 2 * W)).astype(np.float32))
    out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
    kvd = dev_bf16(kv)
    f3dc.attention(dev_bf16(q), W, kvd, kvd[:, W:], 2 * W, out, nq, nk, H, dh)
    torch.cuda.synchronize()
    rows = np.unique(np.concatenate([[0, nq - 1], g.integers(0, nq, 48)]))
    kf = synth.bf16_bits_to_f32(kv)
    ref = orc.attention(synth.bf16_bits_to_f32(q[rows]), kf[:, :W], kf[:, W:], H).astype(np.float64)
    got = out.float().cpu().numpy()[rows]
    assert np.isfinite(got).all()
    assert rel_l2(got, ref) < 1e-2
    assert np.max(np.abs(got - ref)) < 2e-2


def test_attention_rows_beyond_nq_untouched():
    nq, nk, H, dh = 100, 300, 2, 64
    g = np.random.default_rng(0)
    q = dev_bf16(synth.f32_to_bf16_bits(g.standard_normal((128, H * dh)).astype(np.float32)))
    kv = dev_bf16(synth.f32_to_bf16_bits(g.standard_normal((nk, H * dh)).astype(np.float32)))
    out = torch.full((128, H * dh), 3.0, dtype=torch.bfloat16, device="cuda")
    f3dc.attention(q, H * dh, kv, kv, H * dh, out, nq, nk, H, dh)
    torch.cuda.synchronize()
    assert torch.all(out[nq:] == 3.0)
    assert torch.isfinite(out[:nq].float()).all()


def _rescale_case(nq, nk, H, dh, seed):
    """Queries and keys along one direction u per head (entries +-1) so that
    each row's scores are set per key tile.  The first two tiles hold keys of
    strength 1; tile j >= 2 holds keys one strength step above tile j - 2 --
    all its keys, except in the last two tiles, which hold a single such key
    each (at position 37 j within the tile).  A step is worth 8.4-9.3 log2
    units of scaled score for query strengths in [0.9, 1], just past the
    kernel's 2^8 margin, so running maxima are raised (and O and l rescaled
    in place) at every even tile from 2 on, while the full tiles before the
    last ones keep a visible share of the softmax weight; the last tile is
    ragged.  With 900 keys the single strong key of tile 6 sits in the tile's
    second half (position 94)."""
    g = np.random.default_rng(seed)
    W = H * dh
    u = np.where(g.random((H, dh)) < 0.5, -1.0, 1.0)
    c = g.uniform(0.9, 1.0, nq)                        # per-row query strength
    q = np.einsum("r,hd->rhd", c, u).reshape(nq, W) + 0.02 * g.standard_normal((nq, W))
    step = 8.85 / (0.95 * np.sqrt(dh) * np.log2(np.e))
    a = np.full(nk, 1.0)                               # per-key strength
    nkt = (nk + 127) // 128
    for j in range(2, nkt):
        lo, hi = 128 * j, min(nk, 128 * j + 128)
        if j >= nkt - 2:
            a[lo + (j * 37) % (hi - lo)] = 1.0 + step * (j // 2)
        else:
            a[lo:hi] = 1.0 + step * (j // 2)
    k = np.einsum("j,hd->jhd", a, u).reshape(nk, W) + 0.02 * g.standard_normal((nk, W))
    v = g.standard_normal((nk, W))
    return [synth.f32_to_bf16_bits(x.astype(np.float32)) for x in (q, k, v)]


@pytest.mark.parametrize("nq,nk,H,dh", [(256, 700, 2, 64), (200, 900, 2, 32), (256, 900, 2, 64), (130, 641, 1, 64),
                                        (1280, 900, 16, 64)])
def test_attention_reference_max_raised_in_late_tiles(orc, nq, nk, H, dh):
    # the one-tile kernel keeps a reference max per row and parity of key tiles
    # and raises it (rescaling O and l in TMEM) only when a key tile's max
    # exceeds it by more than 2^8; keys drawn N(0, 1) never get there, so these
    # cases place the strongest keys in late tiles and check the outcome
    # against the oracle's fp64 softmax attention.  The
    # 1280-query, 16-head case (160 items) takes the pair kernel, whose first
    # pass keeps the first tile's maximum and raises it once, at the ragged last
    # tile (27 above: no second pass).
    W = H * dh
    q, k, v = _rescale_case(nq, nk, H, dh, nq + nk)
    qf, kf, vf = (synth.bf16_bits_to_f32(x).astype(np.float64) for x in (q, k, v))
    # the branch is taken: per row and head, every tile from the third on
    # beats the tile two before it by more than 8 (log2 units of scaled
    # score), with a margin for fp32 scores; and the raised-over tiles still
    # carry a visible share of the softmax weight
    sc = np.einsum("rhd,jhd->rhj", qf.reshape(nq, H, dh), kf.reshape(nk, H, dh)) * np.log2(np.e) / np.sqrt(dh)
    nkt = (nk + 127) // 128
    tmax = np.stack([sc[:, :, 128 * j:min(nk, 128 * j + 128)].max(axis=2) for j in range(nkt)], axis=2)
    assert nkt >= 4 and np.all(tmax[:, :, 2:] - tmax[:, :, :-2] > 8.2)
    p = np.exp2(sc - sc.max(axis=2, keepdims=True))
    p /= p.sum(axis=2, keepdims=True)
    top = np.argmax(sc, axis=2) // 128  # the tile that holds each row's strongest key
    rest = 1.0 - np.take_along_axis(np.stack([p[:, :, 128 * j:128 * j + 128].sum(axis=2) for j in range(nkt)], 2),
                                    top[:, :, None], axis=2)[:, :, 0]
    assert rest.min() > 0.05
    out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
    kd, vd = dev_bf16(k), dev_bf16(v)
    f3dc.attention(dev_bf16(q), W, kd, vd, W, out, nq, nk, H, dh)
    torch.cuda.synchronize()
    ref = orc.attention(qf.astype(np.float32), kf.astype(np.float32), vf.astype(np.float32), H).astype(np.float64)
    got = out.float().cpu().numpy()
    assert np.isfinite(got).all()
    assert rel_l2(got, ref) < 1e-2
    assert np.max(np.abs(got - ref)) < 2e-2


@pytest.mark.parametrize("nq,nk,H,dh", [(1280, 900, 16, 64), (2600, 700, 8, 32)])
@pytest.mark.parametrize("kind", ["scores", "values", "nan"])
def test_attention_first_pass_reference_is_not_enough(orc, nq, nk, H, dh, kind):
    # the pair kernel takes its reference from an item's first key tile and
    # repeats a CTA's items with running maxima when that does not carry:
    # scores 2^100 and 2^170 above the first tile's, values so large that
    # 2^40 P overflows the fp32 accumulator, and a NaN query row (which must
    # stay NaN and leave the other rows alone)
    g = np.random.default_rng(nq + nk)
    W = H * dh
    u = np.where(g.random((H, dh)) < 0.5, -1.0, 1.0)
    c = g.uniform(0.95, 1.0, nq)
    q = np.einsum("r,hd->rhd", c, u).reshape(nq, W)
    unit = 1.0 / (np.sqrt(dh) * np.log2(np.e))         # key strength worth one log2 unit of scaled score
    up = {"scores": (100.0, 170.0), "values": (40.0, 40.0), "nan": (0.0, 0.0)}[kind]
    a = np.zeros(nk)
    a[256:384] = up[0] * unit
    a[nk - 60:] = up[1] * unit
    k = np.einsum("j,hd->jhd", a, u).reshape(nk, W) + 0.02 * g.standard_normal((nk, W))
    v = g.standard_normal((nk, W)) * (1e30 if kind == "values" else 1.0)
    if kind == "nan":
        q[7, 3] = np.nan
    qb, kb, vb = (synth.f32_to_bf16_bits(x.astype(np.float32)) for x in (q, k, v))
    out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
    f3dc.attention(dev_bf16(qb), W, dev_bf16(kb), dev_bf16(vb), W, out, nq, nk, H, dh)
    assert f3dc.gemm_status() == 0
    rows = np.unique(np.concatenate([[0, 7, 127, 128, nq - 1], g.integers(0, nq, 24)]))
    qf, kf, vf = (synth.bf16_bits_to_f32(x) for x in (qb, kb, vb))
    got = out.float().cpu().numpy()[rows].astype(np.float64)
    if kind == "nan":
        assert np.isnan(got[rows == 7, :dh]).all() and np.isfinite(got[rows == 7, dh:]).all()
        got, rows = got[rows != 7], rows[rows != 7]
    ref = orc.attention(qf[rows], kf, vf, H).astype(np.float64)
    scale = 1e30 if kind == "values" else 1.0
    assert np.isfinite(got).all()
    assert rel_l2(got / scale, ref / scale) < 1e-2
    assert np.max(np.abs(got - ref)) / scale < 2e-2


@pytest.mark.parametrize("nq,nk,H,dh", [(1280, 257, 16, 64), (2600, 257, 8, 32), (1280, 385, 16, 64)])
@pytest.mark.parametrize("middle,last", [(119.0, 127.0), (117.0, 125.0), (133.0, 140.0), (60.0, 187.0)])
def test_attention_ragged_last_tile_far_above_the_first(orc, nq, nk, H, dh, middle, last):
    # scaled scores (log2 units) of 0 in the first key tile, `middle` in the
    # plain tiles after it and `last` on the one key of the ragged last tile:
    # raising the reference by more than 2^126 there flushes the factor that
    # rescales l and O to 0, while the plain tiles, 2^8 below the last key and
    # 128 keys strong, hold a third of the row's weight
    g = np.random.default_rng(nq + nk)
    W = H * dh
    u = np.where(g.random((H, dh)) < 0.5, -1.0, 1.0)
    q = np.broadcast_to(u.reshape(1, W), (nq, W))
    unit = 1.0 / (np.sqrt(dh) * np.log2(np.e))
    a = np.zeros(nk)
    a[128:nk - 1] = middle * unit
    a[nk - 1] = last * unit
    k = np.einsum("j,hd->jhd", a, u).reshape(nk, W)
    v = np.where(np.arange(nk)[:, None] == nk - 1, -0.5, 0.5) + 0.05 * g.standard_normal((nk, W))
    qb, kb, vb = (synth.f32_to_bf16_bits(x.astype(np.float32)) for x in (q, k, v))
    out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
    f3dc.attention(dev_bf16(qb), W, dev_bf16(kb), dev_bf16(vb), W, out, nq, nk, H, dh)
    assert f3dc.gemm_status() == 0
    qf, kf, vf = (synth.bf16_bits_to_f32(x) for x in (qb, kb, vb))
    ref = orc.attention(qf[:1], kf, vf, H).astype(np.float64)  # the rows are equal
    got = out.float().cpu().numpy().astype(np.float64)
    assert np.isfinite(got).all()
    assert np.max(np.abs(got - ref)) < 1e-2  # a bf16 rounding of values up to 0.7 and of P


def _bits(t):
    return t.view(torch.int16).cpu().numpy()


@pytest.mark.parametrize("nq,nk,H,dh", [(2700, 900, 16, 64), (4096, 700, 16, 64), (4096, 700, 16, 32),
                                        (20000, 640, 64, 32)])
@pytest.mark.parametrize("which", ["all", "one"])
def test_attention_second_pass_over_several_items(orc, nq, nk, H, dh, which):
    # 176 and 256 (pair, head) items on 152 SMs: CTAs with one item and CTAs
    # with two, whose second pass starts at other K/V stages, Q buffers and
    # barrier phases than the first did; and 5056 items: 33 or 34 a CTA, more
    # than a window of 32.  "all": every row's scores rise by 2^90 after the
    # first key tile (and no ragged last tile raises the reference), so every
    # item runs twice.  "one": a single row of one head does, in its CTA's last
    # item, and only that item does.  Written over the queries the result is
    # the same.
    g = np.random.default_rng(nq + nk + dh)
    W = H * dh
    u = np.where(g.random((H, dh)) < 0.5, -1.0, 1.0)
    unit = 1.0 / (np.sqrt(dh) * np.log2(np.e))
    a = np.zeros(nk)
    a[200:300] = 90.0 * unit
    a[400:450] = 101.0 * unit
    k = (np.einsum("j,hd->jhd", a, u) + 0.02 * g.standard_normal((nk, H, dh))).reshape(nk, W)
    v = g.standard_normal((nk, W))
    # strength 0.01: scores up to 0.9
    c = np.full((nq, H), 1.0 if which == "all" else 0.01)
    items = (nq + 255) // 256 * H
    item = (items - 1) // 152 * 152 + 3
    row, head = 256 * (item // H) + 5, item % H
    c[row, head] = 1.0
    q = np.einsum("rh,hd->rhd", c, u).reshape(nq, W)
    qb, kb, vb = (synth.f32_to_bf16_bits(x.astype(np.float32)) for x in (q, k, v))
    out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
    f3dc.attention(dev_bf16(qb), W, dev_bf16(kb), dev_bf16(vb), W, out, nq, nk, H, dh)
    assert f3dc.gemm_status() == 0
    qd = dev_bf16(qb)
    f3dc.attention(qd, W, dev_bf16(kb), dev_bf16(vb), W, qd, nq, nk, H, dh)
    assert f3dc.gemm_status() == 0 and torch.equal(qd, out)
    rows = np.unique(np.concatenate([[0, 127, 128, 255, 256, row - 1, row, row + 1, nq - 1], g.integers(0, nq, 40)]))
    qf, kf, vf = (synth.bf16_bits_to_f32(x) for x in (qb, kb, vb))
    ref = orc.attention(qf[rows], kf, vf, H).astype(np.float64)
    got = out.float().cpu().numpy()
    assert np.isfinite(got).all()
    assert rel_l2(got[rows], ref) < 1e-2
    assert np.max(np.abs(got[rows] - ref)) < 2e-2


@pytest.mark.parametrize("nq,nk,H,dh", [(1280, 900, 16, 64), (4096, 700, 16, 32)])
@pytest.mark.parametrize("bad", ["nan", "far"])
def test_attention_rows_do_not_depend_on_others_second_pass(nq, nk, H, dh, bad):
    # a row whose scores are NaN, or 2^90 above those of the first key tile,
    # wants its item done again; every other row keeps its bits (but for the 32
    # rows of its warp and head, which raise their reference together), those of
    # its item, of its CTA's other items and of the other heads.  Key strengths
    # rise by 2^10 and 2^20, so that running maxima would take another
    # reference than the first key tile's.
    g = np.random.default_rng(nq + nk + dh)
    W = H * dh
    u = np.where(g.random((H, dh)) < 0.5, -1.0, 1.0)
    unit = 1.0 / (np.sqrt(dh) * np.log2(np.e))
    a = np.zeros(nk)
    a[150:256] = 10.3 * unit
    a[256:400] = 20.7 * unit
    k = (np.einsum("j,hd->jhd", a, u) + 0.1 * g.standard_normal((nk, H, dh))).reshape(nk, W)
    v = dev_bf16(synth.f32_to_bf16_bits(g.standard_normal((nk, W)).astype(np.float32)))
    q = (np.broadcast_to(u, (nq, H, dh)) + 0.1 * g.standard_normal((nq, H, dh))).astype(np.float32)
    row, head = 300, 3
    kd = dev_bf16(synth.f32_to_bf16_bits(k.astype(np.float32)))

    def run(q):
        out = torch.zeros((nq, W), dtype=torch.bfloat16, device="cuda")
        f3dc.attention(dev_bf16(synth.f32_to_bf16_bits(q.reshape(nq, W))), W, kd, v, W, out, nq, nk, H, dh)
        assert f3dc.gemm_status() == 0
        return _bits(out).reshape(nq, H, dh)

    clean = run(q)
    q2 = q.copy()
    q2[row, head] = np.nan if bad == "nan" else 5.0 * u[head]
    got = run(q2)
    changed = np.any(got != clean, axis=2)
    changed[row // 32 * 32:row // 32 * 32 + 32, head] = False
    assert not changed.any(), np.argwhere(changed)[:5]
    if bad == "nan":
        assert np.isnan(synth.bf16_bits_to_f32(got[row, head].view(np.uint16))).all()
