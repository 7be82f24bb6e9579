"""The row kernels around the shards: vt_combine in its two widths (16-byte loads, or one element a
thread for unaligned buffers and odd counts) against the same fp32 sums in numpy, bit for bit, and
the prefill's combine + RMSNorm at rows of one and of two chunks per thread against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synthetic
from tests.parity import assert_close, shapes_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rows,d,off,residual", [(1, 1, 64, 0, True), (4, 3, 512, 0, True), (3, 1, 1001, 0, True),
                                                   (2, 9, 64, 1, True), (16, 12, 4096, 0, True), (5, 81, 500, 0, False),
                                                   (4, 700, 4096, 4, True), (3, 47, 1001, 0, True), (2, 20, 4096, 1, True),
                                                   (2, 999, 68, 2, False)])
def test_combine_equals_the_ordered_sum(vtlib, n, rows, d, off, residual):
    """off: elements by which every buffer starts past an aligned address."""
    vt = vtlib
    rng = np.random.default_rng(n * 1000 + d + off)
    count = rows * d
    host = [rng.standard_normal(count).astype(np.float32) for _ in range(n)]
    res = rng.standard_normal(count).astype(np.float16)

    def dev(a):
        t = torch.empty(count + off, dtype=torch.float32 if a.dtype == np.float32 else torch.float16, device="cuda")[off:]
        t.copy_(torch.from_numpy(a))
        return t

    out = torch.empty(count + off + 8, dtype=torch.float16, device="cuda")
    out.fill_(7.0)
    vt.vt_combine([dev(p) for p in host], dev(res) if residual else None, out[off:off + count], rows, d)
    acc = res.astype(np.float32) if residual else np.zeros(count, np.float32)
    for p in host:
        acc = acc + p
    got = out.cpu().numpy()
    assert np.array_equal(got[off:off + count].view(np.uint16), acc.astype(np.float16).view(np.uint16))
    assert (got[:off] == 7.0).all() and (got[off + count:] == 7.0).all()


@pytest.mark.parametrize("d_model,n_dev", [(64, 1), (320, 2), (8192, 2), (8256, 5)])
def test_prefill_rows_of_every_width(vtlib, d_model, n_dev):
    """Two layers, so that the combine feeds both norms; five devices take a second batch of partials."""
    vt = vtlib
    from paper_2607_07046_gb300.stack import Stack
    wl = synthetic.small("rows", n_layers=2, d_model=d_model, n_heads=n_dev, n_kv_heads=n_dev, d_head=64, d_ffn=64 * n_dev,
                         head_ranges=tuple((i, i + 1) for i in range(n_dev)),
                         ffn_ranges=tuple((64 * i, 64 * i + 64) for i in range(n_dev)),
                         kv_len=0, decode_steps=0, prompt_len=5, model_id=144)
    X = wl.hidden(5, stream=12)
    ref = X
    for l in range(2):
        kc, vc = oracle.new_cache(wl, 8)
        _, ref, _, _ = oracle.tp_layer(wl, wl.layer_weights(l), ref, 0, kc, vc)
    with Stack(shapes_of(vt, wl, max_seq=16), wl.layer_weights, wl.head_ranges, wl.ffn_ranges, 8) as st:
        out = torch.empty((5, d_model), dtype=torch.float16, device="cuda")
        vt.vt_prefill_tokens(st.part, st.kv, torch.from_numpy(X).cuda(), 5, out)
        assert_close(out.cpu().numpy(), ref, f"prefill at d_model {d_model}")
        assert vt.vt_kv_status(st.kv) == 0


@pytest.mark.parametrize("rows", [1, 8, 9, 120, 128, 129, 256, 257, 400])
def test_prefill_gemm_tile_edges(vtlib, rows):
    """Row counts around the GEMMs' A boxes (rows rounded up to 8, up to 128) and their 128- and
    256-row tiles, an odd number of k-tiles, and down projections whose K is no multiple of 64 and
    starts at columns that are no multiple of 8 (one k-tile per copy, shifted U)."""
    vt = vtlib
    from paper_2607_07046_gb300.stack import Stack
    wl = synthetic.small("edges", n_layers=2, d_model=192, n_heads=6, n_kv_heads=3, d_head=64, d_ffn=424,
                         head_ranges=((0, 2), (2, 6)), ffn_ranges=((0, 101), (101, 424)),
                         kv_len=0, decode_steps=0, prompt_len=rows, model_id=145)
    X = wl.hidden(rows, stream=13)
    ref = X
    for l in range(2):
        kc, vc = oracle.new_cache(wl, rows)
        _, ref, _, _ = oracle.tp_layer(wl, wl.layer_weights(l), ref, 0, kc, vc)
    with Stack(shapes_of(vt, wl, max_seq=512), wl.layer_weights, wl.head_ranges, wl.ffn_ranges, rows) as st:
        out = torch.empty((rows, 192), dtype=torch.float16, device="cuda")
        vt.vt_prefill_tokens(st.part, st.kv, torch.from_numpy(X).cuda(), rows, out)
        assert_close(out.cpu().numpy(), ref, f"prefill of {rows} rows")
        assert vt.vt_kv_status(st.kv) == 0 and vt.vt_partition_status(st.part) == 0
