"""Decode of few slabs.  Lengths at the edges of a warp's 16 rows, of a CTA's second tile (512 rows later, or 640 or 1024 where
ten or sixteen CTAs share a slab) and of its third, with every row that was never written holding NaN; groups of 1, 4, 8, 9 and 16
heads (one or two groups of 8 MMA columns)."""
import numpy as np
import pytest
import torch

import agtest as T
from oracle import ag_oracle as orc
from paper_2410_12876_b200 import binding as ag
from paper_2410_12876_b200 import inputs
from paper_2410_12876_b200.inputs import LayerShape

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    T.ensure_built()


@pytest.mark.parametrize("D,h,hk", [(128, 8, 8), (64, 8, 8), (128, 64, 8), (64, 128, 8), (128, 72, 8)])
def test_lengths_at_the_edges_of_blocks(D, h, hk, lens=(1, 15, 16, 17, 527, 528, 1025, 1551)):
    lens = np.array(lens)
    shape = LayerShape(1, int(lens.max()) + 49, 64, h, D, 1, 64, "bf16", kv_heads=hk)
    cache = ag.RaggedCache.allocate(shape, lens + 20, DEV)
    nan = float("nan")
    cache.k_rows.fill_(nan)
    cache.v_rows.fill_(nan)
    off = cache.row_off.cpu().numpy()
    for s, n in enumerate(lens):
        cache.k_rows[off[s]:off[s] + n] = inputs.randn((int(n), D), 41 + s, DEV, torch.bfloat16)
        cache.v_rows[off[s]:off[s] + n] = inputs.randn((int(n), D), 61 + s, DEV, torch.bfloat16)
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for step in range(2):
        held = T.gpu_cache_as_lists(cache, shape)
        q, kn, vn, fn = inputs.decode_inputs(shape, 50, step, DEV, keep_new=1.0)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=True)
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), held), "bf16", f"step {step}")
    assert np.array_equal(cache.len.cpu().numpy(), lens + 2)
    assert int(status.item()) == 0 and ag.ag_device_wait_timeouts() == 0


@pytest.mark.parametrize("D,h,hk", [(128, 7, 7), (64, 7, 7), (128, 28, 7), (64, 56, 7), (128, 63, 7), (64, 112, 7)])
def test_lengths_at_the_edges_of_sixteen_blocks(D, h, hk):
    test_lengths_at_the_edges_of_blocks(D, h, hk, lens=(16, 17, 1024, 1039, 1040, 1041, 2063))


@pytest.mark.parametrize("D,h,hk", [(128, 8, 8), (64, 8, 8), (64, 32, 8), (128, 24, 8)])
def test_lengths_at_the_edges_of_ten_blocks(D, h, hk):
    test_lengths_at_the_edges_of_blocks(D, h, hk, lens=(1, 17, 640, 655, 656, 657, 1281, 2063))


@pytest.mark.parametrize("B,h,hk,D,longest", [
    (28, 8, 8, 128, 120), (3, 64, 4, 64, 120),           # one CTA per slab, 1 and 16 heads
    (24, 32, 8, 64, 300), (20, 32, 8, 128, 700),         # one and two: what one wave holds
    (12, 16, 8, 128, 400), (60, 8, 8, 128, 2100),        # four: by the wave, by the rows per CTA
    (9, 18, 9, 64, 4200),                                # eight, by the rows per CTA
    (1, 8, 8, 128, 8300), (1, 64, 4, 64, 8300),          # sixteen, few slabs of very many rows
    (2, 40, 8, 128, 8300), (1, 128, 8, 64, 8300),        # the same with more than 64 query heads: the split form
    (5, 18, 1, 128, 300), (3, 34, 1, 64, 300),           # more than 16 heads per slab, more than 64 in all: the split form
])
def test_ctas_per_slab(B, h, hk, D, longest):
    """Each choice of CTAs per slab, over empty, one-row and full slabs among ragged ones, with the append."""
    rng = np.random.default_rng(longest)
    lens = rng.integers(0, longest // 4, size=B * hk)
    lens[:3] = 0, 1, longest
    shape = LayerShape(B, longest + 8, 64, h, D, 1, 64, "bf16", kv_heads=hk)
    cap = lens + 2
    cap[1] = 1                                           # full: the append is refused
    cache = ag.RaggedCache.allocate(shape, cap, DEV)
    cache.k_rows.copy_(inputs.randn(tuple(cache.k_rows.shape), 41, DEV, torch.bfloat16))
    cache.v_rows.copy_(inputs.randn(tuple(cache.v_rows.shape), 42, DEV, torch.bfloat16))
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for step in range(2):
        held = T.gpu_cache_as_lists(cache, shape)
        q, kn, vn, fn = inputs.decode_inputs(shape, 50, step, DEV, keep_new=1.0)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=True)
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), held), "bf16", f"step {step}")
    assert np.array_equal(cache.len.cpu().numpy(), np.minimum(lens + 2, cap))
    rows, off = T.f64(cache.k_rows), cache.row_off.cpu().numpy()
    for s in range(0, B * hk, 5):
        if s != 1:
            assert np.array_equal(rows[off[s] + lens[s] + 1], T.f64(kn).reshape(-1, D)[s])
    assert int(status.item()) == ag.AG_DEV_OVERFLOW and ag.ag_device_wait_timeouts() == 0


@pytest.mark.parametrize("B,h,hk,D,longest", [
    (1, 4, 4, 128, 2060), (2, 20, 4, 64, 2060),          # up to seven slabs, from 2048 rows; eight of five heads: eight CTAs
    (4, 4, 4, 128, 4100), (2, 64, 8, 64, 4100),          # sixteen slabs, too few rows for it
    (1, 64, 4, 128, 520), (1, 48, 3, 64, 1040),          # 16 heads per slab, from 512; a second tile for one rank
])
def test_sixteen_ctas_per_slab(B, h, hk, D, longest):
    test_ctas_per_slab(B, h, hk, D, longest)


@pytest.mark.parametrize("B,h,hk,D,longest", [
    (4, 4, 4, 128, 8300), (4, 16, 4, 64, 8300), (1, 28, 7, 128, 2060),    # sixteen CTAs: up to 16 slabs beyond 8192 rows, seven
    (1, 8, 8, 128, 2060), (2, 16, 4, 128, 2060), (1, 27, 9, 64, 4100),    # ten: eight and nine slabs of 1, 4 and 3 heads
    (20, 16, 1, 128, 1100), (9, 18, 2, 64, 1100),        # 16 and 9 heads, eight CTAs: two heads for a rank
    (20, 16, 1, 128, 400), (17, 12, 1, 64, 500),         # four CTAs, four and three heads for a rank
    (80, 16, 1, 128, 700), (120, 10, 1, 64, 700),        # two CTAs, eight and five
])
def test_heads_shared_among_ranks(B, h, hk, D, longest):
    test_ctas_per_slab(B, h, hk, D, longest)


@pytest.mark.parametrize("D,extra", [(64, 2), (64, 400), (128, 2), (128, 400)])
def test_float32_rounds(D, extra, batch=1, threads=512):
    """The float32 form's last round of rows in a quarter, a half or all of its registers: 512 threads take 32 rows of 64 or 16
    of 128 at a time, eight times a round; one CTA per slab, and eight where the capacity asks for them."""
    step = threads * 4 // D
    lens = np.array([0, 1, 2 * step - 1, 2 * step, 2 * step + 1, 4 * step, 4 * step + 1, 8 * step, 8 * step + 1, 10 * step + 1])
    shape = LayerShape(batch, 16 * step + 400, 64, lens.size, D, 1, 64, "f32")
    lens = np.tile(lens, batch)
    cache = ag.RaggedCache.allocate(shape, lens + extra, DEV)
    cache.k_rows.copy_(inputs.randn(tuple(cache.k_rows.shape), 41, DEV, torch.float32))
    cache.v_rows.copy_(inputs.randn(tuple(cache.v_rows.shape), 42, DEV, torch.float32))
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for t in range(2):
        held = T.gpu_cache_as_lists(cache, shape)
        q, kn, vn, fn = inputs.decode_inputs(shape, 50, t, DEV, keep_new=1.0)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=True)
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), held), "f32", f"step {t}")
    assert np.array_equal(cache.len.cpu().numpy(), lens + 2) and int(status.item()) == 0


@pytest.mark.parametrize("D,extra", [(64, 2), (64, 400), (128, 2), (128, 400)])
def test_float32_rounds_of_chunks(D, extra):
    """The split form's chunks of 128 rows: 256 threads, whole rounds but for a slab's last chunk."""
    test_float32_rounds(D, extra, batch=7, threads=256)


@pytest.mark.parametrize("B,h,hk,D,dtype,longest,untouched", [
    (1, 8, 8, 128, "bf16", 8300, True), (2, 32, 8, 128, "bf16", 8300, True), (1, 64, 4, 64, "bf16", 8300, True),
    (2, 32, 1, 64, "bf16", 300, True), (16, 4, 4, 64, "f32", 300, True),
    (2, 40, 8, 128, "bf16", 8300, False), (17, 4, 4, 64, "f32", 300, False),
])
def test_up_to_64_slabs_leave_the_scratch_alone(B, h, hk, D, dtype, longest, untouched):
    """Callers of ag_decode_attn_noalloc may count on it: calls of so few slabs share no array."""
    shape = LayerShape(B, longest + 8, 64, h, D, 1, 64, dtype, kv_heads=hk)
    lens = np.random.default_rng(1).integers(1, 40, size=B * hk)
    lens[0] = longest
    cache = ag.RaggedCache.allocate(shape, lens, DEV)
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    desc = ag.make_desc(shape)
    ws = ag.workspace(desc, ag.AG_CALL_DECODE)
    ws.fill_(77)
    q, kn, vn, _ = inputs.decode_inputs(shape, 50, 0, DEV)
    ag.ag_decode_attn(desc, q, kn, vn, cache, 0.0, torch.empty_like(q), ws)
    assert bool((ws == 77).all()) == untouched
