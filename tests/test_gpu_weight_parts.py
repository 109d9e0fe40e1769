"""The weights of a softmax enter the weighted sum in two bf16 parts: an output differs from float64 by its own
rounding and by what is left of the weights, on caches of few rows, where a rounded weight would show."""
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


def check_rounding(got, want, v_max, what=""):
    """`got` is the bf16 rounding of a value within 2^-14 max |v| of `want`.  That holds what the sums lose: a weight in
    two bf16 parts is off by 2^-17 of itself, its score (of a few units, summed in float32 over 64 or 128 terms, scaled,
    and put through exp2) by up to 2^-17, and the sum of the weights likewise; the weights add up to one.  One bf16 part
    alone is off by up to 2^-8 of every weight."""
    lo, hi = (torch.from_numpy(want + d).to(torch.bfloat16) for d in (-2.0 ** -14 * v_max, 2.0 ** -14 * v_max))
    out = int(((got.cpu() < lo) | (got.cpu() > hi)).sum()) + int((~torch.isfinite(got)).sum())
    assert out == 0, f"{what}: {out} of {got.numel()} values are another rounding"


@pytest.mark.parametrize("B,h,hk,D,longest", [
    (1, 8, 8, 128, 60), (3, 32, 32, 128, 40), (1, 8, 8, 128, 700), (2, 4, 4, 64, 60), (12, 8, 8, 64, 40),  # one head per slab
    (2, 6, 2, 128, 60), (5, 16, 4, 64, 60), (1, 8, 2, 128, 900),                        # up to 4: repeated columns
    (2, 10, 2, 128, 60), (3, 16, 2, 64, 60), (2, 18, 2, 128, 60), (2, 32, 2, 64, 60),   # 5, 8, 9, 16
    (2, 40, 8, 128, 8300), (2, 72, 8, 64, 8300), (2, 128, 8, 64, 8300),                 # the split form
])
def test_decode(B, h, hk, D, longest):
    rng = np.random.default_rng(h + D)
    lens = rng.integers(1, 24, size=B * hk)
    lens[0] = longest
    shape = LayerShape(B, longest + 8, 64, h, D, 1, 64, "bf16", kv_heads=hk)
    cache = ag.RaggedCache.allocate(shape, lens, DEV)
    cache.k_rows.copy_(inputs.randn(tuple(cache.k_rows.shape), 41, DEV, torch.bfloat16))
    cache.v_rows.copy_(inputs.randn(tuple(cache.v_rows.shape), 42, DEV, torch.bfloat16))
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    q, kn, vn, _ = inputs.decode_inputs(shape, 50, 0, DEV)
    desc = ag.make_desc(shape)
    o = torch.full_like(q, float("nan"))
    ag.ag_decode_attn(desc, q, kn, vn, cache, 0.0, o, ag.workspace(desc, ag.AG_CALL_DECODE))
    want = orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), T.gpu_cache_as_lists(cache, shape))
    check_rounding(o, want, max(np.abs(T.f64(cache.v_rows)).max(), np.abs(T.f64(vn)).max()))


@pytest.mark.parametrize("B,n,h,hk,D,window,keep", [
    (1, 1, 4, 4, 64, 0, 0.5), (2, 40, 4, 4, 64, 0, 0.5), (1, 129, 4, 2, 64, 0, 0.3), (1, 300, 2, 2, 64, 0, 0.9),
    (1, 64, 4, 4, 64, 10, 0.2), (2, 145, 4, 2, 64, 17, 0.1),
    (1, 40, 4, 4, 128, 5, 0.0), (1, 257, 4, 2, 128, 17, 0.0),     # nothing but the window: its dense tiles
])
def test_prefill(B, n, h, hk, D, window, keep):
    shape = LayerShape(B, n, 64, h, D, 1, 64, "bf16", kv_heads=hk, recent_window=window)
    Q, K, V = inputs.qkv_gaussian(shape, 70 + n, DEV)
    flags = torch.from_numpy((np.random.default_rng(n).random((B, hk, n)) < keep).astype(np.uint8)).to(DEV)
    cache, prefix, _, _ = T.gpu_compact(shape, K, V, flags)
    O = T.gpu_prefill(shape, Q, K, V, flags, cache, prefix)
    want = orc.prefill_attention(T.f64(Q), T.f64(K), T.f64(V), flags.cpu().numpy(), window=max(window, 1))
    check_rounding(O, want, np.abs(T.f64(V)).max())
