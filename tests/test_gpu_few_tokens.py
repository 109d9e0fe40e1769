"""The projection GEMMs on few tokens, whose reduction is split over the CTAs of a cluster: every element of the
gate's scores, of the projected Q, K, V (dense and cached) and of the output projection against the oracle, at one
token, at the edges of the 128-token tiles, with k-blocks that do not divide evenly and a ragged last one, and
with tiles of one head (128 columns) and of two."""
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


@pytest.mark.parametrize("B,n,hidden,h,hk,gh", [
    (1, 1, 1152, 8, 0, 2), (1, 127, 1096, 8, 0, 3), (1, 129, 2048, 16, 4, 4), (3, 70, 1536, 9, 3, 1),
    (2, 130, 4096, 6, 2, 4), (1, 333, 2304, 18, 0, 2),
])
def test_projections(B, n, hidden, h, hk, gh):
    shape = LayerShape(B, n, hidden, h, 128, gh, 128, "bf16", kv_heads=hk)
    seed = 300 + n + hidden
    X, W = inputs.hidden_states(shape, seed, DEV), inputs.layer_weights(shape, seed + 1, DEV)
    Wo = inputs.output_weight(shape, seed + 20, DEV)
    scores, _ = T.gpu_gate(shape, X, W, None)
    s_ref, _ = T.oracle_gate(shape, X, W, None)
    assert np.max(np.abs(T.f64(scores) - s_ref)) < 1e-4                # the bound every gate path is held to

    hk = shape.kvh
    desc = ag.make_desc(shape)
    flags = inputs.bernoulli_flags((B, hk, n), 0.5, seed + 2).to(DEV)
    cache = ag.RaggedCache.allocate(shape, [n + 1] * (B * hk), DEV)
    dense = lambda heads: torch.full((B, heads, n, 128), float("nan"), dtype=torch.bfloat16, device=DEV)
    Q, K, V = dense(h), dense(hk), dense(hk)
    prefix = torch.full((B, hk, n + 1), -1, dtype=torch.int32, device=DEV)
    idx = torch.full((B, hk, n), -1, dtype=torch.int32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    ag.ag_qkv_project_cache(desc, X, W["Wq"], W["Wk"], W["Wv"], flags, cache, prefix, idx, Q, K, V, status)
    Q_ref = orc.project_q(T.f64(X), T.f64(W["Wq"]), h)
    K_ref, V_ref = orc.project_kv(T.f64(X), T.f64(W["Wk"]), T.f64(W["Wv"]), hk)
    # one bf16 rounding of the fp64 value, plus the float32 sum's own error (hidden * 2^-24 * O(1))
    for got, ref in ((Q, Q_ref), (K, K_ref), (V, V_ref)):
        assert np.max(np.abs(T.f64(got) - ref) - 2.0 ** -8 * np.abs(ref)) < 1e-5 * (1 + hidden / 2048)
    T.check_compaction(shape, K, V, flags, cache, prefix, idx)         # cached rows: bit copies of the dense ones
    assert int(status.item()) == 0

    O = torch.randn(B, h, n, 128, generator=torch.Generator(DEV).manual_seed(seed), device=DEV).to(torch.bfloat16)
    for res in (X, None):
        Y = torch.full((B, n, hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        ag.ag_out_project(desc, O, Wo, res, Y)
        ref = orc.mha_output(T.f64(O), T.f64(Wo), None if res is None else T.f64(res))
        assert np.max(np.abs(T.f64(Y) - ref) - 2.0 ** -8 * np.abs(ref)) < 2e-5
    assert ag.ag_device_wait_timeouts() == 0
