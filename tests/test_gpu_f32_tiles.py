"""The float32 kernels at the edges of their tile choices: query tiles of 16, 32 and 64 rows, key tiles of 64,
projection tiles of 32 and 64 with a ragged last k-block, 4 or 16 tokens per CTA of the output layer, decode with one CTA
per slab and with a cluster - every call against the oracle."""
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


@pytest.mark.parametrize("B,n,hidden,h,D,gh,gD,causal", [
    (1, 1, 8, 3, 64, 1, 64, 1), (1, 65, 40, 4, 128, 2, 128, 0), (2, 161, 72, 9, 64, 2, 64, 1),     # BM = 16 and 32
    (2, 640, 64, 16, 64, 8, 64, 1), (1, 1250, 32, 16, 128, 4, 128, 0),                             # BM = 64
])
def test_layer(B, n, hidden, h, D, gh, gD, causal):
    shape = LayerShape(B, n, hidden, h, D, gh, gD, "f32", gate_causal=causal)
    seed = 800 + n
    X, W = inputs.hidden_states(shape, seed, DEV), inputs.layer_weights(shape, seed + 1, DEV)
    Q, K, V = inputs.project_qkv(shape, X, W)
    scores, _ = T.gpu_gate(shape, X, W, None)
    s_ref, _ = T.oracle_gate(shape, X, W, None)
    assert np.max(np.abs(T.f64(scores) - s_ref)) < 1e-4                # the bound every gate path is held to
    flags = inputs.bernoulli_flags((B, h, n), 0.6, seed + 2).to(DEV)
    flags[0, 0] = 0
    cache, prefix, idx, status = T.gpu_compact(shape, K, V, flags, cap=[n + 2] * (B * h))
    T.check_compaction(shape, K, V, flags, cache, prefix, idx)
    O = T.gpu_prefill(shape, Q, K, V, flags, cache, prefix)
    f = flags.cpu().numpy()
    T.check_close(T.f64(O), orc.prefill_attention(T.f64(Q), T.f64(K), T.f64(V), f), "f32", "prefill")
    ocache = orc.compact_kv(T.f64(K), T.f64(V), f)
    for step in range(2):                                              # up to 1024 (512) rows: one CTA per slab
        q, kn, vn, fn = inputs.decode_inputs(shape, seed + 5, step, DEV, keep_new=0.7)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=True)
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), ocache), "f32", f"decode {step}")
        orc.cache_append(ocache, T.f64(kn), T.f64(vn), fn.cpu().numpy())
    assert np.array_equal(cache.len.cpu().numpy(), orc.cache_lengths(ocache).reshape(-1))
    assert int(status.item()) == 0
