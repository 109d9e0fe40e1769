"""bf16 layers of 64-wide heads on the tensor cores (gate, prefill attention, decode), and grouped-query
decode where one cluster reads a slab for all its query heads: sizes at the edges of the tiles (128
queries, 64 keys; decode: 64 rows per tile, 8 CTAs per cluster) against the oracle."""
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


@pytest.mark.parametrize("B,n,h,hk,gh,gD,causal,window", [
    (1, 1, 4, 0, 2, 64, 1, 0), (1, 64, 4, 0, 2, 64, 0, 0), (2, 129, 4, 0, 2, 64, 1, 0), (1, 257, 6, 0, 4, 64, 0, 0),
    (2, 333, 8, 2, 2, 64, 1, 5), (1, 640, 4, 2, 2, 128, 1, 0), (3, 100, 4, 4, 3, 64, 1, 0),
])
def test_layer_of_64_wide_heads(B, n, h, hk, gh, gD, causal, window):
    shape = LayerShape(B, n, 192, h, 64, gh, gD, "bf16", gate_causal=causal, kv_heads=hk, recent_window=window)
    seed = 700 + n
    X, W = inputs.hidden_states(shape, seed, DEV), inputs.layer_weights(shape, seed + 1, DEV)
    W["Wo_g"] = inputs.randn(tuple(W["Wo_g"].shape), seed + 2, DEV, shape.torch_dtype, 0.5)
    Q, K, V = inputs.project_qkv(shape, X, W)
    s0, _ = T.oracle_gate(shape, X, W, None)
    gamma = inputs.calibrate_gamma(torch.from_numpy(s0), np.full(shape.kvh, 0.6), float(np.float32(shape.tau))).to(DEV)
    scores, flags = T.gpu_gate(shape, X, W, gamma)
    s_ref, f_ref = T.oracle_gate(shape, X, W, gamma)
    assert np.max(np.abs(T.f64(scores) - s_ref)) < 1e-4                # the bound every gate path is held to
    T.check_flags(shape, flags, s_ref, f_ref, gamma)

    f = np.ascontiguousarray(f_ref).copy()
    f[0, 0] = 0                                                        # a head that keeps nothing
    fl = torch.from_numpy(f).to(DEV)
    steps = 3
    cap = (f.reshape(B * shape.kvh, -1).sum(axis=1) + steps).tolist()  # tight slabs
    cache, prefix, idx, status = T.gpu_compact(shape, K, V, fl, cap=cap)
    T.check_compaction(shape, K, V, fl, cache, prefix, idx)
    O = T.gpu_prefill(shape, Q, K, V, fl, cache, prefix)
    T.check_close(T.f64(O), orc.prefill_attention(T.f64(Q), T.f64(K), T.f64(V), f, window=max(window, 1)), "bf16", "prefill")
    ocache = orc.compact_kv(T.f64(K), T.f64(V), f, window=max(window, 1))
    for step in range(steps):
        q, kn, vn, fn = inputs.decode_inputs(shape, seed + 5, step, DEV, keep_new=0.7)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=bool(step % 2))
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), ocache), "bf16", f"decode {step}")
        orc.cache_append(ocache, T.f64(kn), T.f64(vn), fn.cpu().numpy(), window=max(window, 1))
    assert np.array_equal(cache.len.cpu().numpy(), orc.cache_lengths(ocache).reshape(-1))
    assert int(status.item()) == 0 and ag.ag_device_wait_timeouts() == 0


@pytest.mark.parametrize("D,h,hk,B", [(128, 32, 8, 1), (64, 8, 4, 2), (128, 16, 1, 3), (128, 18, 1, 2), (64, 34, 2, 1),
                                      (128, 24, 8, 9), (64, 16, 8, 12)])
def test_decode_step_of_shared_slabs(D, h, hk, B):
    """ag_decode_step with a group of query heads per slab: lengths at the edges of the 64-row tiles and of
    the 512 rows the eight CTAs of a cluster take at once, a full slab, and the append carried by the
    kernel that reads the slab (groups of up to 16 heads; one launch more beyond)."""
    lens = np.array([0, 1, 63, 64, 65, 511, 512, 513, 577, 1100] * 10)[:B * hk]
    shape = LayerShape(B, 1200, 64, h, D, 1, 64, "bf16", kv_heads=hk)
    cap = lens + 2
    cap[-1] = lens[-1]                                                 # full: the append is refused
    cache = ag.RaggedCache.allocate(shape, cap, DEV)
    cache.k_rows.copy_(inputs.randn(tuple(cache.k_rows.shape), 41, DEV, torch.bfloat16))
    cache.v_rows.copy_(inputs.randn(tuple(cache.v_rows.shape), 42, DEV, torch.bfloat16))
    cache.len.copy_(torch.from_numpy(lens.astype(np.int32)))
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    for step in range(2):
        held = T.gpu_cache_as_lists(cache, shape)
        before = cache.len.cpu().numpy()
        q, kn, vn, fn = inputs.decode_inputs(shape, 50, step, DEV, keep_new=1.0)
        o = T.gpu_decode_step(shape, q, kn, vn, fn, cache, status, fused=True)
        T.check_close(T.f64(o), orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), held), "bf16", f"step {step}")
        after = cache.len.cpu().numpy()
        assert np.array_equal(after, np.minimum(before + 1, cap))
        rows, off = T.f64(cache.k_rows), cache.row_off.cpu().numpy()
        for s in np.nonzero(after > before)[0]:
            assert np.array_equal(rows[off[s] + before[s]], T.f64(kn).reshape(-1, D)[s])
    assert int(status.item()) == ag.AG_DEV_OVERFLOW and ag.ag_device_wait_timeouts() == 0


@pytest.mark.parametrize("n,causal,gh", [(70, 1, 28), (70, 0, 26), (2400, 1, 28)])
def test_gate_of_many_64_wide_heads(n, causal, gh):
    """The widest gates of 64-wide heads: 26 are the last the tensor-core form takes, 28 go to the CUDA cores (4 tokens per
    CTA of its output layer, and 16 beyond 2,368 tokens)."""
    shape = LayerShape(1, n, 128, 32, 64, gh, 64, "bf16", gate_causal=causal)
    X, W = inputs.hidden_states(shape, 900, DEV), inputs.layer_weights(shape, 901, DEV)
    W["Wo_g"] = inputs.randn(tuple(W["Wo_g"].shape), 902, DEV, shape.torch_dtype, 0.1)
    scores, flags = T.gpu_gate(shape, X, W, None)
    s_ref, f_ref = T.oracle_gate(shape, X, W, None)
    assert np.max(np.abs(T.f64(scores) - s_ref)) < 1e-4                # the bound every gate path is held to
    T.check_flags(shape, flags, s_ref, f_ref, None)
    assert ag.ag_device_wait_timeouts() == 0
