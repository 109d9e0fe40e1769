"""Padding that whole tiles of the gate's kernels consist of: the projection GEMMs (single tiles, CTA pairs, reduction split
over a cluster) leave such tiles out, so their part of the workspace keeps what it held - here NaN, which must reach no
valid token.  Lengths at the edges of the 128-token tiles; gate heads of 64 (three bf16 parts) and 128; prefill attention
under a window and the local gate on the same batches."""
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


@pytest.mark.parametrize("causal", [1, 0])
@pytest.mark.parametrize("lens,n,hidden,gh,gD", [
    ((700, 1, 128, 129), 700, 256, 2, 128), ((640, 256, 127), 640, 192, 4, 64), ((300, 5), 300, 2048, 4, 128),
    ((1700, 400, 129, 1), 1700, 128, 6, 128), ((513, 100, 385), 513, 1216, 2, 64),
])
def test_gate(lens, n, hidden, gh, gD, causal):
    shape = LayerShape(len(lens), n, hidden, 8, 128, gh, gD, "bf16", gate_causal=causal)
    X, W = inputs.hidden_states(shape, 70, DEV), inputs.layer_weights(shape, 71, DEV)
    W["Wo_g"] = inputs.randn(tuple(W["Wo_g"].shape), 72, DEV, torch.bfloat16, 0.3)
    lens_dev = torch.tensor(lens, dtype=torch.int32, device=DEV)
    desc = ag.make_desc(shape, lens_dev)
    ws = ag.workspace(desc, ag.AG_CALL_GATE).fill_(255)
    scores = torch.empty(shape.batch, 8, n, dtype=torch.float32, device=DEV)
    flags = torch.full((shape.batch, 8, n), 7, dtype=torch.uint8, device=DEV)
    ag.ag_gate_forward(desc, X, W["Wq_g"], W["Wk_g"], W["Wv_g"], W["Wo_g"], None, scores, flags, ws)
    for b, L in enumerate(lens):
        ref = orc.mha_prime(T.f64(X[b, :L]), *(T.f64(W[k]) for k in ("Wq_g", "Wk_g", "Wv_g", "Wo_g")), gh, causal=bool(causal)).T
        assert np.max(np.abs(T.f64(scores[b, :, :L]) - ref)) < 1e-4
        f = flags[b].cpu().numpy()
        outside = np.abs(ref) >= T.FLAG_BAND                       # tau = 0.5: the threshold lies at 0
        assert np.array_equal(f[:, :L][outside], (ref > 0)[outside]) and not f[:, L:].any()
    assert ag.ag_device_wait_timeouts() == 0


@pytest.mark.parametrize("D,dtype", [(128, "bf16"), (64, "bf16"), (64, "f32")])
def test_window_and_local_gate(D, dtype):
    lens, n, w = (300, 1, 65, 192), 300, 6
    shape = LayerShape(4, n, 128, 8, D, 2, 64, dtype, kv_heads=4, recent_window=w)
    X, W = inputs.hidden_states(shape, 80, DEV), inputs.layer_weights(shape, 81, DEV)
    Wl = inputs.randn((128, 4), 82, DEV, shape.torch_dtype, 0.1)
    Q, K, V = inputs.project_qkv(shape, X, W)
    lens_dev = torch.tensor(lens, dtype=torch.int32, device=DEV)
    desc = ag.make_desc(shape, lens_dev)
    scores = torch.empty(4, 4, n, dtype=torch.float32, device=DEV)
    flags = torch.full((4, 4, n), 7, dtype=torch.uint8, device=DEV)
    ag.ag_gate_linear_forward(desc, X, Wl, None, scores, flags)
    cache = ag.RaggedCache.allocate(shape, [n] * 16, DEV)
    prefix = torch.empty(4, 4, n + 1, dtype=torch.int32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    ag.ag_compact_kv(desc, K, V, flags, cache, prefix, torch.empty(4, 4, n, dtype=torch.int32, device=DEV), status, None)
    O = torch.full_like(Q, float("nan"))
    ag.ag_prefill_attn(desc, Q, K, V, flags, cache, prefix, 0.0, O, ag.workspace(desc, ag.AG_CALL_PREFILL))
    f = flags.cpu().numpy()
    for b, L in enumerate(lens):
        ref = orc.linear_gate_scores(T.f64(X[b:b + 1, :L]), T.f64(Wl))[0]
        assert np.max(np.abs(T.f64(scores[b, :, :L]) - ref)) < 1e-4 and not f[b, :, L:].any()
        o = orc.prefill_attention(*(T.f64(t[b:b + 1, :, :L]) for t in (Q, K, V)), f[b:b + 1, :, :L], window=w)
        T.check_close(T.f64(O[b:b + 1, :, :L]), o, dtype, f"prefill of sequence {b}")
