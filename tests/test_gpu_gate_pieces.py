"""MHA' of the gate takes keys in pairs of 64-wide tiles, K and Q in slices: segments of one pair and of many, query tiles
cut by a segment's end, a second tile that lies past the prompt, gate heads of 128 (two slices) and of 64 (three)."""
import numpy as np
import pytest
import torch

import agtest as T
from paper_2410_12876_b200 import binding as ag
from paper_2410_12876_b200 import inputs
from paper_2410_12876_b200.inputs import LayerShape

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    T.ensure_built()


@pytest.mark.parametrize("gD", [128, 64])
@pytest.mark.parametrize("B,n,gh,causal", [(1, 64, 2, 1), (1, 129, 4, 0), (2, 190, 2, 0), (1, 700, 4, 1), (3, 1025, 4, 1),
                                           (2, 1030, 2, 0)])
def test_scores(B, n, gh, gD, causal):
    shape = LayerShape(B, n, 512, 8, 128, gh, gD, "bf16", gate_causal=causal)
    X, W = inputs.hidden_states(shape, 80 + n, "cuda"), inputs.layer_weights(shape, 81 + n, "cuda")
    first, _ = T.gpu_gate(shape, X, W, None)
    again, _ = T.gpu_gate(shape, X, W, None)
    s_ref, _ = T.oracle_gate(shape, X, W, None)
    assert np.max(np.abs(T.f64(first) - s_ref)) < 1e-4                # the bound every gate path is held to
    assert torch.equal(first, again) and ag.ag_device_wait_timeouts() == 0
