"""Prefill attention whose slabs go in several bands (more keys than stay in L2), the last band smaller: every sequence
bit-equal to the call on it alone (one band), two slabs against the oracle."""
import numpy as np
import pytest
import torch

import agtest as T
from oracle import ag_oracle as orc
from paper_2410_12876_b200 import inputs
from paper_2410_12876_b200.inputs import LayerShape

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("h,kv", [(47, 0), (94, 47)])
def test_bands(h, kv):
    T.ensure_built()
    shape = LayerShape(3, 2050, 64, h, 128, 1, 128, "bf16", kv_heads=kv)
    Q, K, V = inputs.qkv_gaussian(shape, 90, DEV)
    flags = inputs.bernoulli_flags((3, shape.kvh, 2050), 0.3, 91).to(DEV)
    cache, prefix, _, _ = T.gpu_compact(shape, K, V, flags)
    O = T.gpu_prefill(shape, Q, K, V, flags, cache, prefix)
    one = shape.with_(batch=1)
    for b in range(3):
        part = [t[b:b + 1].clone() for t in (Q, K, V, flags)]
        c1, p1, _, _ = T.gpu_compact(one, part[1], part[2], part[3])
        assert torch.equal(T.gpu_prefill(one, *part, c1, p1), O[b:b + 1])
    g = h // shape.kvh
    for b, i in ((0, 0), (2, shape.kvh - 1)):
        ref = orc.prefill_attention(T.f64(Q[b:b + 1, i * g:i * g + 1]), T.f64(K[b:b + 1, i:i + 1]), T.f64(V[b:b + 1, i:i + 1]),
                                    flags[b:b + 1, i:i + 1].cpu().numpy())
        T.check_close(T.f64(O[b:b + 1, i * g:i * g + 1]), ref, "bf16", f"slab {b}, {i}")
