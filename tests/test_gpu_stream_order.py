"""A decode call takes the cache as the work before it on the stream leaves it: where the slabs lie and how large they
are, too, when that is written by a kernel right before the call."""
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


@pytest.mark.parametrize("B,h,hk,D,longest", [(1, 8, 8, 128, 700), (2, 8, 2, 64, 90), (12, 16, 16, 128, 200), (1, 32, 2, 128, 1300)])
@pytest.mark.parametrize("between", [False, True])
def test_slabs_laid_out_right_before_the_step(B, h, hk, D, longest, between):
    """Two layouts of one pool (the slabs in order with tight capacities, then in reverse with other lengths), written in
    turn by kernels right before every step; with `between`, an append that keeps nothing runs in between, a kernel
    that lets its successor start before it has waited for its predecessor."""
    slabs = B * hk
    shape = LayerShape(B, longest + 8, 64, h, D, 1, 64, "bf16", kv_heads=hk)
    rng = np.random.default_rng(longest)
    layouts = []
    for turn in range(2):
        lens = rng.integers(0, 70, size=slabs)
        lens[turn] = longest
        order = np.arange(slabs)[::-1 if turn else 1]
        off = np.zeros(slabs, dtype=np.int64)
        off[order] = np.cumsum(np.concatenate([[0], lens[order][:-1] + 1]))
        layouts.append((off, (lens + 1).astype(np.int32), lens.astype(np.int32)))
    pool = max(int((lay[1]).sum()) for lay in layouts)
    k, v = (inputs.randn((pool, D), 41 + i, DEV, torch.bfloat16) for i in (0, 1))
    dev = [[torch.from_numpy(x).to(DEV) for x in lay] for lay in layouts]
    cache = ag.RaggedCache(k, v, *(t.clone() for t in dev[0]), longest + 1)
    q, kn, vn, _ = inputs.decode_inputs(shape, 50, 0, DEV)
    none = torch.zeros(slabs, dtype=torch.uint8, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    desc, ws = ag.make_desc(shape), ag.workspace(ag.make_desc(shape), ag.AG_CALL_DECODE)
    outs = [torch.full_like(q, float("nan")) for _ in range(16)]
    one, one64 = torch.ones_like(cache.len), torch.ones_like(cache.row_off)
    torch.cuda.synchronize()
    for i, o in enumerate(outs):
        off, cap, length = dev[i % 2]
        torch.mul(length, one, out=cache.len)
        torch.mul(cap, one, out=cache.cap)
        torch.mul(off, one64, out=cache.row_off)
        if between:
            ag.ag_cache_append(desc, kn, vn, none, cache, status)
        ag.ag_decode_step(desc, q, kn, vn, none, cache, 0.0, o, status, ws)
    torch.cuda.synchronize()
    for turn in range(2):
        off, cap, lens = layouts[turn]
        held = [[{"k": T.f64(k[off[s]:off[s] + lens[s]]), "v": T.f64(v[off[s]:off[s] + lens[s]])}
                 for s in range(b * hk, (b + 1) * hk)] for b in range(B)]
        want = orc.decode_attention(T.f64(q), T.f64(kn), T.f64(vn), held)
        T.check_close(T.f64(outs[turn]), want, "bf16", f"layout {turn}")
        for o in outs[turn::2]:
            assert torch.equal(o, outs[turn])
    assert int(status.item()) == 0 and ag.ag_device_wait_timeouts() == 0
