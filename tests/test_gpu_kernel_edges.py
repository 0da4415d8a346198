"""Kernels at the edges of their tiles and of the rules that choose between their forms, against the
oracle."""
import numpy as np
import pytest
import torch

from oracle import sq_oracle as O
from paper_2404_04793_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


def workload(name, wid, **kw):
    base = dict(n_layer=1, n_q_head=4, n_kv_head=2, head_dim=64, hidden=64, batch=1, prompt=96, steps=1,
                dtype=torch.bfloat16, policy=synth.H2O, budget_pct=100.0, p=0.3, heavy_mode="uniform4")
    return synth.Workload(name, wid, **dict(base, **kw))


# Prompt scores on the tensor cores: key tiles cut into pieces by heads (as many pieces as heads, a last
# piece with fewer heads, one piece), one tile, a tile of one key, full and ragged last tiles
@pytest.mark.parametrize("head_dim,hq,hkv,batch,prompt", [
    (64, 71, 1, 1, 128), (64, 71, 1, 2, 385), (64, 71, 1, 9, 1155), (128, 20, 2, 1, 257), (128, 4, 1, 1, 1), (128, 6, 1, 3, 640),
    (64, 3, 3, 2, 300)])
def test_prompt_scores_cut_by_heads(head_dim, hq, hkv, batch, prompt):
    w = workload("edge", 9100 + prompt, head_dim=head_dim, n_q_head=hq, n_kv_head=hkv, batch=batch, prompt=prompt,
                 heavy_mode="uniform4" if prompt > 8 else "none")
    ctx = H.make_ctx(w, b_init=prompt)
    for _ in range(2):                                # the second pass finds the pieces' counters as the first left them
        ctx.begin_sequence_batch(batch, prompt)
        ctx.set_budgets([prompt])                     # keep everything: scores are read back per token
        q, k, v = synth.prompt_qkv(w, 0, DEV)
        ctx.prefill_compress(0, k, v, q)
    g = w.group
    for s in sorted({0, batch - 1}):
        for h in sorted({0, hkv - 1}):
            pos, acc = ctx.get_kept(0, s, h)
            assert pos == list(range(prompt))
            want = O.prefill_scores(H.f64(q[s, h * g:(h + 1) * g]), H.f64(k[s, h]))
            np.testing.assert_allclose(acc, want, rtol=H.RTOL_ACC[w.dtype], atol=1e-6)
    assert ctx.status() == 0
