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


# Prompt scores: key tiles cut into pieces (tensor cores: by heads; as many pieces as heads, a last piece with
# fewer heads, one piece), one tile, a tile of one key, full and ragged last tiles
@pytest.mark.parametrize("head_dim,hq,hkv,batch,prompt", [
    (64, 71, 1, 1, 128), (64, 71, 1, 2, 385), (64, 71, 1, 9, 1155), (128, 20, 2, 1, 257), (128, 4, 1, 1, 1), (128, 6, 1, 3, 640),
    (64, 3, 3, 2, 300)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])   # fp32: both tile heights, one and many pieces
def test_prompt_scores_cut_into_pieces(dtype, head_dim, hq, hkv, batch, prompt):
    w = workload("edge", 9100 + prompt, dtype=dtype, head_dim=head_dim, n_q_head=hq, n_kv_head=hkv, batch=batch, prompt=prompt,
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


# fp32 prompts that go in one launch, and just not: one query, edges of a query tile and of a key tile, the most (head, query
# tile) pairs of a KV head with one head and with several, one more than that
@pytest.mark.parametrize("head_dim,hq,hkv,batch,prompt", [
    (64, 2, 2, 1, 1), (64, 2, 1, 3, 31), (128, 1, 1, 2, 32), (64, 6, 3, 2, 65), (128, 2, 2, 2, 127), (64, 5, 1, 2, 128),
    (128, 5, 1, 1, 129), (64, 1, 1, 2, 640), (128, 2, 2, 1, 639), (64, 1, 1, 1, 641)])
def test_prompt_scores_of_short_fp32_prompts(head_dim, hq, hkv, batch, prompt):
    test_prompt_scores_cut_into_pieces(torch.float32, head_dim, hq, hkv, batch, prompt)


# A row's reference is its maximum so far: some rows rise far above their first keys, by amounts beyond fp32's range too, some
# less, some not at all; both tile widths, both halves of a wide tile, the last tile ragged
@pytest.mark.parametrize("head_dim,hq", [(64, 3), (64, 60), (128, 2)])   # (60 heads: enough CTAs for the narrow tiles)
@pytest.mark.parametrize("prompt", [200, 700])
def test_prompt_scores_of_rising_rows(head_dim, hq, prompt):
    w = workload("rising", 9150 + prompt, head_dim=head_dim, n_q_head=hq, n_kv_head=1, batch=3, prompt=prompt, heavy_mode="none")
    ctx = H.make_ctx(w, b_init=prompt)
    ctx.begin_sequence_batch(3, prompt)
    ctx.set_budgets([prompt])
    q, k, v = synth.prompt_qkv(w, 0, DEV)
    k[1, :, 140:] *= 12.0          # logits of some tens
    k[2, :, 150:170] *= 100.0      # beyond 2^128
    ctx.prefill_compress(0, k, v, q)
    for s in range(3):
        pos, acc = ctx.get_kept(0, s, 0)
        assert pos == list(range(prompt))
        want = O.prefill_scores(H.f64(q[s]), H.f64(k[s, 0]))
        # logits of up to L = 100 * 6 are fp32 sums of head_dim products and meet the stored log-sum-exp at that size: 2^-23 L
        # each in the exponent, twice; scores below 2^-126 of a row count as that
        np.testing.assert_allclose(acc, want, rtol=H.RTOL_ACC[w.dtype] * (10 if s == 2 else 1), atol=1e-6)
    assert ctx.status() == 0


# Rows whose first keys weigh next to nothing and one later key nearly everything, each such key alone seen by one row of one head,
# so that its score is that row's weight and no sum over rows evens the rounding out
@pytest.mark.parametrize("head_dim,hq,batch", [(64, 3, 1), (64, 60, 3), (128, 2, 2)])   # wide tiles, narrow tiles, head_dim 128
def test_prompt_score_of_one_late_key_per_row(head_dim, hq, batch):
    prompt, n = 700, 32
    w = workload("late key", 9180, head_dim=head_dim, n_q_head=hq, n_kv_head=1, batch=batch, prompt=prompt, heavy_mode="none")
    q, k, v = (t.zero_() for t in synth.prompt_qkv(w, 0, DEV))
    gen = torch.Generator().manual_seed(9180 + head_dim)
    scale = 1.4426950408889634 / head_dim ** 0.5               # logits in powers of two
    late = 300 + 7 * torch.arange(n)                           # every place of a tile's pairs; in tiles off the diagonal
    k[:, 0, :, :n] = -26.0 / 4 / scale                         # a late row's other keys: 2^-26 and less
    k[:, 0, late, torch.arange(n)] = ((1 + torch.rand(n, generator=gen)) / 4.25 / scale).to(k)
    k[:, 0, late, 40] = -60.0 / 4 / scale                      # the other rows do not see the late keys
    q[:, :, :, 40] = 4.0
    rows = torch.arange(prompt - n, prompt)
    q[:, 0, rows, 40] = 0.0
    q[:, 0, rows, torch.arange(n)] = (4 + torch.arange(n) % 9 / 32).to(q)
    ctx = H.make_ctx(w, b_init=prompt)
    ctx.begin_sequence_batch(batch, prompt)
    ctx.set_budgets([prompt])
    ctx.prefill_compress(0, k, v, q)
    for s in range(batch):
        _, acc = ctx.get_kept(0, s, 0)
        want = O.prefill_scores(H.f64(q[s]), H.f64(k[s, 0]))
        # The late key's logit and the log-sum-exp lie between 1 and 2 (in powers of two): each is rounded by 2^-24 once it is
        # scaled and once more when it is stored, so the weight by 4 * 2^-24 * ln 2 = 1.7e-7; its exponential by 2.1e-7
        np.testing.assert_allclose(np.asarray(acc)[late], want[late], rtol=3.8e-7, atol=0)
    assert ctx.status() == 0


# Given scores with every bit set (NaN, which no selection has to make sense of): every slot still gets a token of its own and that
# token's rows.  Few heavy rows, copied by the selecting CTA, and more than it copies
@pytest.mark.parametrize("prompt,budget", [(300, 100), (1200, 900), (3000, 1024)])
def test_prompt_selection_with_scores_of_all_ones(prompt, budget):
    w = workload("all ones", 9190 + prompt, prompt=prompt, heavy_mode="none")
    ctx = H.make_ctx(w, b_init=budget)
    ctx.begin_sequence_batch(1, prompt)
    ctx.set_budgets([budget])
    _, k, v = synth.prompt_qkv(w, 0, DEV, need_q=False)
    acc = torch.full((w.n_kv_head, prompt), -1, dtype=torch.int32, device=DEV).view(torch.float32)
    acc[:, 17:budget // 4 + 17:2] = 1.0            # fewer than there are heavy slots
    ctx.prefill_compress(0, k, v, None, acc)
    for h in range(w.n_kv_head):
        pos, _ = ctx.get_kept(0, 0, h)
        assert len(pos) == budget and sorted(set(pos)) == pos and pos[0] >= 0 and pos[-1] == prompt - 1
        assert set(range(17, budget // 4 + 17, 2)) <= set(pos)
        kk, vv = ctx.get_kv(0, 0, h)
        assert torch.equal(kk, k[0, h, pos].cpu()) and torch.equal(vv, v[0, h, pos].cpu())
    assert ctx.status() == 0


# Decode launches of one layer right behind one another start before the launch ahead is done and fetch
# their first rows ahead of it, all but the new token's: its slot goes through every row of the cache,
# and one layer behind itself (n_layer 1) or a stream change must not read ahead
@pytest.mark.parametrize("policy", [synth.SLIDING_WINDOW, synth.H2O])
@pytest.mark.parametrize("dtype,head_dim,hq,hkv,budget", [
    (torch.bfloat16, 128, 2, 2, 70), (torch.bfloat16, 128, 8, 2, 200), (torch.bfloat16, 64, 40, 1, 400), (torch.bfloat16, 64, 128, 1, 140),
    (torch.float32, 64, 6, 2, 50)])
@pytest.mark.parametrize("n_layer", [1, 3])
def test_layer_by_layer_launches_match_the_whole_stack(policy, dtype, head_dim, hq, hkv, budget, n_layer):
    w = workload("chain", 9200 + budget, policy=policy, dtype=dtype, head_dim=head_dim, n_q_head=hq, n_kv_head=hkv,
                 n_layer=n_layer, batch=2, prompt=budget + 9, steps=budget + 5, heavy_mode="none")
    budgets = [max(8, budget - 31 * l) for l in range(n_layer)]
    ctxs = []
    for _ in range(2):
        ctx = H.make_ctx(w, b_init=budget)
        ctx.begin_sequence_batch(w.batch, w.prompt)
        ctx.set_budgets(budgets)
        for l in range(n_layer):
            q, k, v = synth.prompt_qkv(w, l, DEV)
            ctx.prefill_compress(l, k, v, q if policy == synth.H2O else None)
        ctxs.append(ctx)
    stack, chained = ctxs
    side = torch.cuda.Stream()
    for t in range(w.steps):
        q, kn, vn = synth.decode_qkv(w, t, DEV)
        a, b = torch.empty_like(q), torch.empty_like(q)
        torch.cuda.synchronize()
        stack.decode_step(0, n_layer, q, kn, vn, a)
        if t % 7 == 3:                                # the step's last layer on another stream, behind an event
            ev = torch.cuda.Event()
            for l in range(n_layer - 1):
                chained.decode_step(l, l + 1, q[l], kn[l], vn[l], b[l])
            ev.record()
            with torch.cuda.stream(side):
                side.wait_event(ev)
                l = n_layer - 1
                chained.decode_step(l, l + 1, q[l], kn[l], vn[l], b[l])
                ev.record(side)
            torch.cuda.current_stream().wait_event(ev)
        else:
            for l in range(n_layer):
                chained.decode_step(l, l + 1, q[l], kn[l], vn[l], b[l])
        assert torch.allclose(a.float(), b.float(), rtol=0, atol=H.TOL_OUT[dtype])   # other split-K pieces
    for l in range(n_layer):
        for h in range(hkv):
            pa, _ = stack.get_kept(l, 1, h)
            pb, _ = chained.get_kept(l, 1, h)
            assert pa == pb
            ka, va = stack.get_kv(l, 1, h)
            kb, vb = chained.get_kv(l, 1, h)
            assert torch.equal(ka, kb) and torch.equal(va, vb)
    assert stack.status() == 0 and chained.status() == 0


# One bf16 head per KV head keeps its weights at fp32 precision on the tensor cores: with fp32-exact weights
# only the order of the fp32 sums and the bf16 output (half an ulp, 2^-9) separate it from the oracle, where
# bf16 weights would add 2^-9 of the largest term.  Keys that make one weight dominate, after the first
# tile too (the reference moves), lengths around a tile and a warp's share of it
@pytest.mark.parametrize("head_dim,budget", [(128, 1), (128, 17), (128, 64), (128, 65), (64, 300), (128, 1500)])
@pytest.mark.parametrize("hq", [3, 24])
def test_one_and_eight_heads_per_kv_head(head_dim, budget, hq):
    w = workload("one", 9500 + budget, policy=synth.SLIDING_WINDOW, head_dim=head_dim, n_q_head=hq, n_kv_head=3, batch=1,
                 prompt=budget + 3, steps=2, heavy_mode="none")
    ctx = H.make_ctx(w, b_init=budget)
    ctx.begin_sequence_batch(1, w.prompt)
    ctx.set_budgets([budget])
    _, k, v = synth.prompt_qkv(w, 0, DEV, need_q=False)
    k[:, :, 2 * w.prompt // 3:] *= 24.0
    ctx.prefill_compress(0, k, v)
    units = [O.UnitCache(w.policy, budget) for _ in range(3)]
    for h, u in enumerate(units):
        u.prefill(H.f64(k[0, h]), H.f64(v[0, h]))
    for t in range(w.steps):
        q, kn, vn = synth.decode_qkv(w, t, DEV)
        out = torch.empty_like(q)
        ctx.decode_step(0, 1, q, kn, vn, out)
        for h, u in enumerate(units):
            g = w.group
            want = u.decode_step(H.f64(q[0, 0, h * g:(h + 1) * g]), H.f64(kn[0, 0, h]), H.f64(vn[0, 0, h]))
            got = H.f64(out[0, 0, h * g:(h + 1) * g])
            bound = np.abs(want) * 2.0 ** -8 + 1e-4 if g == 1 else np.maximum(H.TOL_OUT[w.dtype], np.abs(want) * 2.0 ** -7)
            assert np.all(np.abs(got - want) <= bound), (t, h, np.max(np.abs(got - want)))
    assert ctx.status() == 0


# The largest weight of a softmax enters the product exactly: it is 1 under a running maximum (or the maximum of the
# first tile), and where the reference stays behind, the weights have more than a bf16's bits.  One key takes a
# good half of the weight, in the second half of a wide tile and past the first tiles of the others; its value
# and the others' nearly cancel, so that the bf16 output does not hide the weights.
@pytest.mark.parametrize("head_dim,group", [(128, 1), (64, 2), (128, 3), (128, 4), (64, 5), (128, 8), (128, 9), (64, 32), (64, 36), (64, 71), (64, 128)])
@pytest.mark.parametrize("policy", [synth.SLIDING_WINDOW, synth.H2O])
def test_the_largest_weight_is_not_rounded(policy, head_dim, group, n=128, at=100):
    w = workload("peak", 9600 + group, policy=policy, head_dim=head_dim, n_q_head=group, n_kv_head=1, prompt=n, steps=1, heavy_mode="none")
    g = torch.Generator().manual_seed(group)
    rnd = lambda *s: torch.randn(*s, generator=g)
    u = rnd(head_dim)
    u /= u.norm()
    k = rnd(1, 1, n + 1, head_dim) * 0.5
    k -= (k @ u).unsqueeze(-1) * u
    k[0, 0, at] = u * 8.0
    x = np.log(n) + (torch.rand(group, generator=g) - 0.5)              # its logit
    q = rnd(1, 1, group, head_dim)
    q += (x * head_dim ** 0.5 / 8.0).view(1, 1, group, 1) * u - (q @ u).unsqueeze(-1) * u
    v = rnd(1, 1, n + 1, head_dim) * 0.3
    v[0, 0, :] -= 1.0
    v[0, 0, at] = 1.0 + rnd(head_dim) * 0.1
    q, k, v = (t.to(torch.bfloat16).to(DEV) for t in (q, k, v))
    ctx = H.make_ctx(w, b_init=n + 8)
    ctx.begin_sequence_batch(1, n)
    ctx.set_budgets([n + 8])
    ctx.prefill_compress(0, k[:, :, :n].contiguous(), v[:, :, :n].contiguous(), None,
                         torch.zeros(1, 1, n, device=DEV) if policy == synth.H2O else None)
    out = torch.empty_like(q)
    ctx.decode_step(0, 1, q, k[:, :, n:].contiguous(), v[:, :, n:].contiguous(), out)
    s = H.f64(q[0, 0]) @ H.f64(k[0, 0]).T / head_dim ** 0.5
    p = np.exp(s - s.max(1, keepdims=True))
    p /= p.sum(1, keepdims=True)
    assert np.all(s.argmax(1) == at)
    vv = H.f64(v[0, 0])
    want = p @ vv
    rest = p.copy()
    rest[:, at] = 0.0
    # independent roundings of the other weights: 2^-8 / sqrt(3) of each at most (rms), five of them for the extreme
    # of some thousand outputs; half an ulp of the output; fp32 sums
    var = (rest ** 2) @ vv ** 2 - 2 * want * ((rest ** 2) @ vv) + want ** 2 * (rest ** 2).sum(1, keepdims=True)
    bound = 5 * 2.0 ** -8 / 3 ** 0.5 * np.sqrt(np.maximum(var, 0)) + 2.0 ** -8 * np.abs(want) + 2e-5
    err = np.abs(H.f64(out[0, 0]) - want)
    assert np.all(err <= bound), float((err / bound).max())
    assert ctx.status() == 0


# Wide groups, few long units: pieces of several tiles on the CTAs of a cluster.  The key lies in a piece's first tile, a later one
# and the new token's tile
@pytest.mark.parametrize("group,at", [(71, 100), (71, 700), (71, 3333), (71, 7980), (33, 1900), (96, 4500)])
@pytest.mark.parametrize("policy", [synth.SLIDING_WINDOW, synth.H2O])
def test_the_largest_weight_of_a_long_unit_is_not_rounded(policy, group, at):
    test_the_largest_weight_is_not_rounded(policy, 64, group, 8000, at)


def lockstep(dtype, head_dim, hq, hkv, batch, budgets, stack, policy=synth.H2O):
    """Decode steps of all layers in one call or layer by layer, each step against the oracle from the library's state."""
    w = workload("fused", 9300 + budgets[0], policy=policy, dtype=dtype, head_dim=head_dim, n_q_head=hq, n_kv_head=hkv, n_layer=len(budgets),
                 batch=batch, prompt=max(budgets) + 5, steps=3, heavy_mode="zipf")
    ctx = H.make_ctx(w, b_init=max(budgets))
    ctx.begin_sequence_batch(batch, w.prompt)
    ctx.set_budgets(budgets)
    g = w.group
    units = {(l, s, h) for l in range(w.n_layer) for s in (0, batch - 1) for h in (0, hkv - 1)}
    for l in range(w.n_layer):
        _, k, v = synth.prompt_qkv(w, l, DEV, need_q=False)
        ctx.prefill_compress(l, k, v, None, synth.prompt_scores_standin(w, l, DEV) if policy == synth.H2O else None)
    for t in range(w.steps):
        q, kn, vn = synth.decode_qkv(w, t, DEV)
        out = torch.empty_like(q)
        # the oracle takes the library's rows and scores before the step: one step's arithmetic is compared
        before = {u: (ctx.get_kept(*u), ctx.get_kv(*u)) for u in units}
        if stack:
            ctx.decode_step(0, w.n_layer, q, kn, vn, out)
        else:
            for l in range(w.n_layer):
                ctx.decode_step(l, l + 1, q[l], kn[l], vn[l], out[l])
        for (l, s, h), ((pos, acc), (kk, vv)) in before.items():
            u = O.UnitCache(w.policy, budgets[l], w.n_sink, w.heavy_num, w.heavy_den)
            u.pos, u.acc, u.K, u.V = list(pos), [float(x) for x in acc], list(H.f64(kk)), list(H.f64(vv))
            u.next_pos = w.prompt + t
            want = u.decode_step(H.f64(q[l, s, h * g:(h + 1) * g]), H.f64(kn[l, s, h]), H.f64(vn[l, s, h]))
            got = H.f64(out[l, s, h * g:(h + 1) * g])
            # outputs beyond 1 meet the bf16 formats: half an ulp of the output, 2^-9 of the weights
            bound = np.maximum(H.TOL_OUT[dtype], np.abs(want) * (2.0 ** -7 if dtype == torch.bfloat16 else 0))
            assert np.all(np.abs(got - want) <= bound)
            pos2, acc2 = ctx.get_kept(l, s, h)
            assert pos2 == u.kept_positions()
            if policy == synth.H2O:
                np.testing.assert_allclose(acc2, u.acc, rtol=H.RTOL_ACC[dtype], atol=1e-6)
    assert ctx.status() == 0


# H2O with the score update inside the attention launch: pieces of a unit on the CTAs of a cluster, with
# empty and ragged pieces, short and long layers, groups that are and are not multiples of four, both
# head dims, and units too long or too many for it
@pytest.mark.parametrize("dtype,head_dim,hq,hkv,batch,budgets", [
    (torch.bfloat16, 128, 8, 2, 1, [1100, 70]), (torch.bfloat16, 128, 5, 1, 2, [129, 2000]), (torch.bfloat16, 64, 32, 1, 1, [513, 64]),
    (torch.bfloat16, 128, 24, 1, 3, [700, 1]), (torch.bfloat16, 64, 6, 3, 50, [300, 290]), (torch.float32, 64, 3, 1, 1, [1400, 33]),
    (torch.float32, 128, 16, 2, 2, [400, 31]), (torch.bfloat16, 128, 3, 3, 2, [900, 260]), (torch.bfloat16, 64, 4, 4, 40, [200, 333]),
    (torch.bfloat16, 128, 31, 1, 1, [9000, 50])])
def test_h2o_scores_in_the_attention_launch(dtype, head_dim, hq, hkv, batch, budgets):
    lockstep(dtype, head_dim, hq, hkv, batch, budgets, stack=False)


# Launches on both sides of the rules that choose between that form and the second launch (started while the attention
# kernel runs out, or after it), and of the one that sends one bf16 head per KV head to the fp32 pipes
@pytest.mark.parametrize("dtype,head_dim,hq,hkv,batch,budgets", [
    (torch.bfloat16, 64, 32, 1, 40, [1500, 200]), (torch.bfloat16, 64, 20, 1, 64, [300, 1400]), (torch.bfloat16, 128, 32, 1, 60, [100, 40]),
    (torch.bfloat16, 128, 16, 2, 160, [400, 130]), (torch.bfloat16, 128, 4, 1, 150, [2900, 700]), (torch.bfloat16, 128, 12, 4, 70, [333, 64]),
    (torch.bfloat16, 64, 10, 10, 130, [60, 200]), (torch.bfloat16, 128, 30, 30, 50, [120, 3]), (torch.float32, 128, 8, 2, 1, [4000, 600]),
    (torch.float32, 64, 16, 2, 70, [1500, 100]), (torch.float32, 64, 6, 6, 210, [200, 90]), (torch.bfloat16, 64, 8, 8, 11, [2049, 300]),
    (torch.bfloat16, 64, 8, 8, 60, [700, 150]), (torch.float32, 128, 8, 2, 4, [330, 80]), (torch.float32, 128, 32, 32, 3, [1300, 40])])
@pytest.mark.parametrize("stack", [False, True])
def test_h2o_forms_of_larger_launches(dtype, head_dim, hq, hkv, batch, budgets, stack):
    lockstep(dtype, head_dim, hq, hkv, batch, budgets, stack)


# Rows of a tile past a unit's heads (decode) or a head's prompt (prompt scores) are the next sequence's: a NaN or an infinity there
# changes no bit of this one's scores.  Wide groups with the scores in the attention launch and in one of their own
@pytest.mark.parametrize("hq,batch,budget", [(71, 3, 400), (33, 2, 150), (97, 2, 300), (65, 160, 140)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_decode_scores_of_a_sequence_stand_alone(hq, batch, budget, bad):
    got = []
    for spoilt in (False, True):
        w = workload("alone", 9250 + hq, n_q_head=hq, n_kv_head=1, batch=batch, prompt=budget + 9, heavy_mode="none")
        ctx = H.make_ctx(w, b_init=budget)
        ctx.begin_sequence_batch(batch, w.prompt)
        ctx.set_budgets([budget])
        _, k, v = synth.prompt_qkv(w, 0, DEV, need_q=False)
        ctx.prefill_compress(0, k, v, None, synth.prompt_scores_standin(w, 0, DEV))
        q, kn, vn = synth.decode_qkv(w, 0, DEV)
        if spoilt:
            q[:, 1] = bad
        out = torch.empty_like(q)
        ctx.decode_step(0, 1, q, kn, vn, out)
        got.append((ctx.get_kept(0, 0, 0), out[0, 0].clone()))
    assert got[0][0] == got[1][0] and torch.equal(got[0][1], got[1][1])


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("head_dim,hq,hkv,prompt", [(64, 4, 2, 333), (64, 130, 2, 333), (128, 4, 2, 200), (64, 2, 2, 31)])
def test_prompt_scores_of_a_sequence_stand_alone(dtype, head_dim, hq, hkv, prompt):
    got = []
    for spoilt in (False, True):
        w = workload("alone", 9260, dtype=dtype, head_dim=head_dim, n_q_head=hq, n_kv_head=hkv, batch=2, prompt=prompt, heavy_mode="none")
        ctx = H.make_ctx(w, b_init=prompt)
        ctx.begin_sequence_batch(2, prompt)
        ctx.set_budgets([prompt])
        q, k, v = synth.prompt_qkv(w, 0, DEV)
        if spoilt:
            q[0, hq // hkv:] = float("nan")
            q[1, 0] = float("inf")
        ctx.prefill_compress(0, k, v, q)
        got.append([ctx.get_kept(0, s, h)[1] for s, h in ((0, 0), (1, hkv - 1))])
    assert got[0] == got[1]


# Wide groups with the pieces of a unit on the CTAs of a cluster: two pieces to the most there are, pieces of one tile and of
# unlike numbers of tiles, a last tile of one slot, the smallest group and the largest that is taken and the next, groups that
# fill no eight, pieces of several tiles whose references follow the maxima, launches whose layers differ too much for the
# form in one call (split-K; the smallest group and the largest too); with the scores and without
@pytest.mark.parametrize("hq,batch,budgets", [
    (71, 1, [1792, 257]), (33, 2, [1921, 129]), (96, 3, [700, 1300]), (97, 2, [300, 260]), (72, 37, [260, 900]), (40, 75, [385, 290]),
    (71, 4, [6000, 300, 260]), (65, 149, [257, 300]), (33, 3, [4000, 150]), (96, 2, [3000, 129, 1000]), (71, 2, [5000, 2600])])
@pytest.mark.parametrize("stack", [False, True])
@pytest.mark.parametrize("policy", [synth.H2O, synth.SLIDING_WINDOW])
def test_wide_groups_over_a_cluster(hq, batch, budgets, stack, policy):
    lockstep(torch.bfloat16, 64, hq, 1, batch, budgets, stack, policy)


# Keys that grow within every piece, so that references move after a piece's first tile: to the maximum of each tile (one long
# unit), or where a weight would be too large (pieces as long as split-K's)
@pytest.mark.parametrize("batch,prompt", [(1, 6000), (33, 2400)])
@pytest.mark.parametrize("policy", [synth.H2O, synth.SLIDING_WINDOW])
def test_growing_logits_over_a_cluster(policy, batch, prompt):
    w = workload("grow", 9280, policy=policy, n_q_head=71, n_kv_head=1, batch=batch, prompt=prompt, steps=2, heavy_mode="none")
    b = prompt + 40
    ctx = H.make_ctx(w, b_init=b)
    ctx.begin_sequence_batch(batch, prompt)
    ctx.set_budgets([b])
    _, k, v = synth.prompt_qkv(w, 0, DEV, need_q=False)
    k *= (1 + torch.arange(prompt, device=DEV) % 384 / 16).to(k)[:, None]
    acc = torch.zeros(batch, 1, prompt, device=DEV) if policy == synth.H2O else None
    ctx.prefill_compress(0, k, v, None, acc)
    units = {s: O.UnitCache(policy, b, w.n_sink, w.heavy_num, w.heavy_den) for s in sorted({0, batch - 1})}
    for s, u in units.items():
        u.prefill(H.f64(k[s, 0]), H.f64(v[s, 0]), None, np.zeros(prompt))
    for t in range(w.steps):
        q, kn, vn = synth.decode_qkv(w, t, DEV)
        out = torch.empty_like(q)
        ctx.decode_step(0, 1, q, kn, vn, out)
        for s, u in units.items():
            want = u.decode_step(H.f64(q[0, s]), H.f64(kn[0, s, 0]), H.f64(vn[0, s, 0]))
            # so peaked that an output is close to one V row: half an ulp of the output, 2^-9 of the weights
            assert np.all(np.abs(H.f64(out[0, s]) - want) <= np.maximum(H.TOL_OUT[w.dtype], 2.0 ** -7 * np.abs(want))), (t, s)
            if policy == synth.H2O:
                # logits of up to 25 * 5, fp32 sums of 64 products: 2^-24 of their size in the exponent, some of them
                np.testing.assert_allclose(ctx.get_kept(0, s, 0)[1], u.acc, rtol=H.RTOL_ACC[w.dtype], atol=1e-6)
    assert ctx.status() == 0


# One bf16 head per KV head on either kernel: few units, between one and two per SM, a few, many; lengths around the
# limits; whole stack (with split units among them) and layer by layer
@pytest.mark.parametrize("head_dim,hkv,batch,budgets", [
    (128, 4, 3, [320, 17, 321]), (64, 16, 9, [320, 64]), (64, 25, 9, [150, 320]), (128, 40, 15, [200, 201]), (64, 40, 15, [190, 260]),
    (64, 60, 20, [1024, 1025, 1]), (128, 60, 20, [512, 600])])
@pytest.mark.parametrize("stack", [False, True])
def test_one_bf16_head_on_either_kernel(head_dim, hkv, batch, budgets, stack):
    w = workload("one head", 9700 + budgets[0], policy=synth.SLIDING_WINDOW, head_dim=head_dim, n_q_head=hkv, n_kv_head=hkv,
                 n_layer=len(budgets), batch=batch, prompt=max(budgets) + 3, steps=2, heavy_mode="none")
    ctx = H.make_ctx(w, b_init=max(budgets))
    ctx.begin_sequence_batch(batch, w.prompt)
    ctx.set_budgets(budgets)
    units = {}
    for l in range(w.n_layer):
        _, k, v = synth.prompt_qkv(w, l, DEV, need_q=False)
        ctx.prefill_compress(l, k, v)
        for s in (0, batch - 1):
            for h in (0, hkv - 1):
                units[l, s, h] = O.UnitCache(w.policy, budgets[l])
                units[l, s, h].prefill(H.f64(k[s, h]), H.f64(v[s, h]))
    for t in range(w.steps):
        q, kn, vn = synth.decode_qkv(w, t, DEV)
        out = torch.empty_like(q)
        if stack:
            ctx.decode_step(0, w.n_layer, q, kn, vn, out)
        else:
            for l in range(w.n_layer):
                ctx.decode_step(l, l + 1, q[l], kn[l], vn[l], out[l])
        for (l, s, h), u in units.items():
            want = u.decode_step(H.f64(q[l, s, h:h + 1]), H.f64(kn[l, s, h]), H.f64(vn[l, s, h]))
            # weights at fp32 precision: the bf16 output (half an ulp, 2^-9) and fp32 sums
            assert np.all(np.abs(H.f64(out[l, s, h:h + 1]) - want) <= np.abs(want) * 2.0 ** -8 + 1e-4), (t, l, s, h)
    assert ctx.status() == 0


# The even-deal form of the wide-group kernel reads ahead in launches right behind one another over different layers: each
# CTA's first tiles, up to the one that holds the new token's slot.  The slots lie in every tile of a unit (H2O: the
# scores decide them, one victim per step in different tiles, so that rows written a step ago are fetched ahead), at the
# front (a full sliding window) or at the end (the last free slot).  New tokens take about half of the weight, so that a
# stale or a missing row shows; every unit is compared.
@pytest.mark.parametrize("policy,room", [(synth.H2O, 0), (synth.SLIDING_WINDOW, 0), (synth.SLIDING_WINDOW, 1)])
def test_even_deal_launches_read_ahead(policy, room):
    batch, b, n_layer, steps, hq, d = 150, 2050 + room, 4, 3, 71, 64
    n = b - room
    w = workload("deal ahead", 9801, policy=policy, n_q_head=hq, n_kv_head=1, n_layer=n_layer, batch=batch, prompt=n, steps=steps, heavy_mode="none")
    ctx = H.make_ctx(w, b_init=b)
    ctx.begin_sequence_batch(batch, n)
    ctx.set_budgets([b] * n_layer)
    g = torch.Generator(device=DEV).manual_seed(5)
    rnd = lambda *sh: torch.randn(*sh, generator=g, device=DEV)
    u = torch.nn.functional.normalize(rnd(d), dim=0)
    keys, vals, order = [], [], []
    for l in range(n_layer):
        k = rnd(batch, 1, n, d) * 0.5
        k = (k - (k @ u).unsqueeze(-1) * u).bfloat16()
        v = rnd(batch, 1, n, d).bfloat16()
        acc = None
        if policy == synth.H2O:
            # the victims of the steps, in order, among the old half: 7, 18 and 11 tiles apart over units and layers
            first = (torch.arange(batch, device=DEV) * 128 * 7 + 128 * 3 * l + 77) % (n // 2)
            vict = torch.stack([(first + i * 419) % (n // 2) for i in range(steps)], 1)
            acc = torch.full((batch, 1, n), 1e4, device=DEV)
            acc[:, 0].scatter_(1, vict, torch.tensor([0.0, 1e3, 2e3], device=DEV).expand(batch, -1))
            order.append(vict)
        ctx.prefill_compress(l, k, v, None, acc)
        keys.append(k[:, 0].double())
        vals.append(v[:, 0].double())
    for t in range(steps):
        q = rnd(n_layer, batch, hq, d)
        # logit of the new token about log(n) + 1
        q = (q + ((np.log(n) + 1) * d ** 0.5 / 8 - (q @ u)).unsqueeze(-1) * u).bfloat16()
        kn = (8.0 * u).expand(n_layer, batch, 1, d).bfloat16().contiguous()
        vn = rnd(n_layer, batch, 1, d).bfloat16()
        out = torch.empty_like(q)
        torch.cuda.synchronize()
        for l in range(n_layer):
            ctx.decode_step(l, l + 1, q[l], kn[l], vn[l], out[l])
        for l in range(n_layer):
            if room and t == 0:
                keys[l] = torch.cat([keys[l], kn[l].double()], 1)
                vals[l] = torch.cat([vals[l], vn[l].double()], 1)
            else:
                slot = order[l][:, t] if policy == synth.H2O else torch.full((batch,), t - room, device=DEV)
                at = torch.arange(batch, device=DEV)
                keys[l][at, slot] = kn[l, :, 0].double()
                vals[l][at, slot] = vn[l, :, 0].double()
            p = torch.softmax(q[l].double() @ keys[l].transpose(1, 2) / d ** 0.5, -1)
            want = p @ vals[l]
            # bf16 weights and output: at most 2^-8 of each term and of the sum
            bound = 2.0 ** -7 * (p @ vals[l].abs())
            assert bool(((out[l].double() - want).abs() <= bound).all()), (t, l, float(((out[l].double() - want).abs() / bound).max()))
            assert float(bound.max()) < 0.1    # a missing new token moves an output by some tenths
    assert ctx.status() == 0


# Selection over the prompt: block sizes by prompt length and the form for longer prompts, ties across the
# threshold, equal scores everywhere, negative scores, all slots heavy but one, none heavy, budgets around the
# prompt; the first victim shows in which token the first append replaces
@pytest.mark.parametrize("prompt", [1, 2, 37, 1024, 1025, 4096, 4097, 9000, 16384, 16385])
@pytest.mark.parametrize("hn,hd", [(1, 2), (0, 1), (9, 10)])
def test_prompt_selection_edges(prompt, hn, hd):
    batch = 6
    w = workload("select", 9400 + prompt, dtype=torch.bfloat16, head_dim=64, n_q_head=2, n_kv_head=1, n_layer=5, batch=batch,
                 prompt=prompt, heavy_num=hn, heavy_den=hd, heavy_mode="none")
    budgets = [max(1, prompt // 3), max(1, prompt - 1), prompt, prompt + 3, 1]
    ctx = H.make_ctx(w, b_init=prompt + 3)
    ctx.begin_sequence_batch(batch, prompt)
    ctx.set_budgets(budgets)
    g = torch.Generator().manual_seed(prompt)
    acc = torch.rand(batch, 1, prompt, generator=g)
    acc[1] = 1.5                                              # all equal
    acc[2] = torch.randint(0, 3, (1, prompt), generator=g)    # a few values, zeros among them
    acc[3] = torch.randn(1, prompt, generator=g)              # negative scores
    acc[4] = torch.round(acc[4] * 64) * 2.0 ** -130           # subnormal
    acc[5, :, : prompt // 2] = -0.0
    _, k, v = synth.prompt_qkv(w, 0, DEV, need_q=False)
    for l in range(w.n_layer):
        ctx.prefill_compress(l, k, v, None, acc.to(DEV))
    for l, b in enumerate(budgets):
        for s in range(batch):
            keep = list(range(prompt)) if prompt <= b else \
                O.c_seq(w.policy, list(range(prompt)), acc[s, 0].double().tolist(), b, w.n_sink, hn, hd)
            pos, got = ctx.get_kept(l, s, 0)
            assert pos == keep, (l, s)
            assert got == [float(acc[s, 0, p]) for p in keep]
    rows = ctx.get_kv(1, 3, 0)[0]
    assert torch.equal(rows, k[3, 0].cpu()[ctx.get_kept(1, 3, 0)[0]])
    before = {(l, s): ctx.get_kept(l, s, 0) for l in range(w.n_layer) for s in range(batch)}
    q, kn, vn = synth.decode_qkv(w, 0, DEV)
    ctx.decode_step(0, w.n_layer, q, kn, vn, torch.empty_like(q))
    for (l, s), (pos, sc) in before.items():
        keep = O.c_seq(w.policy, pos + [prompt], sc + [0.0], budgets[l], w.n_sink, hn, hd) if len(pos) + 1 > budgets[l] else \
            list(range(len(pos) + 1))
        assert ctx.get_kept(l, s, 0)[0] == [(pos + [prompt])[i] for i in keep], (l, s)
    assert ctx.status() == 0


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("hidden,tokens", [(64, 1), (128, 63), (128, 20011), (256, 65), (264, 9)])
def test_importance_of_short_rows(dtype, hidden, tokens):
    """Rows of up to 512 bytes, several per warp; a last group of rows that is not full; rows just longer."""
    w = synth.Workload("short rows", 61, n_layer=1, n_q_head=2, n_kv_head=2, head_dim=64, hidden=hidden, batch=1, prompt=tokens,
                       steps=1, dtype=dtype, policy=synth.SLIDING_WINDOW, budget_pct=100.0, p=1.0)
    g = torch.Generator().manual_seed(tokens + hidden)
    a, d = (torch.randn(tokens, hidden, generator=g).to(dtype) for _ in range(2))
    stored = (a.float() + d.float()).to(dtype)
    x, y = a.double(), stored.double()
    want = float((x * y).sum(1).div(x.norm(dim=1) * y.norm(dim=1)).mean())
    for fused in (False, True):
        ctx = H.make_ctx(w)
        ctx.begin_sequence_batch(1, tokens)
        if fused:
            out = torch.full((tokens, hidden), float("nan"), dtype=dtype, device=DEV)
            ctx.layer_importance_fused(0, a.to(DEV), d.to(DEV), out)
            assert torch.equal(out.cpu(), stored)
        else:
            ctx.layer_importance(0, a.to(DEV), stored.to(DEV))
        ctx.allocate_budgets(tokens, 1.0)
        # three fp32 sums of `hidden` products each and the mean of the fp32 cosines: at most (hidden + warps' rows) ulp
        assert abs(float(ctx.get_cos_sim()[0]) - want) <= (hidden + 64) * 2.0 ** -23
        assert ctx.status() == 0


@pytest.mark.parametrize("hidden,tokens", [(64, 300007), (4096, 20011)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_importance_sums_lose_nothing(dtype, hidden, tokens):
    """Rows whose cosines the kernel's fp32 arithmetic gives exactly (3/5, 4/5, 1 in fp32): their sum over
    many tokens is that of fp64 additions, however few warps share them."""
    w = synth.Workload("exact rows", 62, n_layer=1, n_q_head=2, n_kv_head=2, head_dim=64, hidden=hidden, batch=1, prompt=tokens,
                       steps=1, dtype=dtype, policy=synth.SLIDING_WINDOW, budget_pct=100.0, p=1.0)
    kind = torch.randint(0, 3, (tokens,), generator=torch.Generator().manual_seed(hidden)).to(DEV)
    a = torch.zeros(tokens, hidden, dtype=dtype, device=DEV)
    b = torch.zeros_like(a)
    a[:, 1] = 1.0
    b[:, 1] = torch.tensor([3.0, 4.0, 2.0], device=DEV).to(dtype)[kind]
    b[:, hidden - 1] = torch.tensor([4.0, 3.0, 0.0], device=DEV).to(dtype)[kind]
    want = float(torch.tensor([3.0 / 5.0, 4.0 / 5.0, 1.0], device=DEV).double()[kind].sum())
    for fused in (False, True):
        ctx = H.make_ctx(w)
        ctx.begin_sequence_batch(1, tokens)
        if fused:
            ctx.layer_importance_fused(0, a, b - a, torch.empty_like(a))
        else:
            ctx.layer_importance(0, a, b)
        got, n = ctx.get_importance_state()
        assert n == [tokens]
        assert abs(got[0] - want) <= tokens * 2.0 ** -52 * want     # one rounding of fp64 per addition, both sides
