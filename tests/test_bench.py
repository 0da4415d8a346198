"""The attention kernel that the bench's records name is the one that the library launches."""
import pytest
import torch

import bench
from paper_2404_04793_b200 import synth


@pytest.mark.parametrize("name,over,per_layer,kernel", [
    ("llama2_70b", {}, True, "decode_attn_mma_low_kernel"), ("llama2_70b", {}, False, "decode_attn_mma_low_kernel"),
    ("mistral_7b", {}, True, "decode_attn_mma_low_kernel"), ("llama2_7b", {}, True, "decode_attn_mma_low_kernel"),
    ("llama2_7b", dict(prompt=100), False, "decode_attn_kernel"), ("tiny", {}, False, "decode_attn_kernel"),
    ("falcon_7b_max", {}, True, "decode_attn_tc_stream_kernel"), ("falcon_7b_max", {}, False, "decode_attn_tc_kernel"),
    ("mistral_7b", dict(n_q_head=128), True, "decode_attn_mma_kernel")])
def test_kernel_names(name, over, per_layer, kernel):
    w = synth.WORKLOADS[name]().replace(**over)
    budgets = [max(1, int(w.b_init * w.p)), int(w.b_init * 1.5)]
    assert bench.decode_kernel_of(w, budgets, per_layer) == kernel


@pytest.mark.gpu
@pytest.mark.parametrize("hq,hkv,head_dim,batch,budgets,dtype,policy", [
    (4, 4, 128, 2, [900, 300], torch.bfloat16, synth.SLIDING_WINDOW), (4, 4, 128, 2, [150, 60], torch.bfloat16, synth.SLIDING_WINDOW),
    (8, 8, 64, 128, [600, 900], torch.bfloat16, synth.H2O), (8, 2, 64, 1, [300, 90], torch.bfloat16, synth.H2O),
    (32, 1, 64, 1, [300, 90], torch.bfloat16, synth.H2O), (71, 1, 64, 150, [2100, 2300], torch.bfloat16, synth.SLIDING_WINDOW),
    (40, 1, 128, 1, [100, 64], torch.bfloat16, synth.SLIDING_WINDOW), (2, 2, 64, 1, [100, 64], torch.float32, synth.H2O)])
@pytest.mark.parametrize("per_layer", [True, False])
def test_kernel_names_are_those_launched(hq, hkv, head_dim, batch, budgets, dtype, policy, per_layer):
    from tests import helpers as H
    w = synth.Workload("label", 91, n_layer=2, n_q_head=hq, n_kv_head=hkv, head_dim=head_dim, hidden=64, batch=batch, prompt=max(budgets) + 1,
                       steps=1, dtype=dtype, policy=policy, budget_pct=100.0, p=0.3)
    ctx = H.make_ctx(w, b_init=max(budgets))
    ctx.begin_sequence_batch(batch, w.prompt)
    ctx.set_budgets(budgets)
    _, k, v = synth.prompt_qkv(w, 0, "cuda", need_q=False)
    for l in range(2):
        ctx.prefill_compress(l, k, v, None, torch.rand(batch, hkv, w.prompt, device="cuda") if policy == synth.H2O else None)
    q, kn, vn = synth.decode_qkv(w, 0, "cuda")
    out = torch.empty_like(q)
    torch.cuda.synchronize()
    longest = budgets.index(max(budgets))
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        if per_layer:
            ctx.decode_step(longest, longest + 1, q[longest], kn[longest], vn[longest], out[longest])
        else:
            ctx.decode_step(0, 2, q, kn, vn, out)
        torch.cuda.synchronize()
    names = {e.key.split("<")[0].split("::")[-1] for e in prof.key_averages() if "decode_attn" in e.key}
    assert names == {bench.decode_kernel_of(w, budgets, per_layer)}


@pytest.mark.gpu
@pytest.mark.parametrize("over", [{}, dict(prompt=700), dict(dtype=torch.bfloat16), dict(policy=synth.SLIDING_WINDOW)])
def test_counted_launches_are_made(over):
    """The launches of a pass that the bench counts are at least made, and no more are counted."""
    from paper_2404_04793_b200 import engine
    w = synth.tiny().replace(steps=3, **over)
    job, inp = engine.Job(w, "cuda"), engine.ResidentInputs(w, "cuda")
    job.run(inp)
    torch.cuda.synchronize()
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        job.run(inp)
        torch.cuda.synchronize()
    made = sum(e.count for e in prof.key_averages() if "sq::" in e.key)
    counted = job.kernel_launches_per_pass(inp)
    assert counted <= made <= counted + w.n_layer + w.steps   # copies of many heavy rows, a second launch of a decode step
