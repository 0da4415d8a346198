"""What the host side of a context holds: refused calls leave it as it was, read-backs wait, stream capture."""
import os
import subprocess
import sys

import pytest
import torch

from paper_2404_04793_b200 import binding as B
from paper_2404_04793_b200 import synth
from tests import helpers as H

pytestmark = pytest.mark.gpu
DEV = "cuda"


def workload(**kw):
    base = dict(n_layer=3, n_q_head=4, n_kv_head=2, head_dim=64, hidden=64, batch=2, prompt=96, steps=4,
                dtype=torch.bfloat16, policy=synth.SLIDING_WINDOW, budget_pct=50.0, p=0.3)
    return synth.Workload("host state", 71, **dict(base, **kw))


def filled(w, budgets, **over):
    ctx = H.make_ctx(w, **over)
    ctx.begin_sequence_batch(w.batch, w.prompt)
    ctx.set_budgets(budgets)
    for l in range(w.n_layer):
        _, k, v = synth.prompt_qkv(w, l, DEV, need_q=False)
        ctx.prefill_compress(l, k, v)
    return ctx


def step(ctx, w, t, inputs=None):
    q, kn, vn = inputs or synth.decode_qkv(w, t, DEV)
    out = torch.empty_like(q)
    ctx.decode_step(0, w.n_layer, q, kn, vn, out)
    return out


@pytest.mark.parametrize("per_sequence", [0, 1])
@pytest.mark.parametrize("fault", [dict(budget=0), dict(cap=7), dict(n_unit=99), dict(n_tok=1 << 30)])
def test_a_refused_import_leaves_budgets_and_cache(per_sequence, fault):
    w = workload()
    one = [60, 20, 50]
    budgets = [one, [40, 30, 61]] if per_sequence else one
    ctx, twin = (filled(w, budgets, per_sequence_budgets=per_sequence) for _ in range(2))
    assert torch.equal(step(ctx, w, 0), step(twin, w, 0))
    table = ctx.export_layout()
    for name, value in fault.items():
        setattr(table[len(table) - 1], name, value)          # the last entry
    with pytest.raises(B.SqError) as e:
        ctx.import_layout(table)
    assert e.value.code == B.SQ_ERR_INVALID_ARG
    assert ctx.get_budgets() == twin.get_budgets()
    assert ctx.get_budgets()[0] == budgets
    assert torch.equal(step(ctx, w, 1), step(twin, w, 1))
    tighter = [[b // 2 for b in r] for r in budgets] if per_sequence else [b // 2 for b in budgets]
    for c in (ctx, twin):
        c.evict(0, w.n_layer, tighter)
    assert ctx.get_budgets() == twin.get_budgets()
    assert torch.equal(step(ctx, w, 2), step(twin, w, 2))
    assert ctx.status() == 0


def test_reading_budgets_waits_for_the_device():
    w = workload()
    ctx = filled(w, [60, 20, 50])
    H.feed_importance(ctx, w)
    for allocate in (False, True):
        if allocate:
            ctx.allocate_budgets(w.b_init, w.p)
        else:
            ctx.set_budgets([60, 20, 50])
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(100_000_000)                   # some 50 ms
            done = side.record_event()
        ctx.get_budgets()
        assert done.query()


def test_calls_under_stream_capture():
    """Importance and allocation can be captured and replayed (the budgets are then read back); what uploads host
    tables is refused, changes nothing, and neither leaves anything behind that a later call stumbles on."""
    w = workload()
    hidden = [synth.hidden_pair(w, l, DEV) for l in range(w.n_layer)]

    def measure(ctx):
        ctx.begin_sequence_batch(w.batch, w.prompt)
        for l, (a, b) in enumerate(hidden):
            ctx.layer_importance(l, a, b)
        ctx.allocate_budgets(w.b_init, w.p)

    ctx, twin = filled(w, [60, 20, 50]), filled(w, [60, 20, 50])
    budgets = ctx.get_budgets()
    layout = ctx.export_layout()
    inputs = synth.decode_qkv(w, 0, DEV)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for call in (lambda: ctx.set_budgets([50, 30, 40]), lambda: ctx.evict(0, 3, [30, 10, 25]), lambda: ctx.import_layout(layout)):
            with pytest.raises(B.SqError) as e:
                call()
            assert e.value.code == B.SQ_ERR_CUDA
        out = step(ctx, w, 0, inputs)
    graph.replay()
    assert ctx.get_budgets() == budgets
    assert torch.equal(out, step(twin, w, 0))
    assert torch.equal(step(ctx, w, 1), step(twin, w, 1))
    measure(twin)
    want = twin.get_budgets()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        measure(ctx)
        with pytest.raises(B.SqError):                       # needs the budgets on the host
            step(ctx, w, 0, inputs)
    for _ in range(2):
        graph.replay()
        assert ctx.get_budgets() == want
    for _ in range(3):                                       # more calls than staging slots
        ctx.begin_sequence_batch(w.batch, w.prompt)
        ctx.set_budgets([60, 20, 50])
    twin = filled(w, [60, 20, 50])
    for l in range(w.n_layer):
        _, k, v = synth.prompt_qkv(w, l, DEV, need_q=False)
        ctx.prefill_compress(l, k, v)
    assert torch.equal(step(ctx, w, 0), step(twin, w, 0))
    measure(ctx)
    assert ctx.get_budgets() == want and ctx.status() == 0
    del graph
    ctx.close()
    assert torch.zeros(1, device=DEV).item() == 0.0


_HUGE = """
import ctypes, resource, torch
from paper_2404_04793_b200 import binding as B
torch.zeros(1, device="cuda")
now = 4096 * int(open("/proc/self/statm").read().split()[0])
resource.setrlimit(resource.RLIMIT_AS, (now + (64 << 30), now + (64 << 30)))   # no table may take the machine's memory
cfg = B.make_config(n_layer=256, n_q_head=1, n_kv_head=1, head_dim=64, hidden=64, max_batch=2**31 - 1, max_prompt=1,
                    max_new_tokens=1, dtype=torch.bfloat16, policy=0, page_tokens=1, per_sequence_budgets=1)
pool, ws = B.sq_query_sizes(cfg, 1)
h = ctypes.c_void_p()
print("code", B.lib().sq_ctx_create(ctypes.byref(cfg), 1, 256, pool, 256, ws, ctypes.byref(h)), h.value)
"""


def test_a_context_out_of_reach_is_an_error():
    """Host tables for 5e11 descriptors (the device pointers are never used): an error code, no exception through C."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _HUGE], capture_output=True, text=True, cwd=root, timeout=300)
    assert r.returncode == 0 and f"code {B.SQ_ERR_CUDA} None" in r.stdout, (r.returncode, r.stdout, r.stderr[-500:])
