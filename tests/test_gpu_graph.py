"""One transfer step recorded as CUDA graphs (alignment + plan, transfer)
and replayed: every replay must equal, bit for bit, an eager step on the
same buffer contents (the same kernels with the same parameters), also
after the sender cache changes between replays."""

import pytest
import torch

from gpu_harness import Case
from paper_2609_32259_gb300 import binding as B
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SENTINEL = 77.0


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


CASES = {
    "tiny_f32_overlap_interp": W.tiny,
    "ta_paper3": lambda: W.llama_to_ministral(600).with_(L_s=4, L_r=5),
    "overlap_after_map_paged": lambda: W.qwen25_to_llama_batched(
        n_req=3, lo=40, hi=300, seed=71).with_(L_s=4, L_r=3, align_mode="overlap_mean"),
    "interp_wide": lambda: W.llama_to_ministral(500).with_(L_s=5, L_r=3, layer_mode="interp"),
}


@pytest.mark.parametrize("over", [
    dict(layer_mode="interp"), dict(sender_k_rotated=True),
    dict(layer_mode="interp", align_mode="overlap_mean")])
def test_graphs_of_one_plan_side_by_side(over):
    """Two graphs of one plan with computed map input rows, each on its own
    caches, replayed on two streams beside an eager transfer on a third: none
    takes another's rows."""
    w = W.llama_to_ministral(1500).with_(L_s=6, L_r=5, **over)
    c = Case(w).run()
    plan = c.job.plan
    senders = [c.sender.flip(2 * i % 3).contiguous() if i else c.sender for i in range(3)]
    want, outs = [], [torch.empty_like(c.job.receiver) for _ in senders]
    for s, o in zip(senders, outs):
        B.transfer(plan, s, o)
        torch.cuda.synchronize()
        want.append(o.clone())
    graphs = [torch.cuda.CUDAGraph() for _ in range(2)]
    for g, s, o in zip(graphs, senders, outs):
        with torch.cuda.graph(g):
            B.transfer(plan, s, o, torch.cuda.current_stream())
    streams = [torch.cuda.Stream() for _ in senders]
    for o in outs:
        o.fill_(SENTINEL)
    torch.cuda.synchronize()
    for _ in range(10):
        for i, st in enumerate(streams):
            with torch.cuda.stream(st):
                graphs[i].replay() if i < 2 else B.transfer(plan, senders[i], outs[i], st)
    torch.cuda.synchronize()
    assert c.job.device_status() == 0
    for o, ref in zip(outs, want):
        assert torch.equal(o, ref)


@pytest.mark.parametrize("name", sorted(CASES))
def test_graph_replay_equals_eager_step(name):
    c = Case(CASES[name](), sentinel=SENTINEL).run()
    c.job.capture()
    gen = torch.Generator(device="cuda")
    gen.manual_seed(5)
    for trial in range(3):
        if trial:
            c.sender.copy_(torch.randn(c.sender.shape, generator=gen, device="cuda")
                           .to(c.sender.dtype))
        c.job.step()
        torch.cuda.synchronize()
        ref = c.job.receiver.clone()
        c.job.receiver.fill_(SENTINEL)
        c.job.replay()
        torch.cuda.synchronize()
        assert c.job.device_status() == 0
        assert torch.equal(c.job.receiver, ref), (name, trial)
    # the replayed step also matches the oracle on the last sender contents
    c.check_parity()
