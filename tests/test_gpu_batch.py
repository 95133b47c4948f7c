"""hf_transfer_batch: the six directions of a three-agent message round
(message spans after a context, every family pair) in one launch.  Each
direction must equal, bit for bit, its own hf_transfer (the same tiles, the
same code), and match the fp64 oracle within the parity tolerance."""

import ctypes

import numpy as np
import pytest
import torch

from gpu_harness import Case
from paper_2609_32259_gb300 import binding as B
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SENTINEL = 99.0


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


def test_message_round_batch_matches_single_transfers_and_oracle():
    cases = [Case(w, sentinel=SENTINEL).run() for w in W.message_round(msg_tokens=160)]
    single = [c.job.receiver.clone() for c in cases]
    for c in cases:
        c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                     [c.job.receiver for c in cases])
    torch.cuda.synchronize()
    for c, ref in zip(cases, single):
        assert torch.equal(c.job.receiver, ref), c.w.name
        c.check_parity()


def _captured_nodes(cases):
    """Number of launches of one batch of the cases, as a capture records them."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                         [c.job.receiver for c in cases], torch.cuda.current_stream())
    nodes = ctypes.c_size_t(0)
    cudart = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    assert cudart.cudaGraphGetNodes(ctypes.c_void_p(g.raw_cuda_graph()), None,
                                    ctypes.byref(nodes)) == 0
    return nodes.value


def test_batch_of_short_long_and_empty_directions():
    """Short messages alone would take single-CTA tiles; beside longer ones, and
    beside a direction without tokens, all run in one launch."""
    ws = [W.llama_to_qwen25(400).with_(L_s=4, L_r=3), W.llama_to_ministral(700).with_(L_s=4, L_r=3),
          W.llama_to_qwen25(90).with_(L_s=4, L_r=3, align_mode="same_index")]
    cases = [Case(w, sentinel=SENTINEL).run() for w in ws]
    single = [c.job.receiver.clone() for c in cases]
    empty = Case(W.llama_to_ministral(5).with_(L_s=4, L_r=3))
    empty.job.desc._r[1] = 0  # no receiver token
    empty.job.make_plan()
    empty.job.receiver.fill_(SENTINEL)
    cases.insert(1, empty)
    for c in cases:
        c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                     [c.job.receiver for c in cases])
    torch.cuda.synchronize()
    for c, ref in zip([c for c in cases if c is not empty], single):
        assert torch.equal(c.job.receiver, ref), c.w.name
    assert (empty.job.receiver == SENTINEL).all()
    assert _captured_nodes(cases) == 1


def test_batch_mixing_operand_paths():
    """Plans that differ in dtype or operand path (copied rows vs built rows)
    go to separate launches; results equal their single transfers."""
    ws = [W.message_round(msg_tokens=60)[0], W.tiny(),
          W.llama_to_ministral(300).with_(L_s=3, L_r=3, align_mode="overlap_mean")]
    cases = [Case(w, sentinel=SENTINEL).run() for w in ws]
    single = [c.job.receiver.clone() for c in cases]
    for c in cases:
        c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                     [c.job.receiver for c in cases])
    torch.cuda.synchronize()
    for c, ref in zip(cases, single):
        assert torch.equal(c.job.receiver, ref), c.w.name


def test_batch_of_computed_operand_rows():
    """Directions with computed operand rows (layers blended per sender token,
    overlap pooling after the map), each with its own pass that makes them: each
    equals its single transfer and the oracle."""
    ws = [W.llama_to_ministral(700).with_(L_s=5, L_r=4, layer_mode="interp",
                                          align_mode="overlap_mean"),
          W.llama_to_qwen25(500).with_(L_s=6, L_r=3, layer_mode="interp",
                                       align_mode="overlap_mean"),
          W.qwen25_to_llama_batched(n_req=2, lo=80, hi=300, seed=61).with_(
              L_s=4, L_r=3, layer_mode="interp", align_mode="overlap_mean")]
    cases = [Case(w, sentinel=SENTINEL).run() for w in ws]
    single = [c.job.receiver.clone() for c in cases]
    for c in cases:
        c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                     [c.job.receiver for c in cases])
    torch.cuda.synchronize()
    for c, ref in zip(cases, single):
        assert torch.equal(c.job.receiver, ref), c.w.name
        c.check_parity()


BUILT = {
    # staged blends in wide tiles, pooling after the map
    "overlap_interp": [W.llama_to_ministral(700).with_(L_s=5, L_r=4, layer_mode="interp",
                                                       align_mode="overlap_mean"),
                       W.llama_to_qwen25(500).with_(L_s=6, L_r=3, layer_mode="interp",
                                                    align_mode="overlap_mean")],
    # staged blends, one row per distinct alignment row, paged and not
    "interp": [W.llama_to_ministral(400).with_(L_s=5, L_r=4, layer_mode="interp"),
               W.qwen25_to_llama_batched(n_req=2, lo=80, hi=300, seed=61).with_(
                   L_s=4, L_r=3, layer_mode="interp")],
    # rows built in registers: keys rotated back, pooling before the map
    "rotated": [W.llama_to_ministral(300).with_(L_s=4, L_r=3, sender_k_rotated=True),
                W.llama_to_qwen25(150).with_(L_s=4, L_r=3, sender_k_rotated=True)],
    "pooled_knorm": [W.llama_to_ministral(300).with_(L_s=4, L_r=3, align_mode="overlap_mean",
                                                     knorm=True, sender_k_rotated=True),
                     W.llama_to_qwen25(150).with_(L_s=4, L_r=3, align_mode="overlap_mean",
                                                  knorm=True, sender_k_rotated=True)],
}


def _without_room(job):
    """Makes the plan in a workspace without room for made operand rows (an fp32
    plan's: those make none)."""
    dtype, job.desc.c.dtype = job.desc.c.dtype, B.DTYPES["f32"]
    job.workspace = torch.empty(B.plan_workspace_size(job.desc), dtype=torch.uint8, device="cuda")
    job.desc.c.dtype = dtype
    job.make_plan()


@pytest.mark.parametrize("name", sorted(BUILT))
def test_batch_of_built_operand_rows(name):
    """Directions whose operand rows the loader warps build, in one launch: in
    workspaces without room for made rows, and captured."""
    cases = [Case(w, sentinel=SENTINEL).run() for w in BUILT[name]]
    single = [c.job.receiver.clone() for c in cases]
    args = ([c.sender for c in cases], [c.job.receiver for c in cases])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        B.transfer_batch([c.job.plan for c in cases], *args, torch.cuda.current_stream())
    assert _captured_nodes(cases) == 1
    plans = [c.job.plan for c in cases]  # the graph's
    for c in cases:
        c.job.plan = None
        _without_room(c.job)
    for launch in (g.replay, lambda: B.transfer_batch([c.job.plan for c in cases], *args)):
        for c in cases:
            c.job.receiver.fill_(SENTINEL)
        launch()
        torch.cuda.synchronize()
        for c, ref in zip(cases, single):
            assert c.job.device_status() == 0
            assert torch.equal(c.job.receiver, ref), c.w.name
    del plans


def test_batch_mixing_layer_tables():
    """A KV Ridge direction (an explicit eight-segment table), a paper3
    direction and an interpolated one in one batch: each equals its single
    transfer and stays within the parity tolerance of the oracle."""
    ws = [W.qwen25_to_llama_kv_ridge(600),
          W.qwen25_to_llama_batched(n_req=2, lo=100, hi=400, seed=44).with_(L_s=28, L_r=32),
          W.llama_to_ministral(500).with_(L_s=5, L_r=6, layer_mode="interp")]
    cases = [Case(w, sentinel=SENTINEL).run() for w in ws]
    single = [c.job.receiver.clone() for c in cases]
    for c in cases:
        c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan for c in cases], [c.sender for c in cases],
                     [c.job.receiver for c in cases])
    torch.cuda.synchronize()
    for c, ref in zip(cases, single):
        assert torch.equal(c.job.receiver, ref), c.w.name
    cases[0].check_parity(layers=[0, 13, 31])
    cases[2].check_parity()


def test_batch_of_one_and_empty_batch():
    c = Case(W.message_round(msg_tokens=40)[1], sentinel=SENTINEL).run()
    ref = c.job.receiver.clone()
    c.job.receiver.fill_(SENTINEL)
    B.transfer_batch([c.job.plan], [c.sender], [c.job.receiver])
    B.transfer_batch([], [], [])
    torch.cuda.synchronize()
    assert torch.equal(c.job.receiver, ref)


def test_batch_rejects_a_repeated_plan():
    c = Case(W.message_round(msg_tokens=40)[0]).run()
    with pytest.raises(B.HFError) as e:
        B.transfer_batch([c.job.plan, c.job.plan], [c.sender, c.sender],
                         [c.job.receiver, c.job.receiver])
    assert e.value.status == B.HF_ERR_INVALID_ARGUMENT
