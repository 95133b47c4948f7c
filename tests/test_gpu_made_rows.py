"""Operand rows made by their own pass against rows built by the transfer
kernel's loader warps (a workspace without room for made rows, as
hf_transfer_noalloc has): the same fp32 sums and roundings and the same order of
products, so the caches must agree bit for bit."""

import pytest
import torch

from paper_2609_32259_gb300 import binding as B
from paper_2609_32259_gb300 import pipeline
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


def _explicit(w, n_seg, n_terms):
    layers, weights = W.explicit_table(w.L_s, w.L_r, n_seg, n_terms, seed=3)
    return w.with_(layer_mode="explicit", seg_layer=layers, seg_w=weights)


L = lambda T, **kw: W.llama_to_ministral(T).with_(L_s=4, L_r=3, **kw)
BATCH = W.qwen25_to_llama_batched(n_req=3, lo=30, hi=400, seed=5).with_(L_s=4, L_r=3)
CASES = {
    "interp_one_token": (L(1, layer_mode="interp"), {}),
    "interp_129": (L(129, layer_mode="interp"), {}),
    "interp_one_wide_tile": (L(600, H_r=4, layer_mode="interp"), {}),
    "pooled_one_wide_tile": (L(300, H_r=4, align_mode="overlap_mean"), dict(pool_before_map=True)),
    "interp_same_index": (L(517, layer_mode="interp", align_mode="same_index"), {}),
    "interp_overlap": (L(700, layer_mode="interp", align_mode="overlap_mean"), {}),
    "interp_round_once": (L(300, layer_mode="interp"), dict(round_built_operands=True)),
    "rotated": (L(700, sender_k_rotated=True, s_pos0=(37,)), {}),
    "rotated_head64_narrow": (L(300, H_s=2, D_s=64, H_r=1, sender_k_rotated=True), {}),
    "rotated_head16": (L(260, H_s=8, D_s=16, sender_k_rotated=True), {}),
    "rotated_round_once": (L(300, sender_k_rotated=True), dict(round_built_operands=True)),
    "rotated_interp": (L(300, sender_k_rotated=True, layer_mode="interp"), {}),
    "rotated_overlap": (L(300, sender_k_rotated=True, align_mode="overlap_mean"), {}),
    "rotated_spans_paged": (BATCH.with_(sender_k_rotated=True, span_gap=90, s_pos0=(0, 5, 900)), {}),
    "interp_spans_paged": (BATCH.with_(layer_mode="interp", span_gap=90), {}),
    "pooled_first": (L(400, align_mode="overlap_mean"), dict(pool_before_map=True)),
    "pooled_knorm": (L(400, align_mode="overlap_mean", knorm=True), {}),
    "weighted_8_segments": (_explicit(W.qwen25_to_llama_kv_ridge(300).with_(
        L_s=9, L_r=3, kv_ridge=False), 8, 2), {}),
    # 245 MB a layer: two layers of five at a time
    "rotated_in_groups": (W.llama_to_ministral(20000).with_(L_s=3, L_r=5, sender_k_rotated=True), {}),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_made_rows_equal_built_rows(name):
    w, opts = CASES[name]
    dev = torch.device("cuda")
    tok = W.tokens(w)
    sender = W.sender_kv(w, W.sender_cache_rows(w, tok), dev)
    Wm, b, r = W.maps(w, dev)
    paged = W.paged_layout(w, tok) if w.paged else None
    job = pipeline.job_from_workload(w, tok, sender, Wm, b, r, paged=paged, r_pos0=W.r_pos0(w),
                                     knorm_w=W.knorm_weight(w), device=dev, **opts)
    job.receiver.fill_(3.0)
    made_bytes = job.workspace.numel()
    job.step()
    torch.cuda.synchronize()
    assert job.device_status() == 0
    made = job.receiver.clone()
    # fp32 plans make no rows: their workspace is what a plan cannot do without
    f32, job.desc.c.dtype = job.desc.c.dtype, B.DTYPES["f32"]
    base = B.plan_workspace_size(job.desc)
    job.desc.c.dtype = f32
    assert base < made_bytes
    job.workspace = torch.empty(base, dtype=torch.uint8, device=dev)
    job.receiver.fill_(3.0)
    job.make_plan()
    job.transfer()
    torch.cuda.synchronize()
    assert job.device_status() == 0
    assert torch.equal(made, job.receiver)
    job.close()


def test_made_rows_on_two_streams():
    """The made rows lie in the plan's workspace: transfers of two caches with one
    plan on two streams must not take each other's."""
    w = L(3000, sender_k_rotated=True)
    dev = torch.device("cuda")
    tok = W.tokens(w)
    sender = W.sender_kv(w, tok.T_s, dev)
    other = sender.flip(2).contiguous()
    Wm, b, r = W.maps(w, dev)
    job = pipeline.job_from_workload(w, tok, sender, Wm, b, r, r_pos0=W.r_pos0(w), device=dev)
    job.step()
    senders, outs = [sender, other], [torch.empty_like(job.receiver) for _ in range(2)]
    want = [torch.empty_like(job.receiver) for _ in range(2)]
    for s, o in zip(senders, want):
        B.transfer(job.plan, s, o)
        torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for _ in range(20):
        for s, o, st in zip(senders, outs, streams):
            B.transfer(job.plan, s, o, st)
    torch.cuda.synchronize()
    assert job.device_status() == 0
    assert torch.equal(outs[0], want[0]) and torch.equal(outs[1], want[1])
    job.close()
