"""Pooling after the map: a window's sender rows follow one another and come by
tensor copies, unless the aligned tokens are spans of a longer cache, whose rows
the loader warps copy one by one.  The same tokens either way must give the same
caches bit for bit, at the ends of windows, of 32-row copies and of the cache."""

import numpy as np
import pytest
import torch

from paper_2609_32259_gb300 import pipeline
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


L = lambda T, **kw: W.llama_to_ministral(T).with_(L_s=4, L_r=3, align_mode="overlap_mean", **kw)
CASES = {
    "one_token": L(1),
    "within_a_slab": L(29),
    "slab": L(32),
    "window": L(128),
    "window_and_one": L(131),
    "three_windows": L(390),
    "knorm": L(200, knorm=True),
    "narrow": L(300, H_s=1, D_s=64, H_r=1),
    "requests": W.qwen25_to_llama_batched(n_req=3, lo=30, hi=400, seed=5).with_(
        L_s=4, L_r=3, align_mode="overlap_mean"),
}


def _receiver(w, tok, sender):
    dev = torch.device("cuda")
    Wm, b, r = W.maps(w, dev)
    paged = W.paged_layout(w, tok) if w.paged else None
    job = pipeline.job_from_workload(w, tok, sender, Wm, b, r, paged=paged, r_pos0=W.r_pos0(w),
                                     knorm_w=W.knorm_weight(w), device=dev)
    job.receiver.fill_(3.0)
    job.step()
    torch.cuda.synchronize()
    assert job.device_status() == 0
    out = job.receiver.clone()
    job.close()
    return out


@pytest.mark.parametrize("name", sorted(CASES))
def test_window_rows_equal_span_rows(name):
    w = CASES[name]
    dev = torch.device("cuda")
    tok = W.tokens(w)
    sender = W.sender_kv(w, tok.T_s, dev)
    ws = w.with_(span_gap=3)
    row0, rows = W.span_layout(ws, tok)
    ptr = np.asarray(tok.s_tok_ptr)
    spans = torch.full((*sender.shape[:2], rows, sender.shape[3]), float("nan"),
                       dtype=sender.dtype, device=dev)
    for q, r0 in enumerate(row0):
        n = int(ptr[q + 1] - ptr[q])
        spans[:, :, int(r0):int(r0) + n] = sender[:, :, int(ptr[q]):int(ptr[q + 1])]
    assert torch.equal(_receiver(w, tok, sender), _receiver(ws, tok, spans))
