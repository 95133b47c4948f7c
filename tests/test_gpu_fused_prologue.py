"""The one-launch alignment and plan (up to 32,768 tokens and 64 requests)
against the passes that longer batches take: empty requests appended to a
batch take it past the 64 and change nothing else, so every result must agree
bit for bit."""

import numpy as np
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


def _results(w, extra, **opts):
    n = len(w.r_tokens)
    if extra:
        pos = lambda p: None if p is None else tuple(p) + (0,) * extra
        w = w.with_(r_tokens=w.r_tokens + (0,) * extra, r_pos0=pos(w.r_pos0), s_pos0=pos(w.s_pos0))
    tok = W.tokens(w)
    dev = torch.device("cuda")
    sender = W.sender_kv(w.with_(r_tokens=w.r_tokens[:n]), W.sender_cache_rows(w, tok), dev)
    Wm, b, r = W.maps(w, dev)
    paged = W.paged_layout(w, tok) if w.paged else None
    rows = paged.n_blocks * w.block_size if w.paged else tok.T_r
    receiver = torch.full((w.L_r, 2, rows, w.d_r), 7.0, dtype=w.torch_dtype, device=dev)
    job = pipeline.job_from_workload(w, tok, sender, Wm, b, r, paged=paged, r_pos0=W.r_pos0(w),
                                     device=dev, receiver=receiver, **opts)
    job.step()
    torch.cuda.synchronize()
    out = (*job.csr(), job.align_status(), job.device_status(), job.distinct_rows(),
           job.receiver.cpu())
    job.close()
    return out


# one CTA up to 1,024 tokens on the longer side (here the receiver's), eight above,
# four rows a thread above 8,192, the passes above 32,768; requests that start and end
# inside one thread's rows
SIZES = [(1,), (1024,), (1025,), (300, 1, 2, 500), (4093,), (4097,), (8192,), (8193,), (32760,),
         (32768,), (130, 1, 5000), (3, 1, 9000, 2, 1, 1, 3, 700, 1, 2), tuple([37] * 64)]
FORMS = {
    "ta": {}, "ta_paged": dict(paged=True), "ta_span": dict(span_gap=11),
    "ta_rotated": dict(sender_k_rotated=True), "same_index": dict(align_mode="same_index"),
    "overlap": dict(align_mode="overlap_mean"),
    "overlap_paged_span": dict(align_mode="overlap_mean", paged=True, span_gap=5),
}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("sizes", SIZES, ids=lambda s: f"{len(s)}x{max(s)}")
def test_one_launch_equals_the_passes(sizes, form):
    w = W.llama_to_ministral(1).with_(L_s=2, L_r=2, H_s=1, H_r=1, r_tokens=sizes, seed=len(sizes),
                                      r_pos0=tuple(3 * q for q in range(len(sizes))),
                                      s_pos0=tuple(q for q in range(len(sizes))), **FORMS[form])
    a, b = _results(w, 0), _results(w, 70 - min(len(sizes), 6))
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)
    assert a[3:6] == b[3:6]
    assert torch.equal(a[6], b[6])


def test_layers_past_the_small_table():
    """More than 48 receiver layers: the larger parameter table."""
    w = W.llama_to_ministral(300).with_(L_s=3, L_r=70, H_s=1, H_r=1)
    a, b = _results(w, 0), _results(w, 70)
    assert torch.equal(a[6], b[6]) and a[3:6] == b[3:6]


@pytest.mark.parametrize("mode", ["ta", "overlap_mean"])
@pytest.mark.parametrize("extra", [0, 70])
def test_bad_offsets_are_flagged_on_both_paths(mode, extra):
    s_end = np.arange(1, 6001, dtype=np.int32)
    r_end = np.arange(1, 6001, dtype=np.int32)
    s_end[4500] = s_end[4499]  # not increasing, in the cluster's second half
    ptr = np.array([0] + [6000] * (1 + extra), np.int32)
    d = lambda a: torch.as_tensor(a).cuda()
    row_ptr = torch.zeros(6001, dtype=torch.int32, device="cuda")
    col = torch.zeros(12000, dtype=torch.int32, device="cuda")
    wt = torch.zeros(12000, device="cuda")
    info = torch.full((2,), 99, dtype=torch.int32, device="cuda")
    B.align_build(mode, ptr, ptr, d(s_end), d(r_end), row_ptr, col, wt, 12000, info)
    assert int(info[1]) & 0x01
    c = col[:int(info[0])]
    assert int(c.min()) >= 0 and int(c.max()) < 6000
