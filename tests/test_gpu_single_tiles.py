"""Short transfers on single-CTA tiles of 128 rows (up to 512 receiver tokens)
and their neighbours on pair tiles, against the oracle: one, exactly one and just
over one tile of distinct rows, several heads per tile, one head per tile."""

import pytest
import torch

from gpu_harness import Case
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


@pytest.mark.parametrize("T,heads,width,align,paged", [
    (1, 1, 128, "ta", False), (128, 4, 64, "same_index", False), (129, 3, 128, "same_index", True),
    (512, 8, 32, "ta", True), (512, 2, 128, "same_index", False), (513, 2, 128, "same_index", False),
    (300, 2, 256, "ta", False)])
def test_short_transfers(T, heads, width, align, paged):
    w = W.llama_to_ministral(T).with_(L_s=3, L_r=3, H_s=2, H_r=heads, D_r=width, align_mode=align,
                                      paged=paged, knorm=paged, r_pos0=(70,))
    c = Case(w, sentinel=5.0).run()
    c.check_csr()
    c.check_parity()
