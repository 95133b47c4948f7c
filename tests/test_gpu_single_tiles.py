"""Short transfers on single-CTA tiles of 128 rows and their neighbours on pair
tiles, against the oracle: one row, exactly one and just over one tile of distinct
rows, the last and the first token count of the rule, several heads per tile, one
head per tile, tiles of 128 columns.  Single tiles need more tiles than SM pairs
(twelve layers of four 256-column blocks)."""

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


@pytest.mark.parametrize("T,heads,width,align,paged,layers", [
    (1, 8, 128, "ta", False, 12), (128, 16, 64, "same_index", True, 12),
    (129, 8, 128, "same_index", False, 12), (400, 32, 32, "ta", True, 12),
    (401, 8, 128, "ta", False, 12), (300, 4, 256, "ta", False, 12), (100, 3, 128, "same_index", True, 13)])
def test_short_transfers_of_many_tiles(T, heads, width, align, paged, layers):
    w = W.llama_to_ministral(T).with_(L_s=3, L_r=layers, H_s=2, H_r=heads, D_r=width,
                                      align_mode=align, paged=paged, knorm=paged, r_pos0=(70,))
    c = Case(w, sentinel=5.0).run()
    c.check_parity()


def test_more_rows_than_expected():
    """Sender tokens of one character make every row distinct, where Token Alignment
    is expected to share a quarter: four blocks of rows on single CTAs."""
    c = Case(W.llama_to_ministral(400).with_(L_s=3, L_r=12, H_s=2, mean_s=1.0), sentinel=5.0).run()
    assert c.job.distinct_rows() > 384
    c.check_parity()

