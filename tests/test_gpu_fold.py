"""hf_fold (Eq. 9 folding of the Eq. 7 correction) against the oracle's
fold, and the transfer through GPU-folded maps against the oracle's
unfused path (y0 + (y0 B) G applied at transfer time)."""

import numpy as np
import pytest
import torch

from gpu_harness import Case, MAX_ABS_TOL, REL_FRO_TOL, MapFetcher, RowFetcher
from oracle import heterofold_oracle as O
from paper_2609_32259_gb300 import binding as B
from paper_2609_32259_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g

    g.build()


def _factors(n_maps, d_R, rank, seed, dev, scale=0.5):
    g = torch.Generator(device="cpu").manual_seed(seed)
    Bm = torch.randn((n_maps, d_R, rank), generator=g) / np.sqrt(d_R)
    Gm = torch.randn((n_maps, rank, d_R), generator=g) * scale
    return Bm.to(dev), Gm.to(dev)


@pytest.mark.parametrize("dtype,in_place", [("bf16", False), ("bf16", True), ("f32", False)])
def test_fold_matches_oracle(dtype, in_place):
    dev = torch.device("cuda")
    n_maps, d_R, K, rank = 3, 256, 384, 16
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cpu").manual_seed(5)
    Wm = (torch.randn((n_maps, d_R, K), generator=g) / np.sqrt(K)).to(tdt).to(dev)
    b = (torch.randn((n_maps, d_R), generator=g) * 0.1).to(dev)
    Bm, Gm = _factors(n_maps, d_R, rank, 6, dev)
    W0 = Wm.double().cpu().numpy()
    b0 = b.double().cpu().numpy()
    Wf = Wm if in_place else torch.empty_like(Wm)
    bf = b if in_place else torch.empty_like(b)
    B.fold(dtype, Wm, b, Bm, Gm, Wf, bf)
    torch.cuda.synchronize()
    rel = 2.0 ** -8 if dtype == "bf16" else 1e-5
    for m in range(n_maps):
        Af, bref = O.fold(W0[m].T, b0[m], Bm[m].double().cpu().numpy(),
                          Gm[m].double().cpu().numpy())
        got = Wf[m].double().cpu().numpy()
        assert np.all(np.abs(got - Af.T) <= rel * np.abs(Af.T) + 1e-6), m
        assert np.allclose(bf[m].double().cpu().numpy(), bref, rtol=1e-5, atol=1e-6), m


# The tensor-core form: one row and one column group to its largest d_R, rows
# that no warp's 16 divide, a ragged last unit of columns, padded ranks, more
# units than SMs; a d_R, a K and a rank past it (the other form).
@pytest.mark.parametrize("n_maps,d_R,K,rank", [
    (1, 1, 8, 4), (3, 270, 40, 8), (2, 1024, 104, 16), (1, 1008, 3080, 16), (9, 128, 1024, 16),
    (1, 1040, 64, 16), (2, 64, 36, 16), (2, 64, 64, 32),
    # both sides of the rule: one round of units, and several for one to four blocks of rows
    (1, 191, 4096, 4), (1, 192, 4096, 4), (1, 192, 4904, 4), (9, 191, 1024, 16), (9, 192, 1024, 16),
    (5, 287, 2000, 16), (5, 288, 2000, 16), (3, 768, 2056, 8), (3, 880, 2056, 8), (3, 879, 2056, 8)])
def test_fold_bf16_units(n_maps, d_R, K, rank):
    dev = torch.device("cuda")
    g = torch.Generator(device="cpu").manual_seed(d_R + K)
    Wm = (torch.randn((n_maps, d_R, K), generator=g) / np.sqrt(K)).to(torch.bfloat16).to(dev)
    b = (torch.randn((n_maps, d_R), generator=g) * 0.1).to(dev)
    Bm, Gm = _factors(n_maps, d_R, rank, 6, dev)
    Wf, bf = Wm.clone(), b.clone()
    B.fold("bf16", Wf, bf, Bm, Gm, Wf, bf)   # in place
    for m in range(n_maps):
        Af, bref = O.fold(Wm[m].double().cpu().numpy().T, b[m].double().cpu().numpy(),
                          Bm[m].double().cpu().numpy(), Gm[m].double().cpu().numpy())
        got = Wf[m].double().cpu().numpy()
        # one rounding to bf16 (2^-9 of the value) and fp32 sums
        assert np.all(np.abs(got - Af.T) <= 2.0 ** -8 * np.abs(Af.T) + 1e-6), m
        assert np.allclose(bf[m].double().cpu().numpy(), bref, rtol=1e-5, atol=1e-6), m


def test_transfer_with_folded_maps_matches_unfused_oracle():
    w = W.llama_to_ministral(600).with_(L_s=4, L_r=3)
    c = Case(w)
    dev = c.dev
    n_maps = w.L_r * 2
    rank = 16
    W_orig = c.Wm.clone()
    b_orig = c.b.clone()
    Bm, Gm = _factors(n_maps, w.d_r, rank, 7, dev, scale=0.06)
    Wflat = c.Wm.view(n_maps, w.d_r, w.K)
    bflat = c.b.view(n_maps, w.d_r)
    B.fold("bf16", Wflat, bflat, Bm, Gm, Wflat, bflat)   # in place: the job's maps
    c.run()
    assert c.job.device_status() == 0
    Bn = Bm.double().cpu().numpy().reshape(w.L_r, 2, w.d_r, rank)
    Gn = Gm.double().cpu().numpy().reshape(w.L_r, 2, rank, w.d_r)
    ref = O.transfer_unfused(RowFetcher(c.sender), c.csr, c.segs, MapFetcher(W_orig),
                             b_orig.cpu().numpy(), c.r, Bn, Gn, H_r=w.H_r, D_r=w.D_r,
                             pos=c.pos, inv_freq_r=c.inv_freq_r)
    for (l, cc), y in ref.items():
        gpu = c.gpu_rows(l, cc, np.arange(c.tok.T_r))
        diff = gpu - y
        rel = float(np.linalg.norm(diff) / np.linalg.norm(y))
        assert rel <= REL_FRO_TOL and float(np.abs(diff).max()) <= MAX_ABS_TOL, (l, cc, rel)
    # the correction matters: the unfolded maps give a clearly different cache
    plain = O.transfer(RowFetcher(c.sender), c.csr, c.segs, MapFetcher(W_orig),
                       b_orig.cpu().numpy(), c.r, H_r=w.H_r, D_r=w.D_r, pos=c.pos,
                       inv_freq_r=c.inv_freq_r, layers=[0], roles=(1,))
    d = plain[(0, 1)] - ref[(0, 1)]
    assert np.linalg.norm(d) > 0.1 * np.linalg.norm(ref[(0, 1)])


def test_fold_ragged_tile_and_bad_arguments():
    dev = torch.device("cuda")
    g = torch.Generator(device="cpu").manual_seed(9)
    Wm = (torch.randn((2, 40, 70), generator=g) * 0.1).to(dev)   # K = 70: a ragged last tile
    b = torch.randn((2, 40), generator=g).to(dev)
    Bm, Gm = _factors(2, 40, 8, 10, dev)
    Wf = torch.empty_like(Wm)
    bf = torch.empty_like(b)
    B.fold("f32", Wm, b, Bm, Gm, Wf, bf)
    torch.cuda.synchronize()
    for m in range(2):
        Af, _ = O.fold(Wm[m].double().cpu().numpy().T, b[m].double().cpu().numpy(),
                       Bm[m].double().cpu().numpy(), Gm[m].double().cpu().numpy())
        assert np.allclose(Wf[m].double().cpu().numpy(), Af.T, rtol=1e-5, atol=1e-6)
    Bm6 = torch.zeros((2, 40, 6), device=dev)
    Gm6 = torch.zeros((2, 6, 40), device=dev)
    with pytest.raises(B.HFError) as e:
        B.fold("f32", Wm, b, Bm6, Gm6, Wf, bf)               # rank not a multiple of 4
    assert e.value.status == B.HF_ERR_UNSUPPORTED


def test_fold_infinity_stays_in_its_column():
    """Rows past d_R (1,000 of 1,024) are padding of the tensor-core form: what an
    infinity makes of its column reaches no other column and no later unit."""
    dev = torch.device("cuda")
    n_maps, d_R, K, rank = 2, 1000, 160 * 152, 8
    g = torch.Generator(device="cpu").manual_seed(9)
    Wm = (torch.randn((n_maps, d_R, K), generator=g) / np.sqrt(K)).to(torch.bfloat16).to(dev)
    b = torch.zeros((n_maps, d_R), device=dev)
    Bm, Gm = _factors(n_maps, d_R, rank, 6, dev)
    clean, bf = torch.empty_like(Wm), torch.empty_like(b)
    B.fold("bf16", Wm, b, Bm, Gm, clean, bf)
    cols = torch.arange(0, K, 160, device=dev)
    Wm[:, 3, cols] = float("inf")
    got = torch.empty_like(Wm)
    B.fold("bf16", Wm, b, Bm, Gm, got, bf)
    torch.cuda.synchronize()
    assert not torch.isfinite(got[:, 3, cols]).any()
    got[:, :, cols] = clean[:, :, cols]
    assert torch.equal(got, clean)


@pytest.mark.parametrize("d_R,rank,K,in_place", [
    (1000, 8, 6088, True), (256, 16, 6088, False), (300, 16, 6088, True), (270, 4, 1288, False)])
def test_fold_keeps_infinities(d_R, rank, K, in_place):
    """Infinities and NaN of W, factors that are exact in bf16 (whose residual parts
    are zero) and factors that overflow bf16: the tensor-core form gives infinities,
    NaN and finite values where the fp32 form does."""
    dev = torch.device("cuda")
    n_maps = 3  # a last strip of eight columns each
    g = torch.Generator(device="cpu").manual_seed(d_R)
    Wm = (torch.randn((n_maps, d_R, K), generator=g) / np.sqrt(K)).to(torch.bfloat16)
    Bm, Gm = _factors(n_maps, d_R, rank, 6, "cpu")
    Bm[0, 3], Gm[0] = 0.5, Gm[0].abs()  # one sign: infinite, not NaN
    Bm[1, 3] = Bm[1, 3].to(torch.bfloat16).float()
    Bm[2, 5], Gm[2, 0, 7] = 3.4e38, 3.4e38  # infinite when rounded to bf16
    Wm[2, 5], Wm[2, :, ::3] = 2.0**-120, 2.0**-120
    for m in range(2):
        Wm[m, 3, 1::50] = float("inf")
        Wm[m, 3, 7::50] = -float("inf")
        Wm[m, d_R - 1, 11::50] = float("nan")
    Wm, Bm, Gm = Wm.to(dev), Bm.to(dev), Gm.to(dev)
    b = torch.zeros((n_maps, d_R), device=dev)
    got = Wm.clone() if in_place else torch.empty_like(Wm)
    plain, bf = torch.empty(Wm.shape, device=dev), torch.empty_like(b)
    B.fold("bf16", got if in_place else Wm, b, Bm, Gm, got, bf)
    B.fold("f32", Wm.float(), b, Bm, Gm, plain, bf)
    torch.cuda.synchronize()
    plain = plain.to(torch.bfloat16)
    assert torch.isposinf(got[0, :, 1::50]).all() and torch.isneginf(got[0, :, 7::50]).all()
    assert torch.equal(torch.isnan(got), torch.isnan(plain))
    inf = torch.isinf(plain)
    assert torch.equal(torch.isinf(got), inf) and torch.equal(got[inf], plain[inf])
    finite = torch.isfinite(plain)
    diff = (got[finite].double() - plain[finite].double()).abs()
    # both are rounded once: at most a bf16 ulp apart, beside the fp32 sums
    assert (diff <= 2.0**-7 * plain[finite].double().abs() + 1e-6).all()
