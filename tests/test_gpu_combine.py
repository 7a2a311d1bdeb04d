"""The merge of the forward's partial records (combine_kernels.cu) at the edges of its block
shapes: 8, 16 or 32 rows per block by the anchor size, whole anchors per block, the last block
partly filled, and the large-batch shape of 32 rows, for the full-vocabulary forward, the label
readout and the top-k forward, against the oracle."""

import numpy as np
import pytest
import torch

from oracle import alr_oracle as orc
from paper_2609_38795_gb300 import alr, build_lib, synthetic
from tests import parity as P
from tests import test_gpu_topk as T

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    build_lib.build()
    alr.lib()
    assert alr.alr_device_supported() == alr.ALR_OK, alr.alr_last_error()


# (A, B): one row; a partial 8-row block; anchors of 3 and 8 in 8 rows; 9 and 16 in 16; 17 and
# 32 in 32; many blocks of 30 and of 32 rows; the last shapes with a block per SM on 152 SMs (15 rows
# each, 8 rows each) and the first beyond; the two sides of the readout's choices of lanes per row
SHAPES = [(1, 1), (13, 1), (5, 3), (3, 8), (3, 9), (7, 16), (4, 17), (3, 32), (606, 15),
          (607, 15), (9729, 1), (1023, 1), (1024, 1), (152, 15), (153, 15), (1216, 1), (1217, 1),
          (4865, 1)]


@pytest.mark.parametrize("mode", [alr.ALR_MODE_ERASE_SOFT, alr.ALR_MODE_ERASE_HARD])
@pytest.mark.parametrize("A,B", SHAPES)
def test_forward_merge(A, B, mode):
    """V = 520 fills two vocabulary tiles and 8 columns of a third, so some records are empty."""
    d, V = 64, 520
    b = synthetic.slot_batch(d, V, A, B, 0.5, dtype=torch.bfloat16, device="cuda", seed=A + B)
    b = synthetic.sharpen(b)
    N = A * B
    g = torch.Generator(device="cuda").manual_seed(A)
    mask = (torch.rand(N, generator=g, device="cuda") < 0.9).float()
    mask[0] = 1.0
    greedy = (b["Ht"].float() @ b["W"].float()).argmax(1).to(torch.int32)
    rep, rnd = synthetic.corpus_replacement(N, V, 0.2, device="cuda", seed=A)
    tok = synthetic.corpus_tokens(greedy, rep, rnd)
    sl = P.gpu_forward(b["Hd"], b["Ht"], b["W"], B, mode=mode, row_mask=mask, corpus_tok=tok)
    r = orc.slot_loss_forward(P.np64(b["Hd"]), P.np64(b["Ht"]), P.np64(b["W"]), B, mode=mode,
                              row_mask=P.np64(mask), corpus_tok=P.npi(tok))
    got = P.fwd_to_numpy(sl)
    if mode == alr.ALR_MODE_ERASE_HARD:
        # a hard gate hangs on the greedy token: anchors with a near-tied target row may differ
        near = (r["gap_t"] < P.NEAR_TIE).reshape(A, B).any(1)
        keep = np.repeat(~near, B)
        np.testing.assert_allclose(got["weight"][keep], r["weight"][keep], rtol=1e-5, atol=0)
        assert np.all(P.rel_err(got["loss_row"], r["loss_row"]) <= P.LOSS_RTOL)
    else:
        P.compare_forward(got, r, mode=mode)
    # the batch sums are the fp32 values of fp64 sums of the row results themselves: 2^-24
    # relative for the final rounding, and as much again for the weights' own rounding
    w, l = got["weight"], got["loss_row"]
    np.testing.assert_allclose(got["weight_sum"], w.sum(), rtol=2.0 ** -23)
    np.testing.assert_allclose(got["loss_total"], (w * l).sum() / w.sum(), rtol=2.0 ** -22)
    assert alr.alr_device_status() == alr.ALR_OK


@pytest.mark.parametrize("A,B", SHAPES)
def test_readout_and_topk_merge(A, B):
    d, V = 64, 520
    b = synthetic.sharpen(synthetic.slot_batch(d, V, A, B, 0.5, dtype=torch.bfloat16,
                                               device="cuda", seed=31 * A + B))
    z = orc.label_readout(P.np64(b["Ht"]), P.np64(b["W"]), k=T.K)
    g = T.gpu_readout(b["Ht"], b["W"], B)
    T.compare_readout(g, z)
    lab = dict(idx=g["top_idx"], prob=g["top_prob"], tail=g["tail"])
    labels = T.host_labels(lab)
    _, out = T.gpu_topk_forward(b["Hd"], b["W"], B, lab)
    zd = P.np64(b["Hd"]) @ P.np64(b["W"])
    lse = np.log(np.exp(zd - zd.max(1, keepdims=True)).sum(1)) + zd.max(1)
    rows = np.arange(A * B)[:, None]
    q = np.exp(zd[rows, labels[0]] - lse[:, None])
    rest = np.exp(zd - lse[:, None])
    rest[rows, labels[0]] = 0.0
    loss = -(labels[1] * np.log(q)).sum(1) - labels[2] * np.log(rest.sum(1))
    np.testing.assert_allclose(P.np64(out["lse_d"]), lse, rtol=2e-4)
    np.testing.assert_allclose(P.np64(out["tail_q"]), rest.sum(1), rtol=1e-3)
    assert P.rel_err(P.np64(out["loss_row"]), loss).max() <= P.LOSS_RTOL
    w, l = P.np64(out["weight"]), P.np64(out["loss_row"])
    np.testing.assert_allclose(float(out["weight_sum"].item()), w.sum(), rtol=2.0 ** -23)
    np.testing.assert_allclose(float(out["loss_total"].item()), (w * l).sum() / w.sum(),
                               rtol=2.0 ** -22)
    assert alr.alr_device_status() == alr.ALR_OK


@pytest.mark.parametrize("N", [1104, 2080])
def test_forward_at_uneven_row_blocks(N):
    """9 and 17 row blocks: the split count and the raster groups (9 + 8) that fill the SMs."""
    B, d, V = 16, 64, 20000
    b = synthetic.sharpen(synthetic.slot_batch(d, V, N // B, B, 0.5, dtype=torch.bfloat16,
                                               device="cuda", seed=N))
    r = orc.slot_loss_forward(P.np64(b["Hd"]), P.np64(b["Ht"]), P.np64(b["W"]), B)
    P.compare_forward(P.fwd_to_numpy(P.gpu_forward(b["Hd"], b["Ht"], b["W"], B)), r)
    z = orc.label_readout(P.np64(b["Ht"]), P.np64(b["W"]), k=T.K)
    T.compare_readout(T.gpu_readout(b["Ht"], b["W"], B), z)
    assert alr.alr_device_status() == alr.ALR_OK


@pytest.mark.parametrize("N,d,V", [(192, 320, 1400), (512, 256, 60000), (2000, 704, 20000)])
def test_sums_keep_their_precision_at_large_logits(N, d, V):
    """What the running sums and their merge lose, apart from the products: hidden states of -1, 0
    and 1 and head weights in steps of 2^-8 make every logit exact in fp32 in any order of
    summation (below 2^20 steps), with row maxima of 20 to 40.  Tiles of 128 and of 256 columns.

    A result is rounded once (2^-24).  Its sums take one rounded exponent and one ex2.approx
    (2^-22 at most, 2^-24 rms) per column, whose errors average out over the few columns that
    matter: 2^-23 rms is left for a loss or an entropy, 2^-24 for log S (relative to its
    size, about 30).  Terms summed against an earlier maximum that keep its exponent's
    residual (2^-25 of 40 log2 e, 1.7e-6) do not average out: they gave 1.5e-7 to 3e-7."""
    g = torch.Generator(device="cuda").manual_seed(N)
    w = torch.randn(d, V, device="cuda", generator=g) * (20.0 / d ** 0.5)
    W = (torch.clamp(torch.round(w * 256), -255, 255) / 256).to(torch.bfloat16)
    draw = lambda: ((torch.rand(N, d, device="cuda", generator=g) < 0.25).float()  # noqa: E731
                    * torch.randn(N, d, device="cuda", generator=g).sign()).to(torch.bfloat16)
    Ht = draw()
    Hd = torch.where(torch.rand(N, d, device="cuda", generator=g) < 0.2, draw(), Ht)
    zd, zt = Hd.double() @ W.double(), Ht.double() @ W.double()
    lse_d, lse_t = zd.logsumexp(1), zt.logsumexp(1)
    p = (zt - lse_t[:, None]).exp()
    ref = dict(loss_row=lse_d - (p * zd).sum(1), ent_row=lse_t - (p * zt).sum(1), lse_d=lse_d,
               lse_t=lse_t)
    assert lse_d.min() > 15.0
    out = P.gpu_forward(Hd, Ht, W, 16 if N % 16 == 0 else 8).out
    lab = T.gpu_readout(Ht, W, 16 if N % 16 == 0 else 8)
    ref["top_prob"] = p.gather(1, lab["top_idx"].long())
    # the tail is S minus the eight largest terms over S: no term of S is off by more than 2^-21 of
    # itself (its exponent's rounding and ex2.approx), so neither is the tail by more than that of 1
    tail = p.scatter(1, lab["top_idx"].long(), 0.0).sum(1)
    assert float((lab["tail"].double() - tail).abs().max()) <= 2.0 ** -21
    for k, x in ref.items():
        got = (lab if k == "top_prob" else out)[k].double()
        err = float((got - x).norm() / x.norm())
        print(N, k, err)
        assert err <= 2.0 ** (-24 if k in ("lse_d", "lse_t", "top_prob") else -23), (k, err)
    assert alr.alr_device_status() == alr.ALR_OK


def test_forward_workspace_stays_within_the_fixed_scratch():
    """Every bf16 problem whose records at 19 splits (15 fp32 fields per row, split and
    64-column group: what the no-workspace forward's limit was set for) fit the fixed 64 MiB
    still fits, whatever split count its row blocks take."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    limit = 64 << 20
    up = lambda x: (x + 1023) // 1024 * 1024  # noqa: E731
    for N in list(range(16, 4096, 112)) + list(range(4096, 16000, 592)) + list(range(16000, 120000, 4112)):
        for d, V in ((64, 200), (64, 1000), (256, 8000), (1000, 60000), (4096, 151936)):
            n_vt, rb = (V + 255) // 256, (N + 127) // 128
            vs = min(n_vt, max(1, sms // min(rb, 8)))
            start = up(15 * 4 * vs * 4 * N) + up(16 * (N // 16))
            need = alr.alr_fwd_workspace_size(alr.make_params(N, d, V, 16))
            assert 0 < need <= max(limit, start), (N, d, V, need, start)


@pytest.mark.parametrize("B", [1, 15, 32])
@pytest.mark.parametrize("A", [1, 2, 31, 256, 257])
def test_accept_len_block_edges(A, B):
    """One block up to 256 anchors (1, 2, 31 and 32 warps), one warp per anchor of many past it."""
    g = torch.Generator(device="cuda").manual_seed(A + B)
    t = torch.randint(0, 50, (A * B,), generator=g, device="cuda", dtype=torch.int32)
    same = torch.rand(A * B, generator=g, device="cuda") < 0.8
    d = torch.where(same, t, t + 1)
    active = (torch.rand(A * B, generator=g, device="cuda") < 0.95).float()
    acc = torch.full((A,), -1, dtype=torch.int32, device="cuda")
    hist = torch.full((B + 1,), -1, dtype=torch.int64, device="cuda")
    for w in (active, None):
        alr.alr_accept_len(d, t, B, acc, hist, active=w)
        torch.cuda.synchronize()
        ok = same if w is None else same & (w > 0)
        want = ok.view(A, B).int().cumprod(1).sum(1)
        assert torch.equal(acc, want.to(torch.int32))
        assert torch.equal(hist, torch.bincount(want, minlength=B + 1))
