"""IRA block construction on the GPU against the oracle, bit for bit (Sec. 3.2, In-rollout
anchors; App. A): the anchor and offset draws from given random integers, the block plan they
drive, and the secondary blocks' context rows (the primaries' stored five-layer rollout
features of y*_1..y*_{j-1}) at the paper's sequence length and stored-row count."""

import numpy as np
import pytest
import torch

from oracle import alr_oracle as orc
from paper_2609_38795_gb300 import alr, build_lib
from tests import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    build_lib.build()
    alr.lib()
    assert alr.alr_device_supported() == alr.ALR_OK, alr.alr_last_error()


def _u32(t):
    """The uint32 values an int32 tensor holds."""
    return t.cpu().numpy().view(np.uint32).astype(np.int64)


def _draws(S, L, K, max_b, density, seed):
    g = torch.Generator().manual_seed(seed)
    ok = (torch.rand(S, L, generator=g) < torch.tensor(density)[:, None]).to(torch.uint8)
    keys = torch.randint(-(1 << 31), 1 << 31, (S, L), generator=g, dtype=torch.int64).to(torch.int32)
    keys[0, :64] = 7                                      # equal keys: position order decides
    off_u = torch.randint(-(1 << 31), 1 << 31, (S, max_b // 2), generator=g,
                          dtype=torch.int64).to(torch.int32)
    out = dict(n_valid=torch.empty(S, dtype=torch.int32, device="cuda"),
               anchor_pos=torch.empty(S, max_b, dtype=torch.int32, device="cuda"),
               offsets=torch.empty(S, max_b // 2, dtype=torch.int32, device="cuda"))
    alr.alr_ira_draw(K, max_b, ok.cuda(), keys.cuda(), off_u.cuda(), out)
    torch.cuda.synchronize()
    ref = orc.ira_draw(ok.numpy(), _u32(keys), _u32(off_u), K, max_b)
    return out, ref, ok


@pytest.mark.parametrize("L", [1, 700, 4096])
def test_ira_draw_bit_exact(L):
    """Samples with no, few, exactly 128 and many valid positions; one with ties among keys."""
    K, max_b = 15, 128
    density = [0.0, 0.02, 128.5 / max(L, 1), 0.5, 1.0]
    out, (n_valid, anchor_pos, offsets), _ = _draws(5, L, K, max_b, density, seed=L)
    assert np.array_equal(P.npi(out["n_valid"]), n_valid)
    assert np.array_equal(P.npi(out["anchor_pos"]), anchor_pos)
    assert np.array_equal(P.npi(out["offsets"]), offsets)
    assert alr.alr_device_status() == alr.ALR_OK


def test_ira_plan_and_context_bit_exact():
    """Draws -> block plan -> context rows, at the paper's sequence length (4096), 128 anchors,
    K = 15 and 13 stored rows of five layers' features (d = 64 here), bf16; primary rollouts
    that end early, including one that ends before its secondary's offset."""
    S, L, K, max_b, C, layers, d = 6, 4096, 15, 128, 13, 5, 64
    Pn, H, F = max_b - max_b // 2, max_b // 2, layers * d
    out, (n_valid, anchor_pos, offsets), _ = _draws(S, L, K, max_b, [0.9, 0.01, 0.3, 0.05, 0.6, 0.02],
                                                   seed=9)
    g = torch.Generator().manual_seed(10)
    rlen = torch.full((S * Pn,), K, dtype=torch.int32)
    rlen[torch.randint(0, S * Pn, (40,), generator=g)] = torch.randint(1, K, (40,), generator=g,
                                                                        dtype=torch.int32)
    store = torch.randn(S * Pn, C, F, generator=g).to(torch.bfloat16)
    ctx = torch.full((S, H, C, F), 7.0, dtype=torch.bfloat16, device="cuda")
    ctx_len = torch.full((S, H), -5, dtype=torch.int32, device="cuda")
    prefix_end = torch.full((S, H), -5, dtype=torch.int32, device="cuda")
    alr.alr_ira_context(K, max_b, store.cuda(), out["n_valid"], rlen.cuda(), out["offsets"],
                        out["anchor_pos"], ctx, ctx_len, prefix_end)
    # the block plan from the same draws
    T = S * max_b
    plan = {k: torch.empty(T, dtype=torch.int32, device="cuda")
            for k in ("seq", "pos", "valid_len", "ctx_len")}
    alr.alr_ira_blocks(K, max_b, out["n_valid"], rlen.cuda(), out["offsets"], plan)
    torch.cuda.synchronize()
    c_ref, cl_ref, pe_ref = orc.ira_context(store.float().numpy(), n_valid, rlen.numpy().reshape(S, Pn),
                                            offsets, anchor_pos, K, max_b)
    assert torch.equal(ctx.float().cpu(), torch.from_numpy(c_ref).float())
    assert np.array_equal(P.npi(ctx_len), cl_ref)
    assert np.array_equal(P.npi(prefix_end), pe_ref)
    ref = orc.ira_blocks(n_valid, rlen.numpy().reshape(S, Pn), offsets, K, max_b)
    for k in ("seq", "pos", "valid_len", "ctx_len"):
        assert np.array_equal(P.npi(plan[k]).reshape(S, max_b), ref[k]), k
    # the plan's secondaries and the context agree on which blocks exist
    sec = (P.npi(plan["seq"]).reshape(S, max_b) >= 0) & (P.npi(plan["pos"]).reshape(S, max_b) > 0)
    assert sec.sum() == (pe_ref >= 0).sum()
    assert (cl_ref > 0).sum() > 100 and (rlen.numpy() < K).any()
    assert alr.alr_device_status() == alr.ALR_OK


# key patterns of the draw's radix select: the bits that tell keys apart sit in the digit that
# decides (32 - bits low bits vary), 0: all keys equal, so positions decide
@pytest.mark.parametrize("bits", [0, 3, 8, 14, 20, 32])
@pytest.mark.parametrize("L,max_b", [(40, 64), (1025, 1), (4096, 128), (16384, 7),
                                     (16384, 4000)])
def test_ira_draw_select_digits(L, max_b, bits):
    """Draws whose m-th smallest key shares 0 to 4 leading digits with the others, at 1 to 16
    positions per thread and with every valid position drawn, against the oracle bit for bit."""
    S, K = 3, 15
    g = torch.Generator().manual_seed(L + bits)
    ok = (torch.rand(S, L, generator=g) < torch.tensor([0.3, 0.9, 1.0])[:, None]).to(torch.uint8)
    low = torch.randint(0, 1 << bits, (S, L), generator=g, dtype=torch.int64)
    keys = (low - (1 << 31 if bits == 32 else 0)).to(torch.int32)
    if bits < 32:
        keys[1] ^= 0x5A5A5A5A                             # the same spread over other digit values
    off_u = torch.zeros(S, max(max_b // 2, 1), dtype=torch.int32)[:, :max_b // 2].contiguous()
    out = dict(n_valid=torch.empty(S, dtype=torch.int32, device="cuda"),
               anchor_pos=torch.full((S, max_b), -7, dtype=torch.int32, device="cuda"),
               offsets=torch.empty(S, max_b // 2, dtype=torch.int32, device="cuda"))
    alr.alr_ira_draw(K, max_b, ok.cuda(), keys.cuda(), off_u.cuda(), out)
    torch.cuda.synchronize()
    n_valid, anchor_pos, _ = orc.ira_draw(ok.numpy(), _u32(keys), _u32(off_u), K, max_b)
    assert np.array_equal(P.npi(out["n_valid"]), n_valid)
    assert np.array_equal(P.npi(out["anchor_pos"]), anchor_pos)


def test_chained_calls_read_what_the_call_before_wrote():
    """draw -> context, and draw -> plan -> label gather, issued back to back without a
    synchronisation, each call overlapping the end of the one before, over the same buffers with
    other keys, masks and offsets every round: each round's rows, bit for bit, against the
    oracle.  Stale draws or plans of the round before would move whole rows."""
    S, L, K, max_b, C, F, d, rounds = 5, 600, 15, 64, 13, 64, 32, 24
    Pn, H = max_b - max_b // 2, max_b // 2
    g = torch.Generator().manual_seed(77)
    u32 = lambda *s: torch.randint(-(1 << 31), 1 << 31, s, generator=g,  # noqa: E731
                                   dtype=torch.int64).to(torch.int32)
    i32 = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")  # noqa: E731
    store = torch.randn(S * Pn, C, F, generator=g).to(torch.bfloat16)
    labels = torch.randn(S * Pn, K, d, generator=g).to(torch.bfloat16)
    rlen = torch.randint(1, K + 1, (S * Pn,), generator=g, dtype=torch.int32)
    store_c, labels_c, rlen_c = store.cuda(), labels.cuda(), rlen.cuda()
    ins, dev = [], []
    for _ in range(rounds):
        density = torch.rand(S, 1, generator=g) * 0.3
        ins.append(((torch.rand(S, L, generator=g) < density).to(torch.uint8), u32(S, L), u32(S, H)))
        dev.append([x.cuda() for x in ins[-1]])
    out = dict(n_valid=i32(S), anchor_pos=i32(S, max_b), offsets=i32(S, H))
    plan = {k: i32(S * max_b) for k in ("seq", "pos", "valid_len")}
    new = lambda *s: [torch.empty(*s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
                      for _ in range(rounds)]
    ctx, rows = new(S, H, C, F), new(S * max_b * K, d)
    row_valid = [torch.empty(S * max_b * K, device="cuda") for _ in range(rounds)]
    ctx_len, prefix_end = [[i32(S, H) for _ in range(rounds)] for _ in range(2)]
    torch.cuda.synchronize()
    for i, (ok, keys, off_u) in enumerate(dev):
        alr.alr_ira_draw(K, max_b, ok, keys, off_u, out)
        alr.alr_ira_context(K, max_b, store_c, out["n_valid"], rlen_c, out["offsets"],
                            out["anchor_pos"], ctx[i], ctx_len[i], prefix_end[i])
        alr.alr_ira_draw(K, max_b, ok, keys, off_u, out)
        alr.alr_ira_blocks(K, max_b, out["n_valid"], rlen_c, out["offsets"], plan)
        alr.alr_gather_ira_blocks(labels_c, plan["seq"], plan["pos"], K, rows[i], row_valid[i],
                                  valid_len=plan["valid_len"])
    torch.cuda.synchronize()
    lens = rlen.numpy().reshape(S, Pn)
    for i, (ok, keys, off_u) in enumerate(ins):
        n_valid, anchor_pos, offsets = orc.ira_draw(ok.numpy(), _u32(keys), _u32(off_u), K, max_b)
        c, cl, pe = orc.ira_context(store.float().numpy(), n_valid, lens, offsets, anchor_pos, K,
                                    max_b)
        assert torch.equal(ctx[i].float().cpu(), torch.from_numpy(c).float()), i
        assert np.array_equal(P.npi(ctx_len[i]), cl) and np.array_equal(P.npi(prefix_end[i]), pe), i
        ref = orc.ira_blocks(n_valid, lens, offsets, K, max_b)
        seq, pos, vl = (ref[k].reshape(-1, 1) for k in ("seq", "pos", "valid_len"))
        at = pos + np.arange(K)
        live = (seq >= 0) & (at < np.minimum(vl, K))
        want = labels.float().numpy()[np.where(live, seq, 0), np.where(live, at, 0)]
        want[~live] = 0.0
        assert np.array_equal(rows[i].float().cpu().numpy().reshape(want.shape), want), i
        assert np.array_equal(row_valid[i].cpu().numpy().reshape(live.shape), live), i
    assert alr.alr_device_status() == alr.ALR_OK
