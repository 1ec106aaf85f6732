"""Parity of vardrop_attn_fwd / vardrop_attn_bwd (bf16 tensor-core kernels) with the fp64 oracle.
Tolerance: max-abs 2e-2 and mean-abs 2e-3 on outputs and gradients."""
import numpy as np
import pytest
import torch

import oracle
from paper_2501_14183_b200 import binding as vd
from util import assert_attn_close, bf16_tokens

pytestmark = pytest.mark.gpu


def run_attention(dev, B, N, H, D, sel, poison=True, scale=0.0):
    """Runs forward and backward through the C ABI.  `sel` is None (all tokens) or a sorted int array.
    Returns o[B,Ns,H,D], lse[B,H,Ns], dq, dk, dv (numpy, float64) and the device status."""
    q, k, v, d_full = dev
    cfg = vd.AttnCfg(B, N, H, D, scale)
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
    if poison:
        ws.view(torch.int16).fill_(0x7FC1)        # bf16 NaN pattern everywhere in the scratch
        ws[:4] = 0                                # except the status word, which the caller zeroes (the library only sets it)
    fill = float("nan") if poison else 0.0
    o = torch.full((B, N, H, D), fill, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, N), fill, dtype=torch.float32, device="cuda")
    if sel is None:
        Ns, sel_t, nsel_t, inv_t = N, None, None, None
        d_o = d_full
    else:
        Ns = len(sel)
        sel_pad = np.full(N, -1, np.int32); sel_pad[:Ns] = sel
        inv = np.full(N, -1, np.int32); inv[sel] = np.arange(Ns, dtype=np.int32)
        sel_t = torch.from_numpy(sel_pad).cuda(); inv_t = torch.from_numpy(inv).cuda()
        nsel_t = torch.tensor([Ns], dtype=torch.int32, device="cuda")
        d_o = torch.full((B, N, H, D), fill, dtype=torch.bfloat16, device="cuda")      # rows past Ns may hold anything
        d_o[:, :Ns] = d_full[:, :Ns]
    vd.vardrop_attn_fwd(q, k, v, sel_t, nsel_t, cfg, o, lse, ws)
    dq, dk, dv = (torch.full((B, N, H, D), fill, dtype=torch.bfloat16, device="cuda") for _ in range(3))
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, sel_t, nsel_t, inv_t, cfg, dq, dk, dv, ws)
    torch.cuda.synchronize()
    status = vd.ws_status(ws)
    f = lambda t: t.double().cpu().numpy()
    return f(o)[:, :Ns], f(lse)[:, :, :Ns], f(dq), f(dk), f(dv), status, (o, lse)


def check_case(B, N, H, D, sel, std, seed):
    dev, ref = bf16_tokens(B, N, H, D, std, seed)
    o, lse, dq, dk, dv, status, raw = run_attention(dev, B, N, H, D, sel)
    assert status == vd.OK
    Ns = N if sel is None else len(sel)
    wo, wl = oracle.attn_fwd(ref[0], ref[1], ref[2], sel)
    assert_attn_close(o, wo, "o")
    assert_attn_close(lse, wl, "lse")
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :Ns], sel)
    assert_attn_close(dq, wq, "dq")
    assert_attn_close(dk, wk, "dk")
    assert_attn_close(dv, wv, "dv")
    if sel is not None:
        dropped = np.setdiff1d(np.arange(N), sel)
        for g in (dq, dk, dv):
            assert np.all(g[:, dropped] == 0.0)                      # exact zeros at dropped variates
        # rows of o / lse past n_sel are left untouched (still the NaN fill)
        assert torch.isnan(raw[0][:, Ns:].float()).all() and torch.isnan(raw[1][:, :, Ns:]).all()


def pick(N, Ns, seed):
    return np.sort(np.random.default_rng(seed).choice(N, size=Ns, replace=False)).astype(np.int32)


@pytest.mark.parametrize("B,N,H,D,Ns", [
    (2, 21, 4, 32, 11), (1, 7, 1, 64, 1), (2, 40, 2, 64, 40), (2, 300, 2, 64, 128), (1, 300, 3, 64, 129),
    (2, 321, 2, 64, 97), (1, 600, 2, 64, 300), (1, 500, 2, 32, 257), (3, 130, 1, 64, 127)])
@pytest.mark.parametrize("std", [1.0, 0.3536])
def test_attention_selected(B, N, H, D, Ns, std):
    check_case(B, N, H, D, pick(N, Ns, seed=N + Ns), std, seed=N * 7 + Ns)


@pytest.mark.parametrize("B,N,H,D", [(2, 21, 4, 32), (1, 128, 2, 64), (2, 200, 2, 64), (1, 385, 2, 64), (1, 256, 1, 32), (1, 1, 1, 64)])
def test_attention_all_tokens(B, N, H, D):
    check_case(B, N, H, D, None, 1.0, seed=N)


@pytest.mark.parametrize("B,N,H,D,Ns", [(1, 512, 2, 64, 200), (1, 513, 2, 64, 200), (1, 512, 2, 64, 256), (1, 512, 1, 64, 384),
                                        (1, 512, 1, 64, 512), (1, 640, 2, 32, 384), (2, 1100, 1, 64, 640)])
def test_attention_selected_at_path_boundaries(B, N, H, D, Ns):
    """Kept counts that fill two to five whole tiles exactly, one just past a tile, head size 32: the few-tile kernels, and at 1100 variates (two
    heads and instances in all) the many-tile ones."""
    check_case(B, N, H, D, pick(N, Ns, seed=N * 3 + Ns), 1.0, seed=N + 11 * Ns)


@pytest.mark.parametrize("B,N,H,D,Ns", [(1, 2048, 1, 64, 130), (2, 2049, 1, 64, 1), (1, 2049, 2, 32, 128), (1, 2049, 1, 64, 129), (1, 2300, 3, 64, 384), (1, 257, 2, 64, None), (1, 384, 2, 64, None),
                                        (1, 1024, 2, 64, 256), (1, 1025, 2, 64, 300), (16, 1025, 2, 32, 257), (32, 2048, 1, 32, 700),
                                        (10, 600, 8, 32, None), (8, 2049, 8, 32, 600), (64, 2049, 8, 32, 102), (32, 2049, 8, 64, 128),
                                        (2, 600, 2, 64, None), (2, 2049, 2, 64, 700), (3, 880, 3, 64, None), (24, 600, 8, 32, 300)])
def test_attention_at_the_many_tile_boundary(B, N, H, D, Ns):
    """Both sides of the largest N whose selections count as few tiles (2048, or 1024 with few heads and
    instances; without a selection 256, in the forward pass 384): one kept row, full tiles, remainders; an odd number of key
    tiles with several items a block, so that a team without a key tile in one item has one in the next, or in none of its block's items; several items of one query tile a
    block, where all of an item's hand-offs turn over at every step; blocks whose first item is the odd last
    tiles of two heads over five and more key tiles (the second of which starts a softmax later than the first)."""
    check_case(B, N, H, D, None if Ns is None else pick(N, Ns, seed=N + Ns), 1.0, seed=N + 3 * (Ns or 0))


def test_attention_random_configurations():
    """Seeded random draws of (B, N, H, D, kept count, value scale), with a selection (few-tile kernels) and of all tokens, one to six tiles.
    Value scales stay at or below 1: the absolute tolerance is stated for unit-scale tokens (bf16 rounding of P and dS is
    relative, so gradients of larger tokens carry proportionally larger absolute errors)."""
    rng = np.random.default_rng(2025)
    for it in range(14):
        N = int(rng.integers(2, 760))
        D = int(rng.choice([64, 64, 32]))
        B, H = int(rng.integers(1, 4)), int(rng.integers(1, 4))
        Ns = int(rng.integers(1, N + 1))
        sel = None if it % 4 == 3 else pick(N, Ns, seed=it)
        check_case(B, N, H, D, sel, float(rng.choice([1.0, 0.3536, 0.6])), seed=500 + it)


@pytest.mark.parametrize("B,N,H,D,Ns,std", [(3, 341, 2, 32, 326, 2.0), (2, 604, 1, 64, 210, 2.0), (1, 300, 2, 64, None, 3.0)])
def test_attention_large_tokens_relative_error(B, N, H, D, Ns, std):
    """Tokens a few times the unit scale: peaky softmax rows and gradients of tens.  The errors of the bf16 products are
    relative, so the bound is the unit-scale tolerance times the largest magnitude of the tensor."""
    dev, ref = bf16_tokens(B, N, H, D, std, seed=N + 5)
    sel = None if Ns is None else pick(N, Ns, seed=N)
    o, lse, dq, dk, dv, status, _ = run_attention(dev, B, N, H, D, sel)
    assert status == vd.OK
    n_rows = N if sel is None else len(sel)
    wo, wl = oracle.attn_fwd(ref[0], ref[1], ref[2], sel)
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :n_rows], sel)
    for got, want, name in ((o, wo, "o"), (lse, wl, "lse"), (dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
        bound = 2e-2 * max(1.0, float(np.abs(want).max()))
        err = float(np.abs(got - want).max())
        assert np.all(np.isfinite(got)) and err <= bound, f"{name}: max abs error {err:.3e} > {bound:.3e}"


@pytest.mark.parametrize("N,H,D,Ns", [(257, 2, 64, None), (700, 1, 32, None), (2049, 2, 64, 130), (1030, 1, 32, 257), (300, 1, 64, 200)])
def test_attention_scores_far_below_zero(N, H, D, Ns):
    """Every score near -128 sqrt(D / 64): the exponential of minus a row's log-sum-exp, which a key that does not exist would get, is infinite, and the last
    key tile has such keys.  The bound: as for large tokens."""
    dev, _ = bf16_tokens(2, N, H, D, 0.3536, seed=N)
    dev = [dev[0] + 4.0, dev[1] - 4.0, *dev[2:]]
    ref = [t.double().cpu().numpy() for t in dev]
    sel = None if Ns is None else pick(N, Ns, seed=N)
    o, lse, dq, dk, dv, status, _ = run_attention(dev, 2, N, H, D, sel)
    assert status == vd.OK
    wo, wl = oracle.attn_fwd(ref[0], ref[1], ref[2], sel)
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :Ns or N], sel)
    for got, want, name in ((o, wo, "o"), (lse, wl, "lse"), (dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
        bound = 2e-2 * max(1.0, float(np.abs(want).max()))
        err = float(np.abs(got - want).max())
        assert np.all(np.isfinite(got)) and err <= bound, f"{name}: max abs error {err:.3e} > {bound:.3e}"


@pytest.mark.parametrize("B,N,H,D,Ns", [(2, 257, 2, 64, None), (1, 300, 2, 32, None), (2, 384, 1, 64, None), (1, 385, 2, 64, None), (1, 862, 1, 64, None), (1, 2049, 2, 64, 300)])
def test_attention_probabilities_are_rounded_against_the_first_keys(B, N, H, D, Ns):
    """P is rounded to bf16 relative to the maximum of a row's first 64 keys, whichever kernel serves the call: with that rounding written out
    O is met to its own last bits.  The bound: rows whose last bit falls the other way (fp32 sums, 1e-6 of an element, against a bf16 unit of
    2^-8: one element in 2000) by one unit each, 2^-8 sqrt(1 / 2000) = 9e-5, times four.  Another reference shows as 2.5e-3."""
    dev, _ = bf16_tokens(B, N, H, D, 0.3536, seed=N)
    sel = None if Ns is None else pick(N, Ns, seed=N)
    got = torch.from_numpy(run_attention(dev, B, N, H, D, sel)[0]).cuda()
    idx = slice(None) if sel is None else torch.from_numpy(sel).long().cuda()
    q, k, v = (t[:, idx].double().transpose(1, 2) for t in dev[:3])
    s = q @ k.transpose(-1, -2) * (D ** -0.5 / np.log(2.0))
    p = torch.exp2(s - s[..., :64].amax(dim=-1, keepdim=True))
    want = (p.float().to(torch.bfloat16).double() @ v / p.sum(dim=-1, keepdim=True)).transpose(1, 2).float().to(torch.bfloat16).double()
    assert float((got - want).norm() / want.norm()) <= 3.6e-4


@pytest.mark.parametrize("scale", [2.0 ** -100, 2.0 ** -126, 1e-40, 0.3, 2.0])
@pytest.mark.parametrize("N,D,Ns", [(256, 64, None), (257, 64, None), (300, 32, 200), (1030, 32, 129), (2049, 64, 300)])
def test_attention_of_any_scale(N, D, Ns, scale):
    """Scales of the caller's own, down to the smallest floats, whose quotients of a row's log-sum-exp overflow: every key counts the same then.  The bound: as for large tokens."""
    dev, ref = bf16_tokens(1, N, 2, D, 0.5, seed=N)
    sel = None if Ns is None else pick(N, Ns, seed=N)
    o, lse, dq, dk, dv, status, _ = run_attention(dev, 1, N, 2, D, sel, scale=scale)
    assert status == vd.OK
    wo, wl = oracle.attn_fwd(ref[0], ref[1], ref[2], sel, scale=scale)
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :Ns or N], sel, scale=scale)
    for got, want, name in ((o, wo, "o"), (lse, wl, "lse"), (dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
        bound = 2e-2 * float(np.abs(want).max()) + 1e-37
        err = float(np.abs(got - want).max())
        assert np.all(np.isfinite(got)) and err <= bound, f"{name}: max abs error {err:.3e} > {bound:.3e}"


@pytest.mark.parametrize("where", ["v", "d_o"])
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
@pytest.mark.parametrize("N,D,Ns", [(256, 64, None), (257, 64, None), (700, 32, None), (300, 64, 200), (1030, 32, 129), (2049, 64, 300)])
def test_attention_one_element_that_is_not_finite(N, D, Ns, value, where):
    """An infinity or NaN in one element of V or dO: the gradients that are finite by the chain rule are so (dV of an element of V, every other column of dV of one of dO, the
    other head), whichever kernel serves the call, and within the tolerance."""
    dev, _ = bf16_tokens(1, N, 2, D, 1.0, seed=N)
    sel = None if Ns is None else pick(N, Ns, seed=N)
    dev["q k v d_o".split().index(where)][0, int(sel[5]) if sel is not None and where == "v" else 5, 1, 7] = value
    o, _, dq, dk, dv, status, _ = run_attention(dev, 1, N, 2, D, sel)
    assert status == vd.OK
    ref = [t.double().cpu().numpy() for t in dev]
    wo, _ = oracle.attn_fwd(ref[0], ref[1], ref[2], sel)
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :Ns or N], sel)
    for got, want, name in ((o, wo, "o"), (dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
        finite = np.isfinite(want)
        assert finite.any() and np.array_equal(np.isfinite(got), finite), name
        assert_attn_close(got[finite], want[finite], name)


def test_attention_identity_selection_equals_all_token_path():
    B, N, H, D = 1, 200, 2, 64
    dev, _ = bf16_tokens(B, N, H, D, 1.0, seed=3)
    a = run_attention(dev, B, N, H, D, None, poison=False)
    b = run_attention(dev, B, N, H, D, np.arange(N, dtype=np.int32), poison=False)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])       # forward is bit-reproducible
    for x, y in zip(a[3:5], b[3:5]):
        assert np.array_equal(x, y)                                        # dk, dv too
    np.testing.assert_allclose(a[2], b[2], atol=1e-2)                      # dq: atomics, order may differ


def test_attention_forward_is_deterministic():
    B, N, H, D = 2, 300, 2, 64
    dev, _ = bf16_tokens(B, N, H, D, 1.0, seed=4)
    sel = pick(N, 200, 1)
    a = run_attention(dev, B, N, H, D, sel, poison=False)
    b = run_attention(dev, B, N, H, D, sel, poison=False)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[3], b[3]) and np.array_equal(a[4], b[4])


@pytest.mark.parametrize("B,N,H,D,Ns", [(2, 300, 2, 64, 260), (2, 600, 2, 64, 300), (1, 700, 2, 64, None), (2, 321, 2, 64, 97), (1, 2100, 2, 64, 200),
                                        (2, 2100, 2, 32, 400), (32, 2049, 8, 64, 102), (64, 2049, 8, 32, 128), (20, 2049, 8, 64, 250), (40, 2049, 8, 32, 256), (16, 600, 8, 64, None),
                                        (16, 600, 8, 32, None)])
def test_attention_backward_is_reproducible(B, N, H, D, Ns):
    """Few tiles, many tiles with a selection and of all tokens: every gradient is bit for bit the same from run to run while
    no (instance, head) pair has more than two key tiles' worth of additions per accumulator row (two fp32 addends commute);
    with more tiles dq may differ in the last bits only.  Guards the shared-memory hand-offs inside the backward kernels, and in the many-tile one the order of products that
    it takes for given (scores over probabilities that the product issued before them reads): several items a block, of one, two and five key tiles, at both head sizes."""
    dev, _ = bf16_tokens(B, N, H, D, 1.0, seed=N + (Ns or 0))
    sel = None if Ns is None else pick(N, Ns, 3)
    runs = [run_attention(dev, B, N, H, D, sel, poison=False) for _ in range(3)]
    tiles = -(-(Ns or N) // 128)
    for r in runs[1:]:
        assert np.array_equal(runs[0][3], r[3]) and np.array_equal(runs[0][4], r[4])          # dk, dv
        if tiles <= 2:
            assert np.array_equal(runs[0][2], r[2])                                            # dq
        else:
            np.testing.assert_allclose(runs[0][2], r[2], rtol=0, atol=2e-3)


def test_attention_argument_errors():
    q = torch.zeros((1, 8, 1, 64), dtype=torch.bfloat16, device="cuda")
    lse = torch.zeros((1, 1, 8), device="cuda")
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(vd.AttnCfg(1, 8, 1, 64, 0.0)))
    with pytest.raises(vd.VardropError) as e:
        vd.vardrop_attn_fwd(q, q, q, None, None, vd.AttnCfg(1, 8, 1, 128, 0.0), q, lse, ws)
    assert e.value.status == vd.ERR_UNSUPPORTED
    with pytest.raises(vd.VardropError) as e:
        vd.vardrop_attn_fwd(q, q, q, None, None, vd.AttnCfg(1, 8, 1, 64, 0.0), q, lse, ws[:256])
    assert e.value.status == vd.ERR_WORKSPACE
    with pytest.raises(vd.VardropError) as e:
        vd.vardrop_attn_fwd(q, None, q, None, None, vd.AttnCfg(1, 8, 1, 64, 0.0), q, lse, ws)
    assert e.value.status == vd.ERR_INVALID_ARG


def test_attention_per_instance_selections():
    """One selection per instance (S = B): every instance keeps its own variates, with different counts, spanning one and two tiles."""
    B, N, H, D = 4, 300, 2, 64
    dev, ref = bf16_tokens(B, N, H, D, 1.0, seed=21)
    q, k, v, d_full = dev
    counts = [17, 128, 129, 260]
    sels = [pick(N, c, seed=100 + i) for i, c in enumerate(counts)]
    sel_pad = np.full((B, N), -1, np.int32); inv = np.full((B, N), -1, np.int32)
    for b, s_ in enumerate(sels):
        sel_pad[b, :len(s_)] = s_
        inv[b, s_] = np.arange(len(s_), dtype=np.int32)
    cfg = vd.AttnCfg(B, N, H, D, 0.0, B)
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
    ws.view(torch.int16).fill_(0x7FC1)
    ws[:4] = 0                                    # the status word is the caller's to zero
    nan = float("nan")
    o = torch.full((B, N, H, D), nan, dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, N), nan, dtype=torch.float32, device="cuda")
    d_o = torch.full((B, N, H, D), nan, dtype=torch.bfloat16, device="cuda")
    for b, c in enumerate(counts):
        d_o[b, :c] = d_full[b, :c]
    sel_t, inv_t = torch.from_numpy(sel_pad).cuda(), torch.from_numpy(inv).cuda()
    nsel_t = torch.tensor(counts, dtype=torch.int32, device="cuda")
    vd.vardrop_attn_fwd(q, k, v, sel_t, nsel_t, cfg, o, lse, ws)
    dq, dk, dv = (torch.full((B, N, H, D), nan, dtype=torch.bfloat16, device="cuda") for _ in range(3))
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, sel_t, nsel_t, inv_t, cfg, dq, dk, dv, ws)
    torch.cuda.synchronize()
    assert vd.ws_status(ws) == vd.OK
    for b, (c, s_) in enumerate(zip(counts, sels)):
        cut = [r[b:b + 1] for r in ref]
        wo, wl = oracle.attn_fwd(cut[0], cut[1], cut[2], s_)
        assert_attn_close(o[b:b + 1, :c].double().cpu().numpy(), wo, f"o[{b}]")
        assert_attn_close(lse[b:b + 1, :, :c].double().cpu().numpy(), wl, f"lse[{b}]")
        wq, wk, wv = oracle.attn_bwd(cut[0], cut[1], cut[2], cut[3][:, :c], s_)
        for got, want, name in ((dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
            g = got[b:b + 1].double().cpu().numpy()
            assert_attn_close(g, want, f"{name}[{b}]")
            assert np.all(g[:, np.setdiff1d(np.arange(N), s_)] == 0.0)
        assert torch.isnan(o[b, c:].float()).all()


@pytest.mark.parametrize("B,N,H,D,counts", [
    (20, 140, 8, 64, [60 + 3 * i for i in range(20)][:19] + [140]),            # one instance of two tiles: its CTAs apart from the others
    (24, 260, 8, 32, [100 + (37 * i) % 160 for i in range(24)]),               # many of two and three: every CTA both kinds
    (3, 200, 1, 64, [129, 1, 128]), (2, 300, 2, 64, [130, 300]), (3, 300, 2, 64, [0, 128, 260]),
    # the many-tile kernels: nothing kept, one row, whole tiles, odd and even tile counts, more items than blocks
    (5, 2100, 4, 64, [0, 1, 256, 300, 700]), (9, 1030, 3, 32, [5, 130, 257, 384, 640, 128, 900, 1, 129]), (16, 2060, 8, 32, [100 + 37 * i for i in range(16)]),
    (64, 2049, 8, 32, [(128, 1, 100, 0, 127)[i % 5] for i in range(64)])])
def test_attention_instances_of_one_and_of_several_tiles(B, N, H, D, counts):
    dev, ref = bf16_tokens(B, N, H, D, 1.0, seed=B + N)
    q, k, v, d_o = dev
    sels = [pick(N, c, seed=40 + i) for i, c in enumerate(counts)]
    sel, inv = (torch.full((B, N), -1, dtype=torch.int32) for _ in range(2))
    for b, s_ in enumerate(sels):
        sel[b, :len(s_)] = torch.from_numpy(np.asarray(s_, dtype=np.int32))
        inv[b, torch.from_numpy(np.asarray(s_, dtype=np.int64))] = torch.arange(len(s_), dtype=torch.int32)
    sel, inv, n_sel = sel.cuda(), inv.cuda(), torch.tensor(counts, dtype=torch.int32, device="cuda")
    cfg = vd.AttnCfg(B, N, H, D, 0.0, B)
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
    o, dq, dk, dv = (torch.full((B, N, H, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(4))
    lse = torch.zeros((B, H, N), dtype=torch.float32, device="cuda")
    for _ in range(2):                                                         # a workspace that has been used
        vd.vardrop_attn_fwd(q, k, v, sel, n_sel, cfg, o, lse, ws)
        vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, sel, n_sel, inv, cfg, dq, dk, dv, ws)
    torch.cuda.synchronize()
    assert vd.ws_status(ws) == vd.OK
    for b, s_ in enumerate(sels):
        cut = [r[b:b + 1] for r in ref]
        if len(s_) == 0:
            assert not dq[b].any() and not dk[b].any() and not dv[b].any()
            continue
        wo, _ = oracle.attn_fwd(cut[0], cut[1], cut[2], s_)
        assert_attn_close(o[b:b + 1, :len(s_)].double().cpu().numpy(), wo, f"o[{b}]")
        wq, wk, wv = oracle.attn_bwd(cut[0], cut[1], cut[2], cut[3][:, :len(s_)], s_)
        for got, want, name in ((dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
            g = got[b:b + 1].double().cpu().numpy()
            assert_attn_close(g, want, f"{name}[{b}]")
            assert np.all(g[:, np.setdiff1d(np.arange(N), s_)] == 0.0)


@pytest.mark.parametrize("N", [100, 300, 400])
def test_attention_of_all_tokens_takes_a_configuration_for_selections_per_instance(N):
    """S = B in the configuration and no selection: every token, as with S = 1."""
    B, H, D = 3, 2, 64
    (q, k, v, d_o), _ = bf16_tokens(B, N, H, D, 0.5, seed=N)
    runs = []
    for S in (1, B):
        cfg = vd.AttnCfg(B, N, H, D, 0.0, S)
        ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
        o, dq, dk, dv = (torch.zeros_like(q) for _ in range(4))
        lse = torch.zeros((B, H, N), device="cuda")
        vd.vardrop_attn_fwd(q, k, v, None, None, cfg, o, lse, ws)
        vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, None, None, None, cfg, dq, dk, dv, ws)
        torch.cuda.synchronize()
        assert vd.ws_status(ws) == vd.OK
        runs.append((o, lse, dk, dv, dq))
    for a, b in zip(runs[0][:4], runs[1][:4]):
        assert torch.equal(a, b)
    np.testing.assert_allclose(runs[0][4].float().cpu().numpy(), runs[1][4].float().cpu().numpy(), rtol=0, atol=2e-3)      # dq: fp32 adds in no fixed order


def run_strided(q, k, v, d_full, B, N, H, D, sel):
    """q, k, v are (possibly non-contiguous) views [B, N, H, D] with a contiguous head dimension; their strides go into the config."""
    assert q.stride() == k.stride() == v.stride() and q.stride(3) == 1
    cfg = vd.AttnCfg(B, N, H, D, 0.0, 1, q.stride(0), q.stride(1), q.stride(2))
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
    o = torch.full((B, N, H, D), float("nan"), dtype=torch.bfloat16, device="cuda")
    lse = torch.full((B, H, N), float("nan"), dtype=torch.float32, device="cuda")
    if sel is None:
        Ns, sel_t, nsel_t, inv_t, d_o = N, None, None, None, d_full
    else:
        Ns = len(sel)
        sel_pad = np.full(N, -1, np.int32); sel_pad[:Ns] = sel
        inv = np.full(N, -1, np.int32); inv[sel] = np.arange(Ns, dtype=np.int32)
        sel_t, inv_t = torch.from_numpy(sel_pad).cuda(), torch.from_numpy(inv).cuda()
        nsel_t = torch.tensor([Ns], dtype=torch.int32, device="cuda")
        d_o = torch.full((B, N, H, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        d_o[:, :Ns] = d_full[:, :Ns]
    vd.vardrop_attn_fwd(q, k, v, sel_t, nsel_t, cfg, o, lse, ws)
    dq, dk, dv = (torch.full((B, N, H, D), float("nan"), dtype=torch.bfloat16, device="cuda") for _ in range(3))
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, sel_t, nsel_t, inv_t, cfg, dq, dk, dv, ws)
    torch.cuda.synchronize()
    assert vd.ws_status(ws) == vd.OK
    f = lambda t: t.double().cpu().numpy()
    return f(o)[:, :Ns], f(lse)[:, :, :Ns], f(dq), f(dk), f(dv)


@pytest.mark.parametrize("layout", ["fused_qkv", "padded_heads", "padded_tokens", "token_slice"])
@pytest.mark.parametrize("B,N,H,D,Ns", [(2, 300, 2, 64, 140), (1, 700, 2, 64, 300), (2, 200, 3, 64, None), (1, 600, 2, 64, None), (2, 90, 2, 32, 50),
                                        (1, 2100, 2, 64, 300), (2, 1100, 3, 32, 140)])
def test_attention_strided_qkv(layout, B, N, H, D, Ns):
    """q, k, v as views of larger buffers (the element strides of the configuration): slices of a fused [B, N, 3, H, D] projection,
    heads padded to D + 8, tokens padded by 8 elements, and a slice along N of a longer sequence; with few tiles, with many (rows laid out
    from the strided tensors ahead of the backward pass) and of all tokens.  Results must match the oracle run on contiguous copies."""
    dev, ref = bf16_tokens(B, N, H, D, 0.5, seed=N + H)
    gen = torch.Generator(device="cuda").manual_seed(5)
    junk = lambda *shape: (torch.rand(shape, device="cuda", generator=gen) * 8 - 4).to(torch.bfloat16)       # what lies between the rows
    if layout == "fused_qkv":
        buf = junk(B, N, 3, H, D)
        views = [buf[:, :, i] for i in range(3)]
    elif layout == "padded_heads":
        bufs = [junk(B, N, H, D + 8) for _ in range(3)]
        views = [b[..., :D] for b in bufs]
    elif layout == "padded_tokens":
        bufs = [junk(B, N, H * D + 8) for _ in range(3)]
        views = [b[..., : H * D].unflatten(-1, (H, D)) for b in bufs]
    else:
        bufs = [junk(B, N + 37, H, D) for _ in range(3)]
        views = [b[:, 16: 16 + N] for b in bufs]
    for view, t in zip(views, dev[:3]):
        view.copy_(t)
    sel = None if Ns is None else pick(N, Ns, seed=N)
    o, lse, dq, dk, dv = run_strided(views[0], views[1], views[2], dev[3], B, N, H, D, sel)
    n_rows = N if sel is None else len(sel)
    wo, wl = oracle.attn_fwd(ref[0], ref[1], ref[2], sel)
    wq, wk, wv = oracle.attn_bwd(ref[0], ref[1], ref[2], ref[3][:, :n_rows], sel)
    for got, want, name in ((o, wo, "o"), (lse, wl, "lse"), (dq, wq, "dq"), (dk, wk, "dk"), (dv, wv, "dv")):
        assert_attn_close(got, want, f"{layout} {name}")


def test_attention_stride_validation():
    q = torch.zeros((1, 8, 2, 64), dtype=torch.bfloat16, device="cuda")
    o = torch.zeros_like(q)
    lse = torch.zeros((1, 2, 8), device="cuda")
    ws = vd.alloc_ws(1 << 20)
    for strides in [(8 * 128, 128, 60), (8 * 128, 132, 64), (100, 128, 64), (8 * 128, 64, 128)]:
        with pytest.raises(vd.VardropError) as e:
            vd.vardrop_attn_fwd(q, q, q, None, None, vd.AttnCfg(1, 8, 2, 64, 0.0, 1, *strides), o, lse, ws)
        assert e.value.status == vd.ERR_INVALID_ARG


def test_backward_without_a_fresh_forward_is_reported():
    """The forward pass leaves state for exactly one backward pass in the workspace; a second backward on it is flagged in the
    device status word instead of silently adding into a consumed accumulator."""
    B, N, H, D = 1, 300, 2, 64
    dev, _ = bf16_tokens(B, N, H, D, 1.0, seed=3)
    q, k, v, d_o = dev
    cfg = vd.AttnCfg(B, N, H, D, 0.0)
    ws = vd.alloc_ws(vd.vardrop_attn_workspace_bytes(cfg))
    o = torch.zeros_like(q); lse = torch.zeros((B, H, N), device="cuda")
    dq, dk, dv = (torch.zeros_like(q) for _ in range(3))
    vd.vardrop_attn_fwd(q, k, v, None, None, cfg, o, lse, ws)
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, None, None, None, cfg, dq, dk, dv, ws)
    assert vd.ws_status(ws) == vd.OK
    first = dq.clone()
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, None, None, None, cfg, dq, dk, dv, ws)          # no forward in between
    assert vd.ws_status(ws) == vd.ERR_INVALID_ARG
    ws[:4] = 0                                                                                 # the caller clears the word ...
    vd.vardrop_attn_fwd(q, k, v, None, None, cfg, o, lse, ws)                                  # ... and the pair works again
    vd.vardrop_attn_bwd(q, k, v, o, lse, d_o, None, None, None, cfg, dq, dk, dv, ws)
    assert vd.ws_status(ws) == vd.OK
    np.testing.assert_allclose(dq.float().cpu().numpy(), first.float().cpu().numpy(), rtol=0, atol=2e-3)
