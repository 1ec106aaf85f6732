"""The work whose speed counts: what a program that trains with VarDrop has this library do, over the sizes it does it at.

Kinds of a case (`kind`), each one pass through the public entry points of paper_2501_14183_b200.binding:

  step     one training step's token reduction and attention: vardrop_hash -> vardrop_select -> vardrop_attn_fwd -> vardrop_attn_bwd
  thin     the variates dropped from the lookback window itself, ahead of the embedding: vardrop_hash -> vardrop_select -> vardrop_gather_rows
  ground   training with every token kept (VarDrop off): vardrop_attn_fwd -> vardrop_attn_bwd without a selection
  infer    inference, every token kept: vardrop_attn_fwd alone
  pearson  the redundancy statistic of a batch: vardrop_pearson_max

Ranges: 1 to 32 instances, 16 to 8192 variates, windows of 32 to 1024 steps (mostly the lookbacks 96, 192, 336 and 720 of the
forecasting benchmarks, and any other length), 2 to 5 ranked frequencies, a kept share of 5 to 50 % by rate or by a group cap, 4 or 8
heads of 32 or 64, hashing over the batch or per instance, q / k / v as tensors of their own or as views of one fused projection.
"""
import math

import torch

from paper_2501_14183_b200 import binding as vd

SEED, STEP = 20250114, 1
GAP = 1e-3              # a hash is taken as decided when its ranked amplitudes differ by more than this share


def _step(name, B, N, L, k, H, D, templates, shared, periods, rate=1.0, gs=0, scope=0, fused=False, sigma=0.1, std=math.sqrt(1.0 / 8.0), kind="step"):
    return dict(name=name, kind=kind, B=B, N=N, L=L, k=k, H=H, D=D, templates=templates, shared=shared, periods=periods, rate=rate, gs=gs, scope=scope,
                fused=fused, sigma=sigma, std=std)


_DAY = "24,12,8,72,6"
_WEEK = "24,12,168,48,8,6,336"
_MANY = "336,168,112,84,56,48,42,28,24,16,14,12,8,7,6"


def listed():
    return [
        # the smallest training step: a weather-station set of 21 variates, heads of 32; latency and launches are all there is
        _step("tiny step", 4, 21, 96, 2, 4, 32, 4, 1.0, "24,12,48,8,32,16", rate=0.5, std=1.0),
        # electricity-consumption training step (321 clients): the kept set is one tile per head
        _step("electricity step", 32, 321, 96, 3, 8, 64, 40, 0.8, _DAY, rate=0.3),
        # the same with every instance hashed and sampled on its own, q / k / v views of one fused projection
        _step("electricity step, per instance", 32, 321, 96, 3, 8, 64, 40, 0.8, _DAY, rate=0.3, scope=1, fused=True),
        # solar-plant training step (137 sites): Eq. 1 with a group cap, a window of a week of hours (168 = 2^3 3 7)
        _step("solar step, window 168", 32, 137, 168, 3, 8, 64, 2, 1.0, _DAY, gs=20),
        # road-traffic training step (862 sensors): the kept set is two tiles per head
        _step("traffic step", 32, 862, 96, 3, 8, 64, 60, 0.95, _DAY, rate=0.2, sigma=0.05),
        # the same sensors with a month of lookback
        _step("long lookback step", 16, 862, 720, 5, 8, 64, 80, 1.0, _WEEK, rate=0.2),
        # thousands of variates: a dozen kept tiles per head
        _step("scale step", 8, 8192, 336, 4, 8, 64, 512, 0.95, _MANY, rate=0.1),
        # the drop placed on the raw window (road traffic), ahead of the embedding
        _step("traffic thinning", 32, 862, 96, 3, 8, 64, 60, 0.95, _DAY, rate=0.2, sigma=0.05, kind="thin"),
        # inference on all 321 clients
        dict(name="electricity inference", kind="infer", B=32, N=321, H=8, D=64, fused=False, std=math.sqrt(1.0 / 8.0)),
        # training without the drop: the road-traffic sensors, and thousands of variates (the largest piece of work here)
        dict(name="traffic ground", kind="ground", B=32, N=862, H=8, D=64, fused=False, std=math.sqrt(1.0 / 8.0)),
        dict(name="scale ground", kind="ground", B=8, N=8192, H=8, D=64, fused=False, std=math.sqrt(1.0 / 8.0)),
        # how redundant a batch is: every variate's largest correlation (road traffic)
        dict(name="traffic redundancy", kind="pearson", B=32, N=862, L=96, templates=60, shared=0.95, periods=_DAY, sigma=0.05),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["step", "thin", "ground", "infer", "pearson"], [7, 1, 2, 1, 1])[0]
    B, N = _log_int(rng, 1, 32), _log_int(rng, 16, 8192)
    H, D = rng.choice([4, 8, 8]), rng.choice([32, 64, 64, 64])
    L = rng.choice([96, 96, 192, 336, 720, _log_int(rng, 32, 1024)])
    std = rng.choice([1.0, math.sqrt(1.0 / 8.0)])
    data = dict(L=L, templates=max(2, N // rng.randint(8, 16)), shared=rng.choice([0.8, 0.95, 1.0]), sigma=rng.choice([0.05, 0.1]),
                periods=rng.choice([_DAY, _WEEK, _MANY]) if L >= 48 else "24,12,8,6,16,10")
    tokens = dict(H=H, D=D, fused=rng.random() < 0.3, std=std)
    sampling = dict(rate=1.0, gs=rng.randint(3, 20)) if rng.random() < 0.3 else dict(rate=rng.choice([0.05, 0.1, 0.2, 0.3, 0.5]), gs=0)
    case = dict(kind=kind, B=B, N=N)
    if kind in ("step", "thin", "pearson"):
        case.update(data)
    if kind in ("step", "thin"):
        case.update(k=rng.randint(2, 5), scope=1 if rng.random() < 0.2 else 0, **sampling)
    if kind in ("step", "ground", "infer"):
        case.update(tokens)
    largest = work(listed()[-2])
    while case["B"] > 1 and (case["B"] * N * L > 8 * 8192 * 336 or any(work(case)[w] > 0.8 * largest[w] for w in largest)):
        case["B"] //= 2
    return case


# ---- inputs -----------------------------------------------------------------------------------------------------------------
def _windows(c, gen):
    """x[B, N, L]: variates that mostly share periodic templates (an ordered set of periods with a falling amplitude ladder), each with
    its own amplitudes and phases, a time shift per instance, noise, every window normalised."""
    dev = dict(device="cuda")
    B, N, L = c["B"], c["N"], c["L"]
    periods = torch.tensor([float(p) for p in c["periods"].split(",")], **dev)
    m = min(c.get("k", 3), len(periods))
    T = c["templates"]

    def templates(count):
        order = torch.rand((count, len(periods)), generator=gen, **dev).argsort(dim=1)[:, :m]
        ratio = torch.cat([torch.ones((count, 1), **dev), 1.5 + 1.5 * torch.rand((count, m - 1), generator=gen, **dev)], dim=1)
        return periods[order], 1.0 / torch.cumprod(ratio, dim=1), 2 * math.pi * torch.rand((count, m), generator=gen, **dev)

    own, common = templates(N), templates(T)
    pick = torch.randint(0, T, (N,), generator=gen, **dev)
    shares = (torch.rand((N, 1), generator=gen, **dev) < c["shared"])
    P, A, PH = (torch.where(shares, a[pick], b) for a, b in zip(common, own))
    A = A * (1.0 + 0.4 * (torch.rand((N, m), generator=gen, **dev) - 0.5))
    PH = PH + 0.1 * torch.randn((N, m), generator=gen, **dev)
    tau = torch.randint(0, 4 * L, (B,), generator=gen, **dev).float()
    t = torch.arange(L, **dev).float()[None, :] + tau[:, None]                  # [B, L]
    x = c["sigma"] * torch.randn((B, N, L), generator=gen, **dev)
    for i in range(m):
        x += A[None, :, i, None] * torch.sin(2 * math.pi * t[:, None, :] / P[None, :, i, None] + PH[None, :, i, None])
    x -= x.mean(dim=-1, keepdim=True)
    x /= x.std(dim=-1, keepdim=True) + 1e-12
    return x


def _decided(c, x):
    """Replaces the few variates whose ranked frequencies are nearly tied (a 32-bit transform may rank them either way) by copies of
    decided ones, so that hash values, groups and kept sets are the same for every correct implementation."""
    L, k = c["L"], c["k"]
    f_hi = (L // 2 + 2) // 2
    amp = torch.stack([torch.fft.rfft(xb.double(), dim=-1)[:, 1:f_hi].abs() for xb in x])
    amp = amp.mean(dim=0, keepdim=True) if c["scope"] == 0 else amp              # [S, N, bins]
    top = amp.topk(min(k + 1, f_hi - 1), dim=-1).values
    gap = ((top[..., :-1] - top[..., 1:]) / top[..., :-1]).amin(dim=-1)
    bad = gap <= 2 * GAP
    if not bool(bad.any()) or bool(bad.all(dim=1).any()):
        return x
    for s in range(bad.shape[0]):
        b, good = bad[s].nonzero()[:, 0], (~bad[s]).nonzero()[:, 0]
        if len(b):
            rows = slice(None) if c["scope"] == 0 else slice(s, s + 1)
            x[rows, b] = x[rows, good[torch.arange(len(b), device="cuda") % len(good)]]
    return x


def _tokens(c, gen):
    B, N, H, D = c["B"], c["N"], c["H"], c["D"]
    mk = lambda *shape: (c["std"] * torch.randn(shape, generator=gen, device="cuda")).to(torch.bfloat16)  # noqa: E731
    if c["fused"]:
        qkv = mk(B, N, 3, H, D)
        q, k, v = (qkv[:, :, i] for i in range(3))
        strides = (3 * N * H * D, 3 * H * D, D)
    else:
        q, k, v = (mk(B, N, H, D) for _ in range(3))
        strides = (0, 0, 0)
    return q, k, v, mk(B, N, H, D), strides


def prepare(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(1 + seed)
    B, N = c["B"], c["N"]
    s = dict(kind=c["kind"])
    if c["kind"] == "pearson":
        cfg = vd.PearsonCfg(B, N, c["L"], 0.9)
        s.update(x=_windows(c, gen), pcfg=cfg, max_rho=torch.empty((B, N), device="cuda"), n_above=torch.empty((B,), dtype=torch.int32, device="cuda"),
                 pws=vd.alloc_ws(vd.vardrop_pearson_workspace_bytes(cfg)))
        return s
    S = 1
    if c["kind"] in ("step", "thin"):
        S = B if c["scope"] else 1
        x = _decided(c, _windows(c, gen))
        hcfg = vd.HashCfg(B, N, c["L"], c["k"], 0, 0, c["scope"])
        scfg = vd.SelectCfg(S, N, c["gs"], c["rate"], SEED, STEP)
        keys, freqs, _ = vd.alloc_hash_outputs(hcfg)
        s.update(x=x, hcfg=hcfg, scfg=scfg, keys=keys, freqs=freqs, sel=vd.alloc_select_outputs(scfg),
                 hws=vd.alloc_ws(vd.vardrop_hash_workspace_bytes(hcfg)), sws=vd.alloc_ws(vd.vardrop_select_workspace_bytes(scfg)))
    if c["kind"] == "thin":
        s.update(gcfg=vd.GatherCfg(B, N, c["L"], S), x_sel=torch.zeros_like(s["x"]))
        return s
    q, k, v, d_o, strides = _tokens(c, gen)
    acfg = vd.AttnCfg(B, N, c["H"], c["D"], 0.0, S, *strides)
    s.update(q=q, k=k, v=v, acfg=acfg, o=torch.zeros_like(d_o), lse=torch.zeros((B, c["H"], N), device="cuda"), aws=vd.alloc_ws(vd.vardrop_attn_workspace_bytes(acfg)))
    if c["kind"] != "infer":
        s.update(d_o=d_o, dq=torch.empty_like(d_o), dk=torch.empty_like(d_o), dv=torch.empty_like(d_o))
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "pearson":
        vd.vardrop_pearson_max(s["x"], s["pcfg"], s["max_rho"], s["n_above"], s["pws"])
        return {"max_rho": s["max_rho"], "n_above": s["n_above"]}
    out = {}
    sel_idx = n_sel = inv_idx = None
    if kind == "step" or kind == "thin":
        sel = s["sel"]
        vd.vardrop_hash(s["x"], s["hcfg"], s["keys"], s["freqs"], None, s["hws"])
        vd.vardrop_select(s["keys"], s["scfg"], sel["group_id"], sel["group_offsets"], sel["members"], sel["n_groups"], sel["sel_idx"], sel["n_sel"],
                          sel["inv_idx"], s["sws"])
        sel_idx, n_sel, inv_idx = sel["sel_idx"], sel["n_sel"], sel["inv_idx"]
        out.update(keys=s["keys"], freqs=s["freqs"], **sel)
        if kind == "thin":
            vd.vardrop_gather_rows(s["x"], sel_idx, n_sel, s["gcfg"], s["x_sel"])
            out["x_sel"] = s["x_sel"]
            return out
    vd.vardrop_attn_fwd(s["q"], s["k"], s["v"], sel_idx, n_sel, s["acfg"], s["o"], s["lse"], s["aws"])
    out.update(o=s["o"], lse=s["lse"])
    if kind != "infer":
        vd.vardrop_attn_bwd(s["q"], s["k"], s["v"], s["o"], s["lse"], s["d_o"], sel_idx, n_sel, inv_idx, s["acfg"], s["dq"], s["dk"], s["dv"], s["aws"])
        out.update(dq=s["dq"], dk=s["dk"], dv=s["dv"])
    return out


# ---- what a pass cannot do without ------------------------------------------------------------------------------------------
def _kept(c):
    """Kept variates to expect: a share of every group rounded up (half a variate a group), at most `gs` of a group when there is a cap."""
    n_per = len(c["periods"].split(","))
    orders = math.perm(n_per, min(c["k"], n_per))
    shared = c["shared"] * c["N"]
    groups = min(orders, min(c["templates"], shared) + (c["N"] - shared))
    kept = c["rate"] * c["N"] + 0.5 * groups if c["rate"] < 1.0 else c["N"]
    return min(c["N"], kept, groups * c["gs"]) if c["gs"] > 0 else min(c["N"], kept)


def work(case):
    c = case
    B, N, kind = c["B"], c["N"], c["kind"]
    nbytes = flops = 0.0
    if kind in ("step", "thin", "pearson"):
        nbytes += 4.0 * B * N * c["L"]
    if kind == "pearson":
        return {"bytes": nbytes + 4.0 * B * N, "flops": float(B) * N * N * c["L"]}          # every pair once: a multiply and an add a step
    kept = N
    if kind in ("step", "thin"):
        S = B if c["scope"] else 1
        kept = _kept(c)
        nbytes += S * N * (8 + 4 * c["k"] + 6 * 4)
        flops += 2.5 * B * N * c["L"] * math.log2(c["L"])
    if kind == "thin":
        return {"bytes": nbytes + 4.0 * B * kept * c["L"], "flops": flops}
    row = 2.0 * c["H"] * c["D"]
    nbytes += 4 * B * kept * row + 4.0 * B * kept * c["H"]                                  # q, k, v in, o and lse out
    flops += 4.0 * B * c["H"] * kept * kept * c["D"]
    if kind != "infer":
        nbytes += B * kept * row + 3 * B * N * row                                          # dO in, gradients of the full layout out
        flops += 10.0 * B * c["H"] * kept * kept * c["D"]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "thin":
        return "exact"                      # integers, and copies of floats
    if case["kind"] == "pearson":
        return {"rel": 1e-4}                # correlations from values of 16 mantissa bits
    return {"rel": 1e-2}                    # bf16 operands and results; hash values, groups and kept sets are whole numbers and stay the same
