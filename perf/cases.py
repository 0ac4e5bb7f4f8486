"""What a user of the library has it do, as cases that can be timed.

Five kinds of call, each through the package's public entry points:

  train    one layer's routing-balance step from logits in hand
           (eqb_layer_step: routing, loads, next bias, LEI into the score
           gradients), once per MoE layer and optimizer step
  router   the same from the router input (eqb_router_layer_step)
  serve    inference: project, route, no statistic (eqb_router_route where it
           takes the shape, else eqb_router_logits and eqb_route_topk): a few
           tokens when decoding, thousands at prefill
  dp       one data-parallel rank's share of a training step, through the
           separate calls between which the histograms are all-reduced
           (eqb_layer_forward, then lei_inject_grad)
  compare  the methods that the step is compared with, on one batch:
           gshard_inject_grad, eqb_rank_averaged_bias, eqb_fixed_hist_bias,
           eqb_maxvio

Sizes are the repository's configurations (tiny, tie, mid, global, paper,
wide, router) and ragged ones between them.  `draw` spreads over the range
from 512 to about 4 million tokens, 8 to 1024 experts.

Gradients are N(0, 0.1^2), and the step adds to them in place as it does in
a training loop; the other outputs are written anew by every pass.
"""
import math

import torch

import paper_2609_28053_gb300 as eqb

ETA, C = 2e-5, 1.0        # LEI strength and normalisation (the paper's middle sweep value)
ALPHA = 0.1               # GShard auxiliary-loss weight
BIN_LO, BIN_W = -4.0, 1.0 / 32  # 256 equal bins of the fixed-resolution estimate


def listed():
    return [
        # The smallest training step: four launches' latency and little else.
        {"name": "train_tiny", "kind": "train", "T": 4096, "E": 8, "K": 2, "M": 4, "z": "normal", "b": "zero"},
        # Nearly constant logits per expert: many equal scores, a cold expert set.
        {"name": "train_tie", "kind": "train", "T": 65536, "E": 64, "K": 8, "M": 8, "z": "tie", "b": "narrow"},
        # Hot experts and the bias that one update has made for them: a run in its steady state.
        {"name": "train_mid", "kind": "train", "T": 524288, "E": 128, "K": 8, "M": 32, "z": "hot", "b": "steady"},
        # The headline shape: heavy-tailed logits, a bias away from its fixed point.
        {"name": "train_global", "kind": "train", "T": 2097152, "E": 256, "K": 8, "M": 64, "z": "heavy", "b": "drawn"},
        # The paper's global batch, 64 ranks of 147,456 tokens, top-6, in its steady state.
        {"name": "train_paper", "kind": "train", "T": 9437184, "E": 256, "K": 6, "M": 64, "z": "normal", "b": "steady"},
        # More experts than one block's histogram holds.
        {"name": "train_wide", "kind": "train", "T": 1048576, "E": 512, "K": 8, "M": 32, "z": "normal", "b": "drawn"},
        # An expert count that is no power of two and microbatches of uneven sizes.
        {"name": "train_ragged", "kind": "train", "T": 200003, "E": 96, "K": 6, "M": 7, "ragged": True, "z": "normal", "b": "drawn"},
        # From the router input: the projection is most of the bytes.
        {"name": "router_full", "kind": "router", "T": 1048576, "d": 4096, "E": 128, "K": 8, "M": 16, "b": "zero"},
        # Decoding: one projection tile, latency only.
        {"name": "serve_decode", "kind": "serve", "T": 128, "d": 4096, "E": 128, "K": 8, "b": "narrow"},
        # Prefill with more experts than are routed from the accumulators.
        {"name": "serve_prefill", "kind": "serve", "T": 16411, "d": 2048, "E": 256, "K": 8, "b": "narrow"},
        # One rank's 147,456 tokens of the paper's batch through the separate calls.
        {"name": "dp_rank", "kind": "dp", "T": 147456, "E": 256, "K": 6, "M": 1, "z": "normal", "b": "steady"},
        # The comparison methods on the mid shape.
        {"name": "compare_mid", "kind": "compare", "T": 524288, "E": 128, "K": 8, "M": 32, "P": 16, "z": "hot", "b": "steady"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "router", "serve", "dp", "compare"])
    case = {"kind": kind}
    if kind in ("router", "serve"):
        case["d"] = rng.choice([512, 1024, 2048, 4096])
        case["E"] = rng.choice([16, 48, 64, 128, 128, 256])
        case["T"] = _log_int(rng, 1, 65536) if kind == "serve" else _log_int(rng, 512, 400000)
        case["b"] = rng.choice(["zero", "narrow"])
    else:
        case["E"] = rng.choice([8, 16, 64, 96, 128, 160, 256, 256, 256, 264, 384, 512, 1024])
        case["T"] = _log_int(rng, 512, min(4 << 20, (1 << 30) // case["E"]))
        case["z"] = rng.choice(["normal", "hot", "heavy", "tie"])
        case["b"] = rng.choice(["zero", "narrow", "drawn", "steady"])
    case["K"] = min(rng.choice([1, 2, 4, 6, 8, 8, 12]), case["E"] // 4)
    if kind != "serve":
        case["M"] = rng.randint(1, 64)
        case["ragged"] = rng.random() < 0.5
    if kind in ("train", "router"):
        case["grad"] = rng.random() < 0.8  # without LEI: the forward statistic alone
    if kind == "compare":
        case["P"] = rng.randint(1, 64)
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _offsets(case, gen):
    T, M = case["T"], case["M"]
    if case.get("ragged") and M > 1:
        cuts = torch.randint(0, T + 1, (M - 1,), generator=gen, device="cuda").sort().values
        return torch.cat([cuts.new_zeros(1), cuts, cuts.new_full((1,), T)])
    return (torch.arange(M + 1, dtype=torch.int64, device="cuda") * T) // M


def _logits(case, T, gen):
    """bf16 logits [T,E]: unit normals; per-expert constants with little
    noise; 1/8 of the experts 1.0 hotter; or a tenth of the values from a
    heavy tail (2 x Student-t with 3 degrees of freedom)."""
    E, kind = case["E"], case["z"]
    # the experts' own levels: of the case, not of the batch
    g0 = _gen(1000 + E)
    level = torch.zeros(E, device="cuda")
    if kind == "tie":
        level = torch.randn(E, generator=g0, device="cuda") * 0.5
    elif kind == "hot":
        level[torch.randperm(E, generator=g0, device="cuda")[: max(1, E // 8)]] = 1.0
    z = torch.empty((T, E), dtype=torch.bfloat16, device="cuda")
    for t in range(0, T, 1 << 20):
        n = min(T - t, 1 << 20)
        x = torch.randn((n, E), generator=gen, device="cuda")
        if kind == "tie":
            x.mul_(0.05)
        elif kind == "heavy":
            chi = sum(torch.randn((n, E), generator=gen, device="cuda") ** 2 for _ in range(3))
            tail = torch.rand((n, E), generator=gen, device="cuda") < 0.1
            x = torch.where(tail, 2.0 * x / torch.sqrt(chi / 3.0), x)
        z[t:t + n] = (x + level).to(torch.bfloat16)
    return z


def _bias(case, gen):
    """fp32 bias [E]: zeros (a first step), U(-0.1, 0.1), N(0, 0.2^2), or the
    one that the update makes from a batch like this one."""
    E, K, kind = case["E"], case["K"], case["b"]
    if kind == "zero":
        return torch.zeros(E, device="cuda")
    if kind == "narrow":
        return torch.rand(E, generator=gen, device="cuda") * 0.2 - 0.1
    if kind == "drawn":
        return torch.randn(E, generator=gen, device="cuda") * 0.2
    z = _logits(case, 16384, gen).float()
    m = z.topk(K + 1, dim=1).values[:, K:] - z
    q = m.t().contiguous().kthvalue(-(-16384 * K // E), dim=1).values
    return q - q.mean()


def _grad(case, gen):
    return torch.randn((case["T"], case["E"]), generator=gen, device="cuda").mul_(0.1)


def _inputs(case, seed):
    gen = _gen(seed)
    s = {"case": case}
    T, E, K = case["T"], case["E"], case["K"]
    if case["kind"] in ("router", "serve"):
        d = case["d"]
        s["x"] = torch.randn((T, d), generator=gen, device="cuda", dtype=torch.bfloat16)
        s["W"] = (torch.randn((E, d), generator=gen, device="cuda") / math.sqrt(d)).to(torch.bfloat16)
    else:
        s["z"] = _logits(case, T, gen)
    s["b"] = _bias(case, gen)
    if case["kind"] != "serve":
        s["off"] = _offsets(case, gen)
    if case["kind"] in ("train", "router", "dp"):
        s["g"] = _grad(case, gen) if case.get("grad", True) else None
    if case["kind"] == "compare":
        s["g"] = _grad(case, gen).mul_(1.0 / T)  # a mean loss's gradient, as the auxiliary loss is a mean
        v, idx = (s["z"].float() + s["b"]).topk(K + 1, dim=1)
        s["tau"] = v[:, K].contiguous()
        s["loads"] = _loads(idx[:, :K], s["off"], E).to(torch.int32)
        s["shards"] = [(T * p) // case["P"] for p in range(case["P"] + 1)]
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    T, E, K, kind = case["T"], case["E"], case["K"], case["kind"]

    def new(shape, dtype):
        return torch.zeros(shape, dtype=dtype, device="cuda")

    s["err"] = new(1, torch.int32)
    if kind == "compare":
        s["avg_ws"] = new(eqb.eqb_rank_averaged_workspace_bytes(E, case["P"]), torch.uint8)
        s["fix_ws"] = new(eqb.eqb_layer_workspace_bytes(E), torch.uint8)
        s["avg_b"], s["avg_q"] = new(E, torch.float32), new((case["P"], E), torch.bfloat16)
        s["fix_b"], s["fix_q"] = new(E, torch.float32), new(E, torch.float64)
        s["vio"], s["vio_mb"] = new(2, torch.float64), new(case["M"], torch.float64)
        return s
    s["idx"], s["tau"] = new((T, K), torch.int32), new(T, torch.float32)
    if kind in ("router", "serve"):
        s["z"] = new((T, E), torch.bfloat16)
    if kind != "serve":
        s["loads"], s["b_next"] = new((case["M"], E), torch.int32), new(E, torch.float32)
    if kind in ("train", "router"):
        s["ws"] = new(eqb.eqb_layer_workspace_bytes(E), torch.uint8)
    elif kind == "dp":
        s["ws"] = eqb.EqbWorkspace(E)
    return s


def run(s):
    case = s["case"]
    kind, K, E = case["kind"], case["K"], case["E"]
    if kind == "train":
        eqb.eqb_layer_step(s["z"], s["b"], K, s["off"], s["loads"], s["b_next"], s["ws"], tau=s["tau"],
                           topk_idx=s["idx"], grad_s=s["g"], eta=ETA, c=C, err_flag=s["err"])
        return {k: s[k] for k in ("idx", "tau", "loads", "b_next", "g", "err")}
    if kind == "router":
        eqb.eqb_router_layer_step(s["x"], s["W"], s["b"], K, s["off"], s["loads"], s["b_next"], s["ws"], z=s["z"],
                                  tau=s["tau"], topk_idx=s["idx"], grad_s=s["g"], eta=ETA, c=C, err_flag=s["err"])
        return {k: s[k] for k in ("z", "idx", "tau", "loads", "b_next", "g", "err")}
    if kind == "serve":
        if E in (64, 128) and K <= 8:
            eqb.eqb_router_route(s["x"], s["W"], s["b"], K, z=s["z"], topk_idx=s["idx"], tau=s["tau"],
                                 err_flag=s["err"])
        else:
            eqb.eqb_router_logits(s["x"], s["W"], z=s["z"], err_flag=s["err"])
            eqb.eqb_route_topk(s["z"], s["b"], K, topk_idx=s["idx"], tau=s["tau"], err_flag=s["err"])
        return {k: s[k] for k in ("z", "idx", "tau", "err")}
    if kind == "dp":
        s["loads"].zero_()
        eqb.eqb_layer_forward(s["z"], s["b"], K, s["off"], s["ws"], s["idx"], s["tau"], s["loads"], s["b_next"])
        eqb.lei_inject_grad(s["g"], s["loads"], s["off"], K, ETA, C)
        ws = s["ws"]
        return {"idx": s["idx"], "tau": s["tau"], "loads": s["loads"], "b_next": s["b_next"], "g": s["g"],
                "err": ws.err, "hist_hi": ws.hist_hi, "hist_lo": ws.hist_lo, "q_hat": ws.q_hat}
    eqb.gshard_inject_grad(s["g"], s["z"], s["loads"], s["off"], K, ALPHA)
    eqb.eqb_rank_averaged_bias(s["z"], s["tau"], K, s["shards"], s["avg_ws"], b_out=s["avg_b"], q_shards=s["avg_q"],
                               err_flag=s["err"])
    eqb.eqb_fixed_hist_bias(s["z"], s["tau"], K, BIN_LO, BIN_W, s["fix_ws"], b_out=s["fix_b"], estimate=s["fix_q"],
                            err_flag=s["err"])
    eqb.eqb_maxvio(s["loads"], s["off"], K, out=s["vio"], per_mb=s["vio_mb"])
    return {k: s[k] for k in ("g", "avg_b", "avg_q", "fix_b", "fix_q", "vio", "vio_mb", "err")}


def work(case):
    """Bytes: every input read once, every output written once (gradients
    both).  Operations: the projection's multiply-adds, else one addition
    and one comparison per logit."""
    T, E, K, kind = case["T"], case["E"], case["K"], case["kind"]
    small = 8 * E + 4 * E * case.get("M", 0)
    route = T * (4 * K + 4)
    grad = 8 * T * E if case.get("grad", True) else 0
    if kind in ("router", "serve"):
        d = case["d"]
        return {"bytes": 2 * T * d + 2 * E * d + 2 * T * E + route + small + (grad if kind == "router" else 0),
                "flops": 2 * T * E * d}
    if kind == "compare":
        return {"bytes": 10 * T * E + 4 * T + small + 2 * E * case["P"], "flops": 4 * T * E}
    return {"bytes": 2 * T * E + route + grad + small + (2048 * E if kind == "dp" else 0), "flops": 2 * T * E}


def tolerance(case):
    """From logits in hand everything but the gradients is fixed bit for bit
    by the method's definition; a gradient takes one fp32 addition of a
    coefficient that is itself rounded to fp32 (2.8e-8 from 64 bits).  From
    the router input the projection may sum in another order: with K in four
    parts, 0.02% to 0.26% of the logits round to the other bf16 neighbour
    (rel 1.6e-4, max 7.8e-3 of the result), and 1.6e-4 of the indices change
    places; four times that, and at least a swapped pair."""
    kind = case["kind"]
    if kind in ("router", "serve"):
        return {"rel": 7e-4, "max": 3.1e-2, "differ": max(7e-4, min(0.5, 2.0 / (case["T"] * case["K"])))}
    return {"rel": 1.2e-7, "max": 1e-6}


# ---------------------------------------------------------------- 64 bits

def _loads(idx, off, E):
    """int64 [M,E]: how often each microbatch's tokens chose each expert."""
    T, M = idx.shape[0], off.numel() - 1
    mb = torch.searchsorted(off[1:].contiguous(), torch.arange(T, device="cuda"), right=True)
    return torch.bincount((mb[:, None] * E + idx).reshape(-1), minlength=M * E).view(M, E)


def _route64(z, b, K):
    """Top-K experts (ties to the lower index) and the cutoff of the scores,
    which the method defines as z + b rounded to fp32."""
    T = z.shape[0]
    idx = torch.empty((T, K), dtype=torch.int64, device="cuda")
    tau = torch.empty(T, dtype=torch.float64, device="cuda")
    for t in range(0, T, 1 << 18):
        s = (z[t:t + (1 << 18)].double() + b.double()).float()
        v, i = s.sort(dim=1, descending=True, stable=True)
        idx[t:t + (1 << 18)] = i[:, :K]
        tau[t:t + (1 << 18)] = v[:, K].double()
    return idx, tau


def _margins64(z, tau):
    """tau_t - z_{t,e} as [E,T], rounded through fp32 to bf16: what the method
    takes its quantiles of."""
    T, E = z.shape
    m = torch.empty((E, T), dtype=torch.float32, device="cuda")
    for t in range(0, T, 1 << 18):
        d = tau[t:t + (1 << 18), None] - z[t:t + (1 << 18)].double()
        m[:, t:t + (1 << 18)] = d.float().to(torch.bfloat16).float().t()
    return m


def _kth(m, r):
    return torch.stack([m[e].kthvalue(r).values for e in range(m.shape[0])]).double()


def _lei64(g, loads, off, K):
    """g + eta sigma rho, in 64 bits."""
    E = g.shape[1]
    n = (off[1:] - off[:-1]).double()
    rho = loads.double() * E / (K * n.clamp(min=1.0))[:, None] - 1.0
    xi = rho.abs().max(dim=1, keepdim=True).values / C
    coef = ETA * torch.where(xi > 0, torch.tanh(xi) / xi, torch.ones_like(xi)) * rho
    out = g.double()
    for l in range(n.numel()):
        out[int(off[l]):int(off[l + 1])] += coef[l]
    return out


def exact(case, seed):
    kind, T, E, K = case["kind"], case["T"], case["E"], case["K"]
    s = _inputs(case, seed)
    if kind in ("router", "serve"):
        z = torch.empty((T, E), dtype=torch.float64, device="cuda")
        for t in range(0, T, 1 << 16):
            z[t:t + (1 << 16)] = s["x"][t:t + (1 << 16)].double() @ s["W"].double().t()
        zr = z.to(torch.bfloat16)  # the logits that routing and the quantiles are defined on
        idx, tau = _route64(zr, s["b"], K)
        if kind == "serve":
            return {"z": z, "idx": idx, "tau": tau, "err": None}
        loads = _loads(idx, s["off"], E)
        q = _kth(_margins64(zr, tau), -(-T * K // E))
        return {"z": z, "idx": idx, "tau": tau, "loads": loads, "b_next": q - q.mean(),
                "g": None if s["g"] is None else _lei64(s["g"], loads, s["off"], K), "err": None}
    z = s["z"]
    if kind in ("train", "dp"):
        idx, tau = _route64(z, s["b"], K)
        loads = _loads(idx, s["off"], E)
        q = _kth(_margins64(z, tau), -(-T * K // E))
        out = {"idx": idx, "tau": tau, "loads": loads, "b_next": q - q.mean(),
               "g": None if s["g"] is None else _lei64(s["g"], loads, s["off"], K), "err": None}
        if kind == "dp":
            out.update({"hist_hi": None, "hist_lo": None, "q_hat": q})
        return out
    off, P = s["off"], case["P"]
    n = (off[1:] - off[:-1]).double()
    R = s["loads"].double() / (K * n.clamp(min=1.0))[:, None] - 1.0 / E
    g = s["g"].double()
    for l in range(case["M"]):
        a, e = int(off[l]), int(off[l + 1])
        for t in range(a, e, 1 << 18):
            u = min(e, t + (1 << 18))
            p = torch.sigmoid(z[t:u].double())
            d = p.sum(dim=1, keepdim=True)
            g[t:u] += ALPHA / (n[l] * d) * (R[l] - (p * R[l]).sum(dim=1, keepdim=True) / d)
    m = _margins64(z, s["tau"].double())
    cut = s["shards"]
    some = [p for p in range(P) if cut[p + 1] > cut[p]]
    q = torch.zeros((P, E), dtype=torch.float64, device="cuda")
    for p in some:
        q[p] = _kth(m[:, cut[p]:cut[p + 1]], -(-(cut[p + 1] - cut[p]) * K // E))
    avg = q[some].mean(dim=0)
    kth = _kth(m, -(-T * K // E))
    est = BIN_LO + (((kth - BIN_LO) / BIN_W).floor().clamp(0, 255) + 1.0) * BIN_W
    nz = n > 0
    mb = torch.where(nz, s["loads"].double().max(dim=1).values * E / (K * n.clamp(min=1.0)) - 1.0, n.new_zeros(()))
    vio = torch.stack([s["loads"].double().sum(dim=0).max() * E / (K * T) - 1.0, mb[nz].mean()])
    return {"g": g, "avg_b": avg - avg.mean(), "avg_q": q, "fix_b": est - est.mean(), "fix_q": est, "vio": vio,
            "vio_mb": mb, "err": None}
