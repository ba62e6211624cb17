"""What is measured: one pass of each way in which a program uses the logits-side path.

A case is a dict of plain values.  `kind` says which entry points a pass goes through:

  round       one fused round (BlockRound.run): confidence, schedule and every acceptance rule of one batch of blocks
  pipeline    a queue of independent batches through block_pipelined (the benchmark's form)
  confidence  the pre-verify half alone (confidence, with or without the learned scorer's row features)
  verify      the post-verify half alone, one acceptance rule over the blocks that were not skipped
  loop        one round of the decode loop (DecodeLoop.step): confidence, learned scorer, schedules, verifier pass, commit
  mlp, deep   the survival scorers on a batch of hidden states
  shard       the vocabulary-sharded round, its ranks played in turn on one GPU (vocab_shard.run_local)
  diag        the offline diagnostics over a log of verified blocks

B blocks of gamma drafted positions; logits over V tokens.  Rows lie 16 bytes apart at the least, so an odd V sits in a
padded row, as the output of a padded language-model head does.
"""
import math

import torch

import paper_2608_14787_gb300 as sdd
from paper_2608_14787_gb300 import binding, loop, synth, vocab_shard

V_FULL = synth.QWEN_VOCAB      # 151,936
MOST_LOGITS = 2.6e9            # bytes of logits of the largest round below
TAUS16 = synth.WORKLOADS["c4"].taus


def listed():
    return [
        # One small draft block in fp32: nothing but latency (the smallest workload of the benchmark).
        {"name": "round 1x8x32000 f32", "kind": "round", "rows": "tiny", "B": 1, "gamma": 8, "V": 32000, "dtype": "f32",
         "taus": 1, "rules": 0, "greedy": False, "signal": "raw", "masked": 0},
        # Batch size 1 at the paper's block length and vocabulary: the interactive setting.
        {"name": "round 1x32x151936", "kind": "round", "rows": "temp", "B": 1, "gamma": 32, "V": V_FULL, "dtype": "bf16",
         "taus": 3, "rules": 0, "greedy": False, "signal": "raw", "masked": 0},
        # fp32 logits of a smaller, odd vocabulary with the unused ids masked; greedy verification, lenience and top-k.
        {"name": "round 24x17x32003 f32 greedy", "kind": "round", "rows": "runs", "B": 24, "gamma": 17, "V": 32003,
         "dtype": "f32", "taus": 1, "rules": 3, "greedy": True, "signal": "marginal", "masked": 203},
        # The largest round: 64 blocks of 64 positions, a grid of 16 thresholds (a threshold sweep's shadow verification).
        {"name": "round 64x64x151936", "kind": "round", "rows": "runs", "B": 64, "gamma": 64, "V": V_FULL, "dtype": "bf16",
         "taus": 16, "rules": 0, "greedy": False, "signal": "raw", "masked": 0},
        # The benchmark's workload: batches of 16 blocks, all rules, queued through the pipelined call.
        {"name": "pipeline 4 x 16x32x151936", "kind": "pipeline", "rows": "runs", "n": 4, "B": 16, "gamma": 32, "V": V_FULL,
         "dtype": "bf16", "taus": 1, "rules": 3, "greedy": False, "signal": "raw", "masked": 0},
        # The pre-verify half with the learned scorer's row statistics, for the same batch.
        {"name": "confidence 16x32x151936 feat", "kind": "confidence", "rows": "runs", "B": 16, "gamma": 32, "V": V_FULL,
         "dtype": "bf16", "features": True, "masked": 0},
        # The post-verify half: top-k acceptance of the blocks that the schedule did not skip, odd vocabulary.
        {"name": "verify 128x32x151665 top-k", "kind": "verify", "rows": "runs", "B": 128, "gamma": 32, "V": 151665,
         "dtype": "bf16", "rule": "topk", "share": 0.36, "masked": 0},
        # One round of the decode loop at the benchmark's batch (63 % of its verifier calls are skipped).
        {"name": "loop 128x32x151936", "kind": "loop", "rows": "runs", "B": 128, "gamma": 32, "V": V_FULL, "dtype": "bf16",
         "masked": 0},
        # The one-layer survival scorer on the decode loop's batch of positions.
        {"name": "mlp 4096x3584", "kind": "mlp", "M": 4096, "K": synth.HIDDEN},
        # The learned scorer's full shape over a log of positions (an offline pass over stored hidden states).
        {"name": "deep 20000x3584", "kind": "deep", "M": 20000, "K": synth.HIDDEN},
        # The benchmark's batch with its vocabulary split over two ranks of a tensor-parallel head.
        {"name": "shard 2 of 16x32x151936", "kind": "shard", "rows": "runs", "S": 2, "B": 16, "gamma": 32, "V": V_FULL,
         "dtype": "bf16", "rules": 3, "greedy": False, "masked": 0},
        # Permutation test and positionwise metrics on the log of an evaluation run (about 160 problems of 13 blocks).
        {"name": "diag 2048x32 x100", "kind": "diag", "B": 2048, "gamma": 32, "n_rep": 100, "signal": "raw"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["round", "round", "round", "pipeline", "confidence", "verify", "loop", "mlp", "deep", "shard", "diag"])
    if kind in ("mlp", "deep"):
        return {"kind": kind, "M": _log_int(rng, 32, 20000), "K": 64 * rng.choice([32, 48, 55, 56, 60, 64])}
    if kind == "diag":
        return {"kind": kind, "B": _log_int(rng, 64, 2048), "gamma": rng.randint(8, 32), "n_rep": rng.randint(20, 100),
                "signal": rng.choice(["raw", "marginal", "conditional"])}
    c = {"kind": kind, "rows": rng.choice(["runs", "runs", "temp"]), "gamma": _log_int(rng, 4, 64),
         "V": _log_int(rng, 8000, V_FULL), "dtype": rng.choice(["bf16", "bf16", "f32"]),
         "masked": rng.choice([0, 0, rng.randint(1, 500)])}
    if kind == "loop":
        c["dtype"] = "bf16"
    esz = 2 if c["dtype"] == "bf16" else 4
    most = MOST_LOGITS / (2 if kind == "shard" else 4 if kind == "pipeline" else 1)
    B = max(1, min(128, int(most / ((2 * c["gamma"] + 1) * c["V"] * esz))))
    c["B"] = _log_int(rng, 1, B)
    if kind in ("round", "pipeline"):
        c.update(taus=rng.choice([1, 3, 16]), rules=rng.choice([0, 1, 3]), greedy=rng.random() < 0.3,
                 signal=rng.choice(["raw", "raw", "marginal", "conditional"]))
        if kind == "pipeline":
            c["n"] = rng.randint(2, 4)
    elif kind == "shard":
        c.update(S=rng.randint(2, 4), rules=rng.choice([0, 3]), greedy=rng.random() < 0.3)
    elif kind == "confidence":
        c["features"] = rng.random() < 0.5
    elif kind == "verify":
        c.update(rule=rng.choice(["strict", "greedy", "lenient", "topk"]), share=rng.uniform(0.2, 1.0))
    return c


# --- inputs -----------------------------------------------------------------------------------------------------------


def _dtype(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


def _padded(z, masked):
    """z with rows 16-byte aligned (a view of a padded tensor where V needs it) and the last `masked` ids masked."""
    if masked:
        z[..., z.shape[-1] - masked:] = -math.inf
    q = 16 // z.element_size()
    V = z.shape[-1]
    if V % q == 0:
        return z
    out = torch.zeros(*z.shape[:-1], -(-V // q) * q, dtype=z.dtype, device=z.device)
    out[..., :V] = z
    return out[..., :V]


def _block(case, seed):
    """(z_d [B, gamma, V], z_t [B, gamma + 1, V], x [B, gamma]): drafter and target logits and the drafted tokens."""
    wl = {"tiny": "tiny", "temp": "c2", "runs": "c3"}[case["rows"]]
    blk = synth.make_block(wl, device="cuda", round_=int(seed), B=case["B"], gamma=case["gamma"],
                           V=case["V"] - case["masked"], dtype=_dtype(case))
    if not case["masked"]:
        return _padded(blk.z_d, 0), _padded(blk.z_t, 0), blk.x
    wide = [torch.empty(*z.shape[:-1], case["V"], dtype=z.dtype, device="cuda") for z in (blk.z_d, blk.z_t)]
    for w, z in zip(wide, (blk.z_d, blk.z_t)):
        w[..., :z.shape[-1]] = z
    return _padded(wide[0], case["masked"]), _padded(wide[1], case["masked"]), blk.x


def _taus(n):
    return {1: (0.9,), 3: (0.8, 0.9, 0.95), 16: TAUS16}[n]


def _rules(n):
    """Lenience factors (the paper's convention) and top-k sizes: the benchmark's grids, cut to n entries each."""
    return (1 / 1.5, 0.5, 0.25)[:n], (2, 5, 10)[:n]


_SIGNALS = {"raw": sdd.SIG_RAW, "marginal": sdd.SIG_MARGINAL, "conditional": sdd.SIG_CONDITIONAL}


def _round(case, seed):
    z_d, z_t, x = _block(case, seed)
    ells, ks = _rules(case["rules"])
    rnd = sdd.BlockRound(case["B"], case["gamma"], case["V"], dtype=_dtype(case), taus=_taus(case["taus"]), ells=ells,
                         ks=ks, greedy=case["greedy"], signal=_SIGNALS[case["signal"]])
    return {"rnd": rnd, "z_d": z_d, "z_t": z_t, "x": x, "seed": int(seed)}


def _log(case, seed):
    """Scores q and strict accepted lengths L of a log: a block-level difficulty shared by its positions, and positionwise
    noise; a position is accepted with about its score's probability."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    B, gamma = case["B"], case["gamma"]
    shared = torch.randn(B, 1, generator=g, device="cuda") * 1.5 + 2.5
    q = torch.sigmoid(shared + 1.5 * torch.randn(B, gamma, generator=g, device="cuda"))
    ok = torch.rand(B, gamma, generator=g, device="cuda") < q
    return q, ok.int().cumprod(1).sum(1).to(torch.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "round":
        return {"kind": kind, **_round(case, seed)}
    if kind == "pipeline":
        return {"kind": kind, "rounds": [_round(case, 16 * int(seed) + i) for i in range(case["n"])]}
    if kind == "confidence":
        z_d, _, x = _block(case, seed)
        B, gamma, f = case["B"], case["gamma"], case["features"]
        return {"kind": kind, "z_d": z_d, "x": x, "features": f, "ws": sdd.Workspace(B, gamma, case["V"]),
                "status": sdd.new_status(), "out": sdd.confidence_buffers(B, gamma, z_d.device, f)}
    if kind == "verify":
        z_d, z_t, x = _block(case, seed)
        B, gamma = case["B"], case["gamma"]
        g = torch.Generator().manual_seed(int(seed))
        n = max(1, int(case["share"] * B))
        rows = torch.randperm(B, generator=g)[:n].sort().values.to(torch.int32).cuda()
        s = {"kind": kind, "rule": case["rule"], "z_t": z_t, "x": x, "rows": rows, "seed": int(seed),
             "ws": sdd.Workspace(B, gamma, case["V"]), "status": sdd.new_status()}
        if case["rule"] == "strict":
            s.update(z_d=z_d, draft=sdd.confidence(z_d, x))
        return s
    if kind == "loop":
        z_d, z_t, x = _block(case, seed)
        B, gamma = case["B"], case["gamma"]
        h = synth.make_hidden(B * gamma, device="cuda", round_=int(seed))
        return {"kind": kind, "loop": loop.DecodeLoop(B, gamma, case["V"]), "z_d": z_d, "z_t": z_t, "x": x, "h": h, "r": 0}
    if kind == "mlp":
        W1, b1, w2, b2 = synth.make_mlp(device="cuda", hidden=case["K"])
        return {"kind": kind, "h": synth.make_hidden(case["M"], device="cuda", round_=int(seed), hidden=case["K"]),
                "w": (W1, b1, w2, float(b2.item())), "ws": binding.scorer_workspace(case["M"], "cuda"),
                "out": torch.empty(case["M"], device="cuda")}
    if kind == "deep":
        M = case["M"]
        return {"kind": kind, "h": synth.make_hidden(M, device="cuda", round_=int(seed), hidden=case["K"]),
                "f": synth.make_features(M, device="cuda", round_=int(seed)),
                "w": synth.make_scorer_deep(device="cuda", hidden=case["K"]),
                "act": torch.empty(M, binding.MLP_HIDDEN, dtype=torch.bfloat16, device="cuda"),
                "ws": binding.scorer_workspace(M, "cuda"), "out": torch.empty(M, device="cuda")}
    if kind == "shard":
        z_d, z_t, x = _block(case, seed)
        ells, ks = _rules(case["rules"])
        cuts = vocab_shard.slice_bounds(case["V"], case["S"])
        ranks = [vocab_shard.ShardRound(case["B"], case["gamma"], case["V"], v0, v1, dtype=_dtype(case), ells=ells, ks=ks,
                                        greedy=case["greedy"]) for v0, v1 in cuts]
        return {"kind": kind, "ranks": ranks, "x": x, "seed": int(seed),
                "zd": [vocab_shard.slice_logits(z_d, *c) for c in cuts],
                "zt": [vocab_shard.slice_logits(z_t, *c) for c in cuts]}
    if kind == "diag":
        q, L = _log(case, seed)
        return {"kind": kind, "q": q, "L": L, "seed": int(seed), "signal": case["signal"], "n_rep": case["n_rep"]}
    raise ValueError(kind)


# --- one pass ---------------------------------------------------------------------------------------------------------

_FLOATS = ("q", "logq", "maxprob", "lse", "entropy")
_WHOLE = ("argmax", "K_hat", "K", "D_out", "L_strict", "tokens_strict", "n_strict", "commit_tokens", "commit_n")


def _outputs(r):
    a = r.args
    out = {n: getattr(r, n) for n in _FLOATS + _WHOLE + ("agreement",)}
    if a.n_ell:
        out.update(L_lenient=r.L_lenient, tokens_lenient=r.tokens_lenient, n_lenient=r.n_lenient)
    if a.n_k:
        out.update(L_topk=r.L_topk, tokens_topk=r.tokens_topk, n_topk=r.n_topk)
    return out


def run(s):
    kind = s["kind"]
    if kind == "round":
        r = s["rnd"]
        r.set_inputs(s["z_d"], s["z_t"], s["x"], seed=s["seed"])
        r.run()
        return _outputs(r)
    if kind == "pipeline":
        prev = None
        for q in s["rounds"]:
            q["rnd"].set_inputs(q["z_d"], q["z_t"], q["x"], seed=q["seed"])
            sdd.block_pipelined(q["rnd"], prev)
            prev = q["rnd"]
        sdd.block_pipelined(None, prev)
        # (the agreement counters of the whole queue and the per-round results that a decoder goes on with)
        keep = _FLOATS + ("K", "D_out", "L_strict", "tokens_strict", "commit_tokens", "commit_n", "agreement")
        return [{n: getattr(q["rnd"], n) for n in keep} for q in s["rounds"]]
    if kind == "confidence":
        c = sdd.confidence(s["z_d"], s["x"], ws=s["ws"], status=s["status"], features=s["features"], out=s["out"])
        out = {n: getattr(c, n) for n in _FLOATS + ("argmax",)}
        if s["features"]:
            out.update(margin=c.margin, top5=c.top5)
        return out
    if kind == "verify":
        kw = dict(rows=s["rows"], ws=s["ws"], status=s["status"])
        if s["rule"] == "strict":
            return sdd.verify_strict(s["z_t"], s["x"], z_d=s["z_d"], draft=s["draft"], seed=s["seed"], **kw)
        if s["rule"] == "greedy":
            return sdd.verify_strict(s["z_t"], s["x"], greedy=True, **kw)
        if s["rule"] == "lenient":
            return sdd.verify_lenient(s["z_t"], s["x"], _rules(3)[0], **kw)
        return sdd.verify_topk(s["z_t"], s["x"], _rules(3)[1], **kw)
    if kind == "loop":
        o = s["loop"].step(s["z_d"], s["z_t"], s["x"], s["h"], round_=s["r"])
        s["r"] += 1
        return {n: getattr(o, n) for n in ("score", "K_raw", "K_mlp", "K_per", "L", "tokens", "n", "n_verified")}
    if kind == "mlp":
        return binding.survival_mlp(s["h"], *s["w"], workspace=s["ws"], out=s["out"])
    if kind == "deep":
        return binding.scorer_deep(s["h"], s["f"], *s["w"], act=s["act"], workspace=s["ws"], out=s["out"])
    if kind == "shard":
        vocab_shard.run_local(s["ranks"], s["zd"], s["zt"], s["x"], seed=s["seed"])
        return _outputs(s["ranks"][0])
    sums = binding.permutation_diagnostic(s["q"], s["L"], signal=_SIGNALS[s["signal"]], n_rep=s["n_rep"], seed=s["seed"])
    m = binding.position_metrics(s["q"], s["L"], conditional=s["signal"] == "conditional")
    return (sums, *m)


# --- what a pass cannot do without, and how exact it is ----------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("mlp", "deep"):
        M, K, H = case["M"], case["K"], binding.MLP_HIDDEN
        K1 = K + (H if kind == "deep" else 0)
        layers = 2 * H * H if kind == "deep" else 0
        return {"bytes": 2 * M * K1 + 2 * H * K1 + 2 * layers + 4 * M, "flops": 2 * M * (H * K1 + layers + H)}
    if kind == "diag":
        # every (repetition, position, block): a partner's draw (ten Philox rounds), a move and the gates
        B, gamma = case["B"], case["gamma"]
        return {"bytes": 4 * B * (gamma + 1) + 8 * case["n_rep"], "flops": case["n_rep"] * gamma * B * 100}
    B, gamma, V = case["B"], case["gamma"], case["V"]
    esz = 2 if case["dtype"] == "bf16" else 4
    drafter, target = B * gamma * V * esz, B * (gamma + 1) * V * esz
    outs = B * gamma * 28
    if kind == "confidence":
        nbytes = drafter + outs
    elif kind == "verify":
        nbytes = int(max(1, int(case["share"] * B)) * (target + (V * esz if case["rule"] == "strict" else 0)) / B)
    elif kind == "loop":
        # the verifier reads the blocks that were not skipped: about 0.36 of them
        nbytes = drafter + int(0.36 * target) + B * gamma * (2 * synth.HIDDEN + 512) + outs
    else:
        nbytes = (drafter + target + outs) * case.get("n", 1)
    # one exponential and its two sums for each logit
    return {"bytes": nbytes, "flops": 4 * nbytes // esz + (2 * B * gamma * 256 * 4352 if kind == "loop" else 0)}


def tolerance(case):
    kind = case["kind"]
    if kind == "verify":
        return "exact"
    if kind in ("deep", "loop"):
        return {"rel": 1e-4, "max": 1e-3}      # activations rounded to bf16 between layers: 2e-5 off 64 bits
    if kind == "mlp":
        return {"rel": 2e-6, "max": 2e-5}      # fp32 sums of 3,584 exact products: 1e-7
    if kind == "diag":
        return {"rel": 1e-13, "max": 1e-12}    # fp64 sums: 1e-16
    # fp32 statistics of given logits: 3e-7; decisions and tokens are whole numbers and stay the same
    return {"rel": 2e-6, "max": 2e-5}


def _stats64(z, x, features=False):
    """Row statistics of logits z [B, G, V] and tokens x [B, G] in 64 bits."""
    out = {n: torch.empty(x.shape, dtype=torch.float64, device=z.device) for n in _FLOATS + ("margin", "top5")}
    for b in range(z.shape[0]):
        zb = z[b].double()
        lse = torch.logsumexp(zb, -1, keepdim=True)
        lp = zb - lse
        p = lp.exp()
        out["lse"][b] = lse[:, 0]
        out["logq"][b] = lp.gather(1, x[b].long().unsqueeze(1))[:, 0]
        out["q"][b] = out["logq"][b].exp()
        out["maxprob"][b] = p.amax(-1)
        out["entropy"][b] = -torch.where(p > 0, p * lp, p).sum(-1)
        if features:
            top = p.topk(5, -1).values
            out["margin"][b], out["top5"][b] = top[:, 0] - top[:, 1], top.sum(-1)
    return out


def _gelu64(z):
    return 0.5 * z * (1 + torch.erf(z / math.sqrt(2)))


def _deep64(u, w):
    W1, b1, W2, b2, W3, b3, w4, b4 = w
    for W, b in ((W1, b1), (W2, b2), (W3, b3)):
        u = _gelu64(u @ W.double().T + b.double())
    return torch.sigmoid(u @ w4.double() + b4)


def _metrics64(q, L, conditional):
    B, gamma = q.shape
    q, L = q.double().cpu(), L.cpu()
    bce, base, auroc = (torch.full((gamma,), math.nan, dtype=torch.float64) for _ in range(3))
    for j in range(gamma):
        valid = L >= j if conditional else torch.ones(B, dtype=torch.bool)
        y, s = (L >= j + 1)[valid], q[valid, j]
        if not len(s):
            continue
        c = s.clamp(1e-7, 1 - 1e-7)
        bce[j] = -torch.where(y, c.log(), torch.log1p(-c)).mean()
        r = y.double().mean()
        base[j] = -(r * r.log() + (1 - r) * torch.log1p(-r)) if 0 < r < 1 else 0.0
        pos, neg = s[y], s[~y]
        if len(pos) and len(neg):
            d = pos[:, None] - neg[None, :]
            auroc[j] = ((d > 0).double() + 0.5 * (d == 0).double()).mean()
    return bce, base, auroc


def exact(case, seed):
    """The floating outputs of a pass in 64 bits (the whole-number ones follow from thresholds and draws: None)."""
    kind = case["kind"]
    if kind == "verify":
        return None
    s = prepare(case, seed)
    if kind == "mlp":
        W1, b1, w2, b2 = s["w"]
        return torch.sigmoid(_gelu64(s["h"].double() @ W1.double().T + b1.double()) @ w2.double() + b2)
    if kind == "deep":
        return _deep64(torch.cat([s["h"], s["f"]], 1).double(), s["w"])
    if kind == "diag":
        return (None, *_metrics64(s["q"], s["L"], case["signal"] == "conditional"), None, None)
    if kind == "pipeline":
        return [{n: v for n, v in _stats64(q["z_d"], q["x"]).items() if n in _FLOATS} for q in s["rounds"]]
    if kind == "loop":
        st = _stats64(s["z_d"], s["x"], True)
        B, gamma = s["x"].shape
        f = torch.zeros(B, gamma, binding.MLP_HIDDEN, dtype=torch.float64, device="cuda")
        f[..., 4], f[..., 5] = st["maxprob"], st["maxprob"].log()
        f[..., 6], f[..., 7], f[..., 8], f[..., 9] = st["entropy"], -st["entropy"], st["margin"], st["top5"]
        f[..., 14] = torch.arange(gamma, device="cuda") / gamma      # block position; generated length 0 in round 0
        u = torch.cat([s["h"].double(), f.reshape(B * gamma, -1)], 1)
        return {"score": _deep64(u, s["loop"].deep).reshape(B, gamma)}
    if kind == "shard":
        z_d = torch.cat(s["zd"], -1)
        return {n: v for n, v in _stats64(z_d, s["x"]).items() if n in _FLOATS}
    feat = kind == "confidence" and case["features"]
    return {n: v for n, v in _stats64(s["z_d"], s["x"], feat).items() if feat or n in _FLOATS}
