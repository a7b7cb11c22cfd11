"""What the performance of this library is measured on.

Every case is one call (or, for the report, two) of the Python binding, as a
reinforcement-learning trainer makes it: the fused loss and its gradient from
logits or from hidden states, the rescoring of sampled tokens, the mismatch
diagnostics and the confidence-binned report.  Sizes are those of the synthetic
workloads, the tests and the benchmark, with odd ones beside them.

Families (a case's "family"):
  pass         cis_loss_fwd_bwd: log-softmax, weight, loss and dlogits.
  logprobs     cis_token_logprobs: log p of the sampled tokens.
  lmhead       cis_lmhead_fused: the pass through the unembedding.
  diagnostics  cis_mismatch_diagnostics: both engines' full logits.
  report       cis_weights, then cis_binned_sums of its outputs.
"""
import math

import torch

from paper_2609_32444_gb300 import binding as B

DEV = "cuda"
LAM, KAPPA, TIS_CAP, ICEPOP, KPOP_PHI = 2.3, 5e-3, 2.0, (0.5, 5.0), 2.0
EXACT, SEQ_CAP, SEQ_MIS, CLIP = (1e-6, 1e6), 2.0, (0.5, 2.0), (0.2, 0.28)
TOKEN_MODES = ("cis", "tis", "exact", "none", "band", "icepop", "kpop")
# the operators that act on single candidates of these rows: the others' bias is zero
CANDIDATE_MODES = ("cis", "tis", "none", "band", "icepop")


def _pass(T, V, mode="cis", dtype="bf16", grad="bf16", pad=0.0, old=False, seq_mean=False,
          entropy=False, stats=True):
    return {"family": "pass", "T": T, "V": V, "mode": mode, "dtype": dtype, "grad": grad,
            "pad": pad, "old": old, "seq_mean": seq_mean, "entropy": entropy, "stats": stats}


def _logprobs(T, V, dtype="bf16", pad=0.0, lse=False, entropy=False):
    return {"family": "logprobs", "T": T, "V": V, "dtype": dtype, "pad": pad, "lse": lse,
            "entropy": entropy}


def _lmhead(T, V, H, mode="cis", grad="f32", pad=0.0, old=False):
    return {"family": "lmhead", "T": T, "V": V, "H": H, "mode": mode, "grad": grad, "pad": pad,
            "old": old}


def _diagnostics(T, V, mode="cis", dtype="bf16", pad=0.0):
    return {"family": "diagnostics", "T": T, "V": V, "mode": mode, "dtype": dtype, "pad": pad}


def _report(T, nbins=18, mode="cis", pad=0.0):
    return {"family": "report", "T": T, "nbins": nbins, "mode": mode, "pad": pad}


def listed():
    return [
        # the smallest step (workload 1, also the smoke test): a toy vocabulary in fp32,
        # where a call's own cost and its launches count; statistics are not looked at
        dict(_pass(256, 1024, dtype="f32", grad="f32", stats=False), name="pass_small"),
        # workload 2's size: responses of a padded batch, each response weighing the same
        dict(_pass(4096, 32000, pad=0.25, seq_mean=True), name="pass_padded"),
        # workload 3, the benchmark: a whole batch of a large vocabulary
        dict(_pass(16384, 151936), name="pass_batch"),
        # a vocabulary that tokens were added to, so that its rows are not aligned; a later
        # minibatch of the update (log p of the snapshot given, the clip at work)
        dict(_pass(4096, 32003, mode="tis", pad=0.25, old=True), name="pass_odd_vocab"),
        # fp32 logits and gradients with the binary-KL operator, the entropy logged
        dict(_pass(1024, 151936, mode="kpop", dtype="f32", grad="f32", entropy=True),
             name="pass_f32"),
        # a sequence operator, which needs every log p of a response before its weight
        dict(_pass(2048, 151936, mode="seq_tis", pad=0.25), name="pass_sequence"),
        # rescoring a rollout batch with the training engine (the old log-probabilities)
        dict(_logprobs(8192, 151936, lse=True, entropy=True), name="logprobs_batch"),
        # the tokens of one decoding step of a few dozen requests
        dict(_logprobs(24, 151936), name="logprobs_few"),
        # the fused head on a micro-batch
        dict(_lmhead(512, 151936, 2048), name="lmhead_micro"),
        # the fused head on workload 5's batch with workload 4's share of padding
        dict(_lmhead(16384, 151936, 2048, pad=0.4), name="lmhead_batch"),
        # the diagnostics of an evaluation batch, both engines' logits kept
        dict(_diagnostics(4096, 151936), name="diagnostics"),
        # the statistics of a training run's tokens by confidence: 18 logarithmic bins
        dict(_report(1000003, mode="band"), name="report"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng, lo=1000, hi=151936):
    v = _log_int(rng, lo, hi)
    return v if rng.random() < 0.3 else -(-v // 8) * 8  # most vocabularies are padded


def draw(rng):
    pad = rng.choice([0.0, 0.0, 0.25, 0.4])
    kind = rng.random()
    if kind < 0.45:
        V = _vocab(rng)
        dtype = rng.choice(["bf16", "bf16", "f32"])
        T = max(1, _log_int(rng, 8, min(16384, 1500000000 // V)))
        mode = rng.choice(["cis", "cis", "cis"] + list(TOKEN_MODES) + ["seq_tis", "seq_mis"])
        return _pass(T, V, mode, dtype, rng.choice([dtype, dtype, "bf16", "f32"]), pad,
                     rng.random() < 0.4, rng.random() < 0.3, rng.random() < 0.25)
    if kind < 0.6:
        V = _vocab(rng)
        return _logprobs(max(1, _log_int(rng, 4, min(16384, 1500000000 // V))), V,
                         rng.choice(["bf16", "bf16", "f32"]), pad, rng.random() < 0.5,
                         rng.random() < 0.4)
    if kind < 0.75:
        H = 256 * rng.choice([1, 2, 3, 4, 5, 8, 12, 16])
        V = _vocab(rng)
        T = max(16, _log_int(rng, 64, min(16384, 2500000000000 // (V * H))))
        return _lmhead(T, V, H, rng.choice(["cis", "cis", "tis", "exact", "kpop"]),
                       rng.choice(["f32", "f32", "bf16"]), pad, rng.random() < 0.4)
    if kind < 0.87:
        V = _vocab(rng)
        return _diagnostics(max(1, _log_int(rng, 16, min(8192, 600000000 // V))), V,
                            rng.choice(CANDIDATE_MODES), rng.choice(["bf16", "bf16", "f32"]),
                            pad)
    return _report(_log_int(rng, 2000, 4000000), rng.randint(5, 64), rng.choice(TOKEN_MODES), pad)


# ------------------------------------------------------------------ inputs
def _dtype(name):
    return torch.bfloat16 if name == "bf16" else torch.float32


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _slots(T, pad):
    """Responses' slots (start, valid length): slots of up to 256 tokens, right-padded so
    that round(pad T) tokens of the batch are padding, unevenly over the slots."""
    n = max(1, T // 256)
    start = [i * T // n for i in range(n + 1)]
    left, out = int(round(pad * T)), []
    for i in range(n):
        size, rest = start[i + 1] - start[i], n - i
        cut = left if rest == 1 else int(left / rest * (0.4 + 1.2 * ((i * 7 + 3) % 11) / 10.0))
        cut = max(left - (T - start[i + 1]), min(cut, left, size - 1 if rest > 1 else size))
        left -= cut
        out.append((start[i], size - cut))
    return start, out


def _valid(case):
    return case["T"] - int(round(case["pad"] * case["T"]))


def _batch(case, g):
    """Mask, response boundaries and advantages of a padded batch of responses: binary
    rewards normalised within groups of 8, so all tokens of a response share one."""
    T = case["T"]
    start, slots = _slots(T, case["pad"])
    n = len(slots)
    mask = torch.zeros(T, dtype=torch.uint8)
    for a, length in slots:
        mask[a:a + length] = 1
    r = (torch.rand(-(-n // 8) * 8, generator=g, device=DEV) < 0.5).double().view(-1, 8)
    adv = ((r - r.mean(1, keepdim=True)) / (r.std(1, keepdim=True) + 0.1)).view(-1)[:n] + 0.05
    cu = torch.tensor(start, dtype=torch.int32)
    size = (cu[1:] - cu[:-1]).long().to(DEV)
    return {"mask": mask.to(DEV) if case["pad"] > 0 else None, "cu": cu.to(DEV),
            "adv": adv.float().repeat_interleave(size)}


def _displaced(lp, g, scale=0.15):
    """The other engine's log-probability: the log-odds moved by N(0, scale^2), on 1% of
    the tokens by a heavy tail."""
    d = torch.randn(lp.shape, generator=g, device=DEV, dtype=torch.float64) * scale
    tail = torch.rand(lp.shape, generator=g, device=DEV) < 0.01
    u = torch.rand(lp.shape, generator=g, device=DEV, dtype=torch.float64).clamp(min=1e-3)
    d = torch.where(tail, 1.5 / u.sqrt() * torch.sign(d), d).clamp(-8, 8)
    logit = lp - torch.log(-torch.expm1(lp.clamp(max=-1e-9)))
    return (-torch.nn.functional.softplus(-(logit + d))).clamp(max=-1e-7).float()


def _confidence(n, g):
    """Probabilities of the sampled tokens: most near 1, the others over the whole range."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    high = torch.rand(n, generator=g, device=DEV) < 0.7
    return torch.where(high, 1 - torch.exp(-4.6 - 5 * u), torch.exp(-8 * u).clamp(max=0.999))


def _logits(case, g, both=False):
    """Rows of logits with a token of the wanted probability in each, that token (or, for a
    few rows, another one) as the sampled one, and its log p.  `both`: the inference
    engine's logits too, perturbed entry by entry, with a heavy tail (1% of the entries
    moved by up to 4 either way, the likely token of 30% of the rows lowered by 2)."""
    T, V, dt = case["T"], case["V"], _dtype(case["dtype"])
    z = torch.empty((T, V), dtype=dt, device=DEV)
    zi = torch.empty((T, V), dtype=dt, device=DEV) if both else None
    ids = torch.randint(0, V, (T,), generator=g, device=DEV)
    p = _confidence(T, g)
    spread = torch.exp(0.5 + torch.rand(T, generator=g, device=DEV)).view(-1, 1)
    other = torch.rand(T, generator=g, device=DEV) < 0.05
    lp = torch.empty(T, dtype=torch.float64, device=DEV)
    step = max(1, (1 << 28) // V)
    for a in range(0, T, step):
        b = min(T, a + step)
        x = torch.randn((b - a, V), generator=g, device=DEV) * spread[a:b]
        r = torch.arange(b - a, device=DEV)
        x[r, ids[a:b]] = (torch.logsumexp(x, 1).double() + torch.logit(p[a:b])).float()
        q = x.to(dt)
        z[a:b] = q
        if both:
            x[r, ids[a:b]] -= 2.0 * (torch.rand(b - a, generator=g, device=DEV) < 0.3)
            x += 0.15 * torch.randn(x.shape, generator=g, device=DEV)
            u = torch.rand(x.shape, generator=g, device=DEV)
            zi[a:b] = torch.where(u < 0.01, x + (800 * u - 4), x).to(dt)
        y = torch.where(other[a:b], (ids[a:b] + V // 2) % V, ids[a:b])
        ids[a:b] = y
        x = q.float()
        zy = x[r, y].double()
        x[r, y] = -math.inf
        lp[a:b] = -torch.nn.functional.softplus(torch.logsumexp(x, 1).double() - zy)
    return z, zi, ids.int(), lp


def _params(case):
    p = B.cis_default_params(case["mode"], lam=LAM, kappa=KAPPA)
    if case.get("seq_mean"):
        p.agg = B.CIS_AGG_SEQ_MEAN_TOKEN_MEAN
    return p


def prepare(case, seed):
    g = _gen(seed)
    s = {"case": case}
    fam, T = case["family"], case["T"]
    if fam == "report":
        p = _confidence(T, g)
        lp = torch.log(p).clamp(max=-1e-6)
        s["lp"], s["lp_infer"] = lp.float(), _displaced(lp, g)
        s["key"] = (-torch.expm1(lp)).float()
        s["mask"] = _batch(case, g)["mask"] if case["pad"] > 0 else None
        n = case["nbins"]
        s["edges"] = [10.0 ** (-6 + 6.0 * i / n) for i in range(n)] + [1.0]
        s["params"] = _params(case)
        return s
    s.update(_batch(case, g))
    if fam == "lmhead":
        V, H = case["V"], case["H"]
        s["ids"] = torch.randint(0, V, (T,), generator=g, device=DEV).int()
        w = torch.randn((V, H), generator=g, device=DEV) * 0.02
        s["weight"] = w.to(torch.bfloat16)
        wy = w[s["ids"].long()]
        del w
        lift = 4 + 16 * torch.rand((T, 1), generator=g, device=DEV)
        h = torch.randn((T, H), generator=g, device=DEV)
        s["hidden"] = (h + lift * wy / (wy * wy).sum(1, keepdim=True)).to(torch.bfloat16)
        del h, wy
        lp = torch.empty(T, dtype=torch.float64, device=DEV)
        step = max(1, (1 << 28) // V)
        for a in range(0, T, step):
            b = min(T, a + step)
            x = (s["hidden"][a:b] @ s["weight"].t()).float()
            lp[a:b] = torch.log_softmax(x, 1)[torch.arange(b - a, device=DEV),
                                              s["ids"][a:b].long()].double()
        lp = lp.clamp(max=-1e-6)
        s["params"] = _params(case)
    else:
        s["logits"], s["infer"], s["ids"], lp = _logits(case, g, fam == "diagnostics")
        if fam != "logprobs":
            s["params"] = _params(case)
    if fam in ("pass", "lmhead"):
        s["lp_old"] = _displaced(lp, g, 0.05) if case["old"] else None
        s["lp_infer"] = _displaced(lp, g)
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    fam = case["family"]
    if fam == "pass":
        o = B.cis_loss_fwd_bwd(s["logits"], s["ids"], s["lp_infer"], s["adv"], s["params"],
                               lp_old=s["lp_old"], mask=s["mask"], cu_seqlens=s["cu"],
                               dlogits_dtype=_dtype(case["grad"]), want_entropy=case["entropy"])
        out = {k: o[k] for k in ("dlogits", "lp", "w", "trunc", "entropy", "loss")}
        if case["stats"]:  # the logged sums (loss, excess) and counts (valid, truncated)
            out["sums"] = o["stats"].view(torch.float64)[:2]
            out["counts"] = o["stats"].view(torch.int64)[2:4]
        return out
    if fam == "logprobs":
        return B.cis_token_logprobs(s["logits"], s["ids"], mask=s["mask"], want_lse=case["lse"],
                                    want_entropy=case["entropy"])
    if fam == "lmhead":
        o = B.cis_lmhead_fused(s["hidden"], s["weight"], s["ids"], s["lp_infer"], s["adv"],
                               s["params"], lp_old=s["lp_old"], mask=s["mask"],
                               cu_seqlens=s["cu"], grad_dtype=_dtype(case["grad"]))
        return {k: o[k] for k in ("dhidden", "dweight", "lp", "w", "trunc", "loss")}
    if fam == "diagnostics":
        return B.cis_mismatch_diagnostics(s["logits"], s["infer"], s["ids"], s["params"],
                                          mask=s["mask"])
    w, trunc, eps = B.cis_weights(s["lp"], s["lp_infer"], s["params"], mask=s["mask"],
                                  want_eps=True)
    counts, sums = B.cis_binned_sums(s["key"], s["edges"], (w, eps), mask=s["mask"])
    return {"w": w, "trunc": trunc, "eps": eps, "counts": counts, "sums": sums}


def work(case):
    fam, T, n = case["family"], case["T"], _valid(case)
    size = {"bf16": 2, "f32": 4}
    if fam == "report":  # both log-probabilities; key, w and eps again; w, trunc and eps out
        return {"bytes": T * (8 + 9 + 12), "flops": 60 * T}
    V = case["V"]
    if fam == "pass":  # padding is only written
        return {"bytes": V * (n * size[case["dtype"]] + T * size[case["grad"]]) + 40 * T,
                "flops": 12 * n * V}
    if fam == "logprobs":
        return {"bytes": V * n * size[case["dtype"]] + 12 * T, "flops": 5 * n * V}
    if fam == "diagnostics":
        return {"bytes": 2 * V * n * size[case["dtype"]] + 28 * T, "flops": 50 * n * V}
    H = case["H"]
    return {"bytes": 2 * H * (n + V) + size[case["grad"]] * H * (T + V) + 30 * T,
            "flops": 6 * n * V * H}


def tolerance(case):
    fam = case["family"]
    if fam == "lmhead":  # dz enters the products in bf16
        return {"rel": 8e-3, "max": 0.5, "differ": 2e-3}
    if fam == "diagnostics":  # bias2 is a small difference of fp32 terms
        return {"rel": 1e-3, "max": 0.1}
    if fam == "pass" and case["grad"] == "bf16":  # dlogits rounded to bf16
        return {"rel": 2e-3, "max": 0.05, "differ": 2e-3}
    if fam == "pass" and case["mode"] in ("seq_tis", "seq_mis"):  # sums of log p over a response
        return {"rel": 5e-5, "max": 1e-2, "differ": 2e-3}
    return {"rel": 2e-5, "max": 1e-2, "differ": 2e-3}


# ------------------------------------------------------------------ 64 bits
def _weight64(mode, lw, linf):
    """The token operator on fp64 log-probabilities."""
    lk = lw - linf
    k = lk.exp()
    om = -torch.expm1(lw)
    cap = 1 + LAM * om.clamp(min=KAPPA)
    if mode == "cis":
        return torch.minimum(k, cap)
    if mode == "tis":
        return k.clamp(max=TIS_CAP)
    if mode == "exact":
        return k.clamp(*EXACT)
    if mode == "band":
        return torch.maximum(torch.minimum(k, cap), 0.5 * (1 + lw.exp()))
    if mode == "icepop":
        return torch.where((k >= ICEPOP[0]) & (k <= ICEPOP[1]), k, torch.zeros_like(k))
    if mode == "kpop":
        p, q = lw.exp().clamp(1e-8, 1 - 1e-8), linf.exp().clamp(1e-8, 1 - 1e-8)
        a = p * (p / q).log() + (1 - p) * ((1 - p) / (1 - q)).log()
        b = q * (q / p).log() + (1 - q) * ((1 - q) / (1 - p)).log()
        return torch.where(torch.maximum(a, b) <= KPOP_PHI, k, torch.zeros_like(k))
    return torch.ones_like(k)


def _tokens64(case, s, lp):
    """w, the loss terms and the gradient's factor c of every token, from fp64 log p."""
    T = case["T"]
    on = torch.ones(T, dtype=torch.bool, device=DEV) if s["mask"] is None else s["mask"] != 0
    seg = torch.searchsorted(s["cu"].long()[1:], torch.arange(T, device=DEV), right=True)
    linf, adv = s["lp_infer"].double(), s["adv"].double()
    lw = lp if s["lp_old"] is None else s["lp_old"].double()
    B_ = s["cu"].shape[0] - 1
    zero = torch.zeros(T, dtype=torch.float64, device=DEV)
    if case["mode"] in ("seq_tis", "seq_mis"):
        total = torch.zeros(B_, dtype=torch.float64, device=DEV)
        total.index_add_(0, seg, torch.where(on, lw - linf, zero))
        K = total.exp()
        if case["mode"] == "seq_tis":
            K = K.clamp(max=SEQ_CAP)
        else:
            K = torch.where((K >= SEQ_MIS[0]) & (K <= SEQ_MIS[1]), K, torch.zeros_like(K))
        w = K[seg]
    else:
        w = _weight64(case["mode"], lw, linf)
    w = torch.where(on, w, zero)
    if case.get("seq_mean"):
        per = torch.zeros(B_, dtype=torch.float64, device=DEV).index_add_(0, seg, on.double())
        scale = 1 / ((per > 0).sum() * per[seg].clamp(min=1))
    else:
        scale = 1 / on.sum().double()
    scale = torch.where(on, scale, zero)
    rho = torch.ones_like(lp) if s["lp_old"] is None else (lp - s["lp_old"].double()).exp()
    clipped = rho.clamp(1 - CLIP[0], 1 + CLIP[1])
    loss = -(scale * w * torch.minimum(rho * adv, clipped * adv)).sum().view(1)
    c = torch.where(rho * adv <= clipped * adv, scale * w * rho * adv, zero)
    return on, w, loss, c


def _rows64(z, ids):
    """fp64 rows: (logits, log p of the sampled token, logsumexp, entropy)."""
    z = z.double()
    r = torch.arange(z.shape[0], device=DEV)
    y = ids.long()
    zy = z[r, y]
    rest = z.clone()
    rest[r, y] = -math.inf
    odds = zy - torch.logsumexp(rest, 1)
    lse = torch.logsumexp(z, 1)
    lp = -torch.nn.functional.softplus(-odds)
    return z, lp, lse


def exact(case, seed):
    fam, T = case["family"], case["T"]
    if fam == "lmhead" and 6 * _valid(case) * case["V"] * case["H"] > 4e12:
        return None  # over 20 seconds of fp64 products
    s = prepare(case, seed)
    if fam == "report":
        on = s["mask"] != 0 if s["mask"] is not None else torch.ones(T, dtype=torch.bool,
                                                                     device=DEV)
        lp, linf = s["lp"].double(), s["lp_infer"].double()
        zero = torch.zeros_like(lp)
        w = torch.where(on, _weight64(case["mode"], lp, linf), zero)
        eps = (lp - linf) - torch.log(-torch.expm1(lp)) + torch.log(-torch.expm1(linf))
        eps = torch.where(on, eps, zero)
        edges = torch.tensor(s["edges"], dtype=torch.float64, device=DEV)
        key, n = s["key"].double(), case["nbins"]
        b = torch.searchsorted(edges, key, right=True) - 1
        b = torch.where(key == edges[n], torch.full_like(b, n - 1), b)
        ok = on & (key >= edges[0]) & (key <= edges[n])
        sums = torch.zeros((2, n), dtype=torch.float64, device=DEV)
        for i, v in enumerate((w, eps)):
            sums[i].index_add_(0, b[ok], v[ok])
        return {"w": w, "trunc": None, "eps": eps, "counts": None, "sums": sums}
    if fam == "lmhead":
        h, wt = s["hidden"].double(), s["weight"].double()
        z, lp, lse = _rows64(h @ wt.t(), s["ids"])
        on, w, loss, c = _tokens64(case, s, lp)
        dz = (z - lse.view(-1, 1)).exp_().mul_(c.view(-1, 1))
        dz[torch.arange(T, device=DEV), s["ids"].long()] -= c
        dh, dw = dz @ wt, dz.t() @ h
        return {"dhidden": dh, "dweight": dw, "lp": lp.masked_fill(~on, 0), "w": w,
                "trunc": None, "loss": loss}
    step = max(1, (1 << 27) // case["V"])
    if fam == "diagnostics":
        return _diagnostics64(case, s, step)
    lp = torch.empty(T, dtype=torch.float64, device=DEV)
    lse, ent = torch.empty_like(lp), torch.empty_like(lp)
    on = torch.ones(T, dtype=torch.bool, device=DEV) if s["mask"] is None else s["mask"] != 0
    for a in range(0, T, step):
        b = min(T, a + step)
        z, lp[a:b], lse[a:b] = _rows64(s["logits"][a:b], s["ids"][a:b])
        ls = z.sub_(lse[a:b].view(-1, 1))
        ent[a:b] = -(ls.exp() * ls).sum(1)
    ent = ent.masked_fill(~on, 0)
    if fam == "logprobs":
        out = [lp.masked_fill(~on, 0)]
        if case["entropy"]:
            return out + [lse.masked_fill(~on, 0) if case["lse"] else None, ent]
        return out + [lse.masked_fill(~on, 0)] if case["lse"] else out[0]
    on, w, loss, c = _tokens64(case, s, lp)
    dz = torch.empty((T, case["V"]), dtype=torch.float64, device=DEV)
    for a in range(0, T, step):
        b = min(T, a + step)
        d = (s["logits"][a:b].double() - lse[a:b].view(-1, 1)).exp_().mul_(c[a:b].view(-1, 1))
        r = torch.arange(b - a, device=DEV)
        y = s["ids"][a:b].long()
        d[r, y] = c[a:b] * torch.expm1(lp[a:b])
        dz[a:b] = d
    out = {"dlogits": dz, "lp": lp.masked_fill(~on, 0), "w": w, "trunc": None,
           "entropy": ent if case["entropy"] else None, "loss": loss}
    if case["stats"]:
        out["sums"] = out["counts"] = None
    return out


def _diagnostics64(case, s, step):
    T = case["T"]
    on = torch.ones(T, dtype=torch.bool, device=DEV) if s["mask"] is None else s["mask"] != 0
    out = {k: torch.zeros(T, dtype=torch.float64, device=DEV)
           for k in ("eps", "logk", "p", "bias2", "dvar")}
    for a in range(0, T, step):
        b = min(T, a + step)
        y = s["ids"][a:b]
        r = torch.arange(b - a, device=DEV)
        zt, lp, lset = _rows64(s["logits"][a:b], y)
        zi, lq, lsei = _rows64(s["infer"][a:b], y)
        rest_t, rest_i = zt.clone(), zi.clone()
        zyt, zyi = zt[r, y.long()], zi[r, y.long()]
        rest_t[r, y.long()] = -math.inf
        rest_i[r, y.long()] = -math.inf
        out["eps"][a:b] = ((zyt - torch.logsumexp(rest_t, 1)) -
                           (zyi - torch.logsumexp(rest_i, 1)))
        out["logk"][a:b] = lp - lq
        out["p"][a:b] = lp.exp()
        del rest_t, rest_i
        lpj, lqj = zt.sub_(lset.view(-1, 1)), zi.sub_(lsei.view(-1, 1))
        f = _weight64(case["mode"], lpj, lqj)
        p, q = lpj.exp_(), lqj.exp_()
        qf = q * f
        res = qf - p
        out["bias2"][a:b] = (res - p * res.sum(1, keepdim=True)).square_().sum(1)
        P2 = p.square().sum(1, keepdim=True)
        g2 = 1 - 2 * p + P2
        F = qf.sum(1)
        mean_f = (qf.square().sum(1) - 2 * F * (qf * p).sum(1) + F * F * P2.view(-1))
        out["dvar"][a:b] = ((qf * f * g2).sum(1) - mean_f -
                            ((q * g2).sum(1) - (q - p).square().sum(1)))
    return {k: v.masked_fill(~on, 0) for k, v in out.items()}
