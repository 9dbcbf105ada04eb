"""The work that this framework is used for, as cases to time and to compare.

A user of the framework does three things with it: rolls a policy out (prefill of every
environment's prefix, then 7 sampled action tokens, turn after turn), re-scores stored actions for
the PPO ratio, and computes the learning-phase quantities (GAE, the clipped objective).  The cases
are those calls through the public binding, over the range of batch sizes, contexts and model
shapes that the repository's workloads span.  Single layers cost the same at any depth, so most
cases run a stack of two 7B-shaped layers; one runs all 32.

A rollout here replays a recorded one: the sampler's noise gives the recorded bin a Gumbel value
above every other bin's, so the sampled tokens are known and two implementations that differ in
rounding see the same contexts.  Everything else is the usual sampling path.
"""
import dataclasses
import math

import torch

from paper_2505_18719_gb300 import inputs as I
from paper_2505_18719_gb300 import vla as V

DEV = "cuda"
F64 = torch.float64
BIAS = 2.0            # bias of the value head: the scale of a return
GAMMA, LAM, EPS = 0.99, 0.95, 0.2


# ------------------------------------------------------------------------------------- cases
def _policy(name, kind, model, layers, batch, visual, text_min, text_max, turns=1, score=False,
            temperature=1.0):
    return {"name": name, "kind": kind, "model": model, "layers": layers, "batch": batch, "visual": visual,
            "text_min": text_min, "text_max": text_max, "turns": turns, "score": score,
            "temperature": temperature}


def listed():
    return [
        # advantages of one PPO batch: 128 environment steps of 256 environments
        {"name": "gae_128x256", "kind": "gae", "steps": 128, "envs": 256},
        # the clipped objective over that batch: 32768 samples of 7 token log-probs
        {"name": "ppo_32768x7", "kind": "ppo", "samples": 32768, "tokens": 7},
        # the smallest configuration, one turn: bound by launches and latency
        _policy("tiny_b4_turn", "rollout", "tiny", 2, 4, 64, 16, 16),
        # the small configuration with the PPO ratio pass (64-wide heads)
        _policy("small_b16_turn_score", "rollout", "small", 8, 16, 256, 24, 24, score=True),
        # one robot served alone by the 7B shape: one turn of a single environment
        _policy("7b_l2_b1_turn", "rollout", "7b", 2, 1, 256, 32, 32),
        # the 7 action tokens at small, ordinary and large batch; the last over a long
        # multi-turn context (320 + 3 * 257 positions)
        _policy("7b_l2_b16_decode", "decode", "7b", 2, 16, 256, 32, 32),
        _policy("7b_l2_b64_decode", "decode", "7b", 2, 64, 256, 16, 48),
        _policy("7b_l2_b256_long_decode", "decode", "7b", 2, 256, 256, 64, 64, turns=4),
        # prefill of 64 ragged prefixes with the value model's estimate of each state
        _policy("7b_l2_b64_prefill", "prefill", "7b", 2, 64, 256, 16, 48),
        # a 4-turn episode: prefill, then appended chunks over a growing context, with decode
        _policy("7b_l2_b16_episode", "rollout", "7b", 2, 16, 256, 64, 64, turns=4, temperature=1.5),
        # the PPO ratio pass: 6 teacher-forced rows of each of 64 environments
        _policy("7b_l2_b64_score", "score", "7b", 2, 64, 256, 16, 48),
        # the whole 7B rollout step of 64 environments: prefill, decode, score
        _policy("7b_b64_turn_score", "rollout", "7b", 32, 64, 256, 16, 48, score=True),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gae", "ppo", "rollout", "rollout", "decode", "decode", "prefill", "score"])
    if kind == "gae":
        return {"kind": "gae", "steps": _log_int(rng, 1, 1024), "envs": _log_int(rng, 1, 4096)}
    if kind == "ppo":
        return {"kind": "ppo", "samples": _log_int(rng, 1, 1 << 20), "tokens": rng.randint(1, 16)}
    model = rng.choice(["tiny", "small", "7b", "7b", "640x64", "1536x128", "2560x128"])
    layers = rng.randint(1, 8 if model in ("tiny", "small") else 2)
    text_min = rng.randint(1, 48)
    text_max = text_min + rng.choice([0, rng.randint(0, 48)])
    visual = rng.choice([0, rng.randint(1, 256), 256])
    turns = rng.randint(1, 4)
    case = _policy("", kind, model, layers, 1, visual, text_min, text_max,
                   turns=turns, score=kind == "rollout" and rng.random() < 0.4,
                   temperature=rng.choice([0.7, 1.0, 1.5]))
    del case["name"]
    # batches whose contexts stay within what the largest listed case holds
    most = max(1, min(256, 32768 // (turns * (visual + text_max + 1))))
    case["batch"] = _log_int(rng, 1, most)
    return case


# ------------------------------------------------------------------------------------ shapes
def _shape(case):
    named = {"tiny": I.TINY, "small": I.SMALL, "7b": I.LLAMA7B}
    if case["model"] in named:
        return dataclasses.replace(named[case["model"]], n_layers=case["layers"])
    d, hd = (int(x) for x in case["model"].split("x"))
    ffn = (d * 8 // 3 + 7) // 8 * 8
    return I.ModelShape(case["model"], case["layers"], d, d // hd, hd, ffn)


def _lengths(case):
    """Text ids of each environment: fixed by the case, spread over [text_min, text_max]."""
    span = case["text_max"] - case["text_min"] + 1
    return [case["text_min"] + (b * 29 + 7) % span for b in range(case["batch"])]


def _chunks(case):
    """Per turn, per environment: rows of that turn's prefill (with the pending action token)."""
    first = [case["visual"] + n for n in _lengths(case)]
    later = max(1, case["visual"])  # later turns append a7 and a new image (or one id)
    return [first] + [[later + 1] * case["batch"] for _ in range(case["turns"] - 1)]


# ------------------------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _normal(g, shape, std):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(0.0, std, generator=g)


def _policy_inputs(case, seed):
    sh = _shape(case)
    g = _generator(seed)
    L, d, F, std = sh.n_layers, sh.d_model, sh.d_ffn, sh.weight_std
    ones = torch.ones(L, d, dtype=torch.bfloat16, device=DEV)
    w = {"embed": _normal(g, (sh.vocab, d), std), "attn_norm": ones, "wqkv": _normal(g, (L, 3 * d, d), std),
         "wo": _normal(g, (L, d, d), std), "ffn_norm": ones.clone(), "w_gate_up": _normal(g, (L, 2 * F, d), std),
         "w_down": _normal(g, (L, d, F), std), "final_norm": torch.ones(d, dtype=torch.bfloat16, device=DEV),
         "lm_head": _normal(g, (sh.vocab, d), std)}
    B, A = case["batch"], sh.action_dim
    turns = []
    for t in range(case["turns"]):
        # the first turn has the instruction; later ones an image, or one id where there are none
        lengths = _lengths(case) if t == 0 else [0 if case["visual"] else 1] * B
        width = max(lengths)
        visual = _normal(g, (B, case["visual"], d), 1.0) if case["visual"] else None
        ids = torch.randint(0, sh.vocab - 256, (B, width), generator=g, device=DEV, dtype=torch.int32) if width else None
        bins = torch.randint(0, 256, (B, A), generator=g, device=DEV)
        noise = torch.rand(B, A, 256, generator=g, device=DEV) * 0.98 + 0.005
        noise.scatter_(2, bins[:, :, None], 1.0 - 2.0 ** -24)  # the recorded bin wins
        turns.append({"visual": visual, "ids": ids, "lengths": lengths, "noise": noise,
                      "tokens": (bins + (sh.vocab - 256)).to(torch.int32)})
    w_value = _normal(g, (d,), std)
    return sh, w, turns, w_value


def _learning_inputs(case, seed):
    g = _generator(seed)
    r = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    u = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    if case["kind"] == "gae":
        M, B = case["steps"], case["envs"]
        return {"rewards": r(M, B), "values": 2.0 * r(M + 1, B), "dones": (u(M, B) < 0.1).float()}
    N, A = case["samples"], case["tokens"]
    old = -6.0 * u(N, A)
    return {"old": old, "new": old + 0.06 * (2.0 * u(N, A) - 1.0), "adv": r(N)}


def prepare(case, seed):
    if case["kind"] in ("gae", "ppo"):
        s = _learning_inputs(case, seed)
        s["case"] = case
        s["stream"] = torch.cuda.current_stream().cuda_stream
        return s
    sh, w, turns, w_value = _policy_inputs(case, seed)
    chunks = _chunks(case)
    capacity = max(sum(c[b] for c in chunks) for b in range(case["batch"])) + 6 * case["turns"]
    pol = V.Policy(sh, w, case["batch"], (capacity + 31) // 32 * 32,
                   max(max(sum(c) for c in chunks), 6 * case["batch"]))
    s = {"case": case, "policy": pol, "turns": turns, "w_value": w_value}
    if case["kind"] in ("decode", "score"):
        for t, turn in enumerate(turns):
            pol.prefill(turn["visual"], turn["ids"], turn["lengths"])
            if t + 1 < len(turns):
                pol.decode(turn["noise"], case["temperature"], want_logits=False)
        pol.sync()
    return s


# --------------------------------------------------------------------------------------- run
def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "gae":
        r = state["rewards"]
        adv, ret = torch.empty_like(r), torch.empty_like(r)
        _ok(V.vla_gae(r.data_ptr(), state["values"].data_ptr(), state["dones"].data_ptr(), case["steps"],
                      case["envs"], GAMMA, LAM, adv.data_ptr(), ret.data_ptr(), state["stream"]))
        return {"advantages": adv, "returns": ret}
    if kind == "ppo":
        n = case["samples"]
        obj, frac, ratio = (torch.empty(k, dtype=torch.float32, device=DEV) for k in (1, 1, n))
        _ok(V.vla_ppo_clip(state["new"].data_ptr(), state["old"].data_ptr(), state["adv"].data_ptr(), n,
                           case["tokens"], EPS, obj.data_ptr(), ratio.data_ptr(), frac.data_ptr(), state["stream"]))
        return {"objective": obj, "ratio": ratio, "clip_fraction": frac}
    pol, turns, T = state["policy"], state["turns"], case["temperature"]
    last = turns[-1]
    if kind == "decode":  # decoding again re-decodes the latest turn
        return pol.decode(last["noise"], T)
    if kind == "score":
        return pol.score(last["tokens"], T)
    pol.reset()
    if kind == "prefill":
        for turn in turns:
            pol.prefill(turn["visual"], turn["ids"], turn["lengths"])
        return {"values": pol.value(state["w_value"], BIAS)}
    out = []
    for turn in turns:
        pol.prefill(turn["visual"], turn["ids"], turn["lengths"])
        d = pol.decode(turn["noise"], T)
        out.append({"decode": d})
        if case["score"]:
            out[-1]["score"] = pol.score(d["tokens"], T)
    return out


def _ok(rc):
    if rc != V.VLA_OK:
        raise V.VlaError(rc, V.vla_last_error())


# -------------------------------------------------------------------------------------- work
def _layer_params(sh):
    return 4 * sh.d_model * sh.d_model + 3 * sh.d_model * sh.d_ffn


def _pass_work(sh, chunks, start, pruned):
    """One forward over rows appended at positions start[b] ..: (bytes, flops).  `pruned`: past
    q|k|v the last layer is needed for each environment's final row only."""
    L, d, P = sh.n_layers, sh.d_model, _layer_params(sh)
    rows, B = sum(chunks), len(chunks)
    tail = B if pruned else rows
    flops = 2.0 * ((L - 1) * P * rows + 3 * d * d * rows + (P - 3 * d * d) * tail)
    nbytes = 2.0 * P * L + 4.0 * d * rows
    for n, s in zip(chunks, start):
        pairs = n * s + n * (n + 1) / 2.0
        flops += 4.0 * d * ((L - 1) * pairs + (s + n if pruned else pairs))
        nbytes += L * 5.0 * d * (s + n)  # cached keys and values: 2.5 bytes each
    return nbytes, flops


def work(case):
    if case["kind"] == "gae":
        n = case["steps"] * case["envs"]
        return {"bytes": 4.0 * (5 * n + case["envs"]), "flops": 8.0 * n}
    if case["kind"] == "ppo":
        n = case["samples"]
        return {"bytes": 4.0 * (2 * n * case["tokens"] + 2 * n), "flops": n * (2.0 * case["tokens"] + 10)}
    sh = _shape(case)
    B, d, A = case["batch"], sh.d_model, sh.action_dim
    head = (2.0 * 256 * d + B * (4.0 * d + 2048.0), 2.0 * 256 * d * B)
    total = [0.0, 0.0]

    def add(w, n=1):
        total[0] += n * w[0]
        total[1] += n * w[1]

    pos = [0] * B
    for t, chunk in enumerate(_chunks(case)):
        before = case["kind"] in ("decode", "score")  # prepared state: its prefill is not timed
        if not before:
            add(_pass_work(sh, chunk, pos, True))
        pos = [p + c for p, c in zip(pos, chunk)]
        if case["kind"] == "prefill":
            continue
        if not before or t + 1 == case["turns"]:
            if case["kind"] != "score":
                add(head, A)
                for i in range(A - 1):
                    add(_pass_work(sh, [1] * B, [p + i for p in pos], False))
            if case["kind"] == "score" or case["score"]:
                add(head, A)
                add(_pass_work(sh, [A - 1] * B, pos, False))
        pos = [p + A - 1 for p in pos]
    return {"bytes": total[0], "flops": total[1]}


# --------------------------------------------------------------------------------- tolerance
def tolerance(case):
    if case["kind"] == "gae":  # 32-bit sums: 1.8e-7 off the 64-bit result
        return {"rel": 1e-6, "max": 1e-4}
    if case["kind"] == "ppo":
        # 32-bit sums: 6e-8 off on the listed case; the objective is a mean of terms of both signs,
        # which may come out a hundred times smaller than they are
        return {"rel": 1e-5, "max": 1e-4}
    # fp16 operands (the low half kept for some projections), fp32 sums: the logits are 2.5e-4 to
    # 7e-4 off the 64-bit model over 2 to 8 layers, and the error grows with the depth
    return {"rel": 1e-2, "max": 0.2} if case["layers"] > 8 else {"rel": 3e-3, "max": 0.1}


# ------------------------------------------------------------------------------------- exact
def exact(case, seed):
    if case["kind"] == "gae":
        s = {k: v.to(F64) for k, v in _learning_inputs(case, seed).items()}
        adv = torch.zeros_like(s["rewards"])
        nxt = torch.zeros_like(adv[0])
        for t in range(case["steps"] - 1, -1, -1):
            live = 1.0 - s["dones"][t]
            nxt = s["rewards"][t] + GAMMA * live * s["values"][t + 1] - s["values"][t] + GAMMA * LAM * live * nxt
            adv[t] = nxt
        return {"advantages": adv, "returns": adv + s["values"][:-1]}
    if case["kind"] == "ppo":
        s = {k: v.to(F64) for k, v in _learning_inputs(case, seed).items()}
        rho = torch.exp((s["new"] - s["old"]).sum(-1))
        obj = torch.minimum(rho * s["adv"], rho.clamp(1.0 - EPS, 1.0 + EPS) * s["adv"]).mean()
        return {"objective": obj[None], "ratio": rho, "clip_fraction": ((rho - 1.0).abs() > EPS).to(F64).mean()[None]}
    sh = _shape(case)
    B, A = case["batch"], sh.action_dim
    rows = sum(sum(c) for c in _chunks(case)) + B * (A - 1) * case["turns"]
    d = sh.d_model
    if 2.0 * rows * ((sh.n_layers - 1) * _layer_params(sh) + 3 * d * d) > 1.3e13:
        return None  # over about 20 seconds of 64-bit matrix products
    sh, w, turns, w_value = _policy_inputs(case, seed)

    # every row of every environment's context, its actions included, in one causal pass
    emb = w["embed"]
    rows_of, heads_at = [], []  # per environment: [n, d] rows; per turn, the head's rows
    for b in range(B):
        parts, at, n = [], [], 0
        for t, turn in enumerate(turns):
            if turn["visual"] is not None:
                parts.append(turn["visual"][b])
            if turn["ids"] is not None and turn["lengths"][b]:
                parts.append(emb[turn["ids"][b, :turn["lengths"][b]].long()])
            n += (turn["lengths"][b] if turn["ids"] is not None else 0) + case["visual"]
            if case["kind"] == "prefill":
                at.append([n - 1])
                continue
            at.append(list(range(n - 1, n + A - 1)))
            last = t + 1 == len(turns)
            parts.append(emb[turn["tokens"][b, :A - 1 if last else A].long()])
            n += A - 1 if last else A
        rows_of.append(torch.cat(parts).to(F64))
        heads_at.append(at)
    states = _forward64(sh, w, rows_of, [sorted({i for t in at for i in t}) for at in heads_at])
    fin = w["final_norm"].to(F64)
    if case["kind"] == "prefill":
        h = torch.stack([states[b][-1] for b in range(B)])
        return {"values": _rms64(h, fin, sh.rms_eps) @ w_value.to(F64) + BIAS}
    out = []
    T = case["temperature"]
    hw = w["lm_head"][sh.vocab - 256:].to(F64)
    for t, turn in enumerate(turns):
        h = torch.stack([states[b][t * A:(t + 1) * A] for b in range(B)])
        z = _rms64(h, fin, sh.rms_eps) @ hw.T
        lp = torch.log_softmax(z / T, -1)
        bins = (turn["tokens"] - (sh.vocab - 256)).long()
        res = {"logits": z, "logprobs": lp.gather(-1, bins[:, :, None])[:, :, 0],
               "entropy": -(lp.exp() * lp).sum(-1)}
        dec = dict(res, tokens=None, actions=(2.0 * bins.to(F64) + 1.0) / 256.0 - 1.0)
        out.append({"decode": dec, "score": res} if case["score"] else {"decode": dec})
    if case["kind"] == "decode":
        return out[-1]["decode"]
    if case["kind"] == "score":
        return res
    return out


def _rms64(x, w, eps):
    return x / torch.sqrt((x * x).mean(-1, keepdim=True) + eps) * w


def _forward64(sh, w, rows_of, wanted):
    """The decoder over each environment's rows in 64 bits; the final states of `wanted` rows."""
    d, H, hd, F = sh.d_model, sh.n_heads, sh.head_dim, sh.d_ffn
    count = [r.shape[0] for r in rows_of]
    h = torch.cat(rows_of)
    inv = sh.rope_theta ** (-2.0 * torch.arange(hd // 2, dtype=F64, device=DEV) / hd)
    pos = torch.cat([torch.arange(n, dtype=F64, device=DEV) for n in count])
    c, s = torch.cos(pos[:, None] * inv)[:, None], torch.sin(pos[:, None] * inv)[:, None]
    keep = torch.cat([torch.tensor(k, device=DEV) + sum(count[:b]) for b, k in enumerate(wanted)])

    def rotate(x):
        x1, x2 = x[..., :hd // 2], x[..., hd // 2:]
        return torch.cat([x1 * c - x2 * s, x2 * c + x1 * s], -1)

    for l in range(sh.n_layers):
        y = _rms64(h, w["attn_norm"][l].to(F64), sh.rms_eps)
        q, k, v = (y @ m.to(F64).T for m in w["wqkv"][l].split(d))
        q, k, v = rotate(q.view(-1, H, hd)), rotate(k.view(-1, H, hd)), v.view(-1, H, hd)
        o = torch.empty_like(q)
        at = 0
        for n in count:
            qb, kb, vb = (x[at:at + n].transpose(0, 1) for x in (q, k, v))
            score = qb @ kb.transpose(1, 2) / math.sqrt(hd)
            score.masked_fill_(torch.ones(n, n, dtype=torch.bool, device=DEV).triu(1), -math.inf)
            o[at:at + n] = (torch.softmax(score, -1) @ vb).transpose(0, 1)
            at += n
        o = o.view(-1, d)
        if l + 1 == sh.n_layers:
            h, o = h[keep], o[keep]
        h = h + o @ w["wo"][l].to(F64).T
        y = _rms64(h, w["ffn_norm"][l].to(F64), sh.rms_eps)
        gate, up = (y @ m.to(F64).T for m in w["w_gate_up"][l].split(F))
        h = h + (gate * torch.sigmoid(gate) * up) @ w["w_down"][l].to(F64).T
    return h.split([len(k) for k in wanted])
