"""What a user of the decode library has it do, as cases that can be timed: whole generations, Jacobi-window
iterations over a filled cache, and prompts, on the model shapes of `workload.CONFIGS`.

A case is a dict: `model` (a key of CONFIGS), `kind`, `batch`, `c` (window rows per sequence), `length` (tokens cached, or
prompt ids, of the longest sequence) and, by kind, what follows.

  step      `steps` iterations of fc_jacobi_step over a cache of `length` tokens; the first takes its window from the
            caller, the others go on with the window that the iteration before left
  prefill   fc_prefill of `batch` prompts, then the first iteration over them
  generate  fc_prefill, then fc_generate of `tokens` tokens
  request   the whole method: fc_prefill, `tokens` iterations, then the approximate rationale handed to an answer
            trigger of `trigger` ids and `answer` answer tokens

Weights are random of the shape's own distribution, prompts random ids, cached keys and values N(0, 1).  The sequences of
a batch have different lengths.  The logit bonus on a seeded permutation of the input token is larger than in CONFIGS (24
instead of 6 for the bf16 shapes): as with a trained model, the greedy token of nearly every row is then far from a tie.
"""
import math

import torch

from paper_2311_08263_b200 import engine
from paper_2311_08263_b200.workload import CONFIGS

BETA = {"tiny": 4.0, "1b": 24.0, "7b": 24.0, "13b": 24.0}
PAD = 1


def listed():
    return [
        # the fp32 shape from prompt to last token: every call is small, launches and host round trips are what counts
        dict(name="tiny-generate", model="tiny", kind="generate", batch=1, c=8, length=32, tokens=64),
        # one user, the smallest bf16 shape (GQA, head_dim 64), in the middle of a generation
        dict(name="1b-step-c16", model="1b", kind="step", batch=1, c=16, length=641, steps=4),
        # one user from prompt to answer on the same shape: prompt, iterations, hand-off to the trigger, answer
        dict(name="1b-request", model="1b", kind="request", batch=1, c=16, length=512, tokens=24, trigger=7, answer=8),
        # one user, plain autoregressive decoding (a window of one row)
        dict(name="7b-step-c1", model="7b", kind="step", batch=1, c=1, length=512, steps=4),
        # one user, the window of the paper's experiments behind a few-shot prompt
        dict(name="7b-step-c16", model="7b", kind="step", batch=1, c=16, length=803, steps=4),
        # a batch decoded autoregressively: as many rows, 30 times the cache
        dict(name="7b-step-b16-c1", model="7b", kind="step", batch=16, c=1, length=2048, steps=4),
        # a few users with very long contexts
        dict(name="7b-step-b4-c8-long", model="7b", kind="step", batch=4, c=8, length=8190, steps=4),
        # a few users, ordinary window and context
        dict(name="7b-step-b4-c16", model="7b", kind="step", batch=4, c=16, length=2048, steps=4),
        # a busy server: many rows per forward
        dict(name="7b-step-b16-c32", model="7b", kind="step", batch=16, c=32, length=515, steps=2),
        # the largest shape, its serving batch
        dict(name="13b-step-b8-c32", model="13b", kind="step", batch=8, c=32, length=1024, steps=2),
        # a few-shot prompt on its way into the cache
        dict(name="7b-prefill", model="7b", kind="prefill", batch=1, c=16, length=800),
        # the prompts of the serving batch
        dict(name="13b-prefill-b8", model="13b", kind="prefill", batch=8, c=32, length=1024),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    dearest = {k: max(work(c)[k] for c in listed()) for k in ("bytes", "flops")}
    while True:
        model = rng.choice(["tiny", "1b", "1b", "7b", "7b", "7b", "13b"])
        kind = rng.choice(["generate", "request"] if model == "tiny" else ["step", "step", "step", "step", "prefill", "request"])
        case = dict(model=model, kind=kind, batch=_log_int(rng, 1, 4 if model == "tiny" else 16),
                    c=_log_int(rng, 1, 16 if model == "tiny" else 64),
                    length=_log_int(rng, 16, 200) if model == "tiny" else _log_int(rng, 64, 8192 if kind == "step" else 1500))
        if kind == "step":
            case["steps"] = 2
        elif kind == "generate":
            case["tokens"] = rng.randint(16, 64)
        elif kind == "request":
            case.update(tokens=rng.randint(8, 24), trigger=rng.randint(0, 12), answer=rng.randint(1, 12))
        w = work(case)
        tokens_held = case["batch"] * case["length"] * CONFIGS[model].kv_bytes_per_token()
        if case["batch"] * case["c"] <= 512 and tokens_held < 18e9 and all(w[k] <= dearest[k] for k in dearest):
            return case


def _lengths(case):
    """Different lengths for the sequences of a batch, the first the longest."""
    n = case["length"]
    return [n - (i * 61) % (n // 4 + 1) for i in range(case["batch"])]


def _rows(case):
    """(rows of every forward with an LM head, ids cached before them, tokens already in the cache) of one pass."""
    b, c, lens = case["batch"], case["c"], _lengths(case)
    if case["kind"] == "step":
        return [c] * case["steps"], [0] * b, lens
    ids = [n - 1 for n in lens]
    if case["kind"] == "prefill":
        return [c], ids, [0] * b
    if case["kind"] == "generate":
        return [c] * case["tokens"], ids, [0] * b
    return [c] * case["tokens"] + [1] * case["answer"], [n + c + case["trigger"] - 1 for n in ids], [0] * b


def work(case):
    """One pass over the weights for every forward that has to follow another one, each cached key and value read by every
    forward behind it and written once, the embedding rows read, the logits written."""
    cfg, b = CONFIGS[case["model"]], case["batch"]
    s, d = cfg.elem_bytes, cfg.d_model
    head, layers = cfg.vocab * d, cfg.weight_params() - cfg.vocab * d
    per_pair = 4.0 * cfg.n_layers * cfg.n_heads * cfg.head_dim          # Q.K and P.V for one query row and one key
    kv = cfg.kv_bytes_per_token()
    rows, ids, held = _rows(case)
    n_ids = sum(ids)
    by = n_ids * (kv + d * s) + (layers * s if n_ids else 0)
    fl = 2.0 * n_ids * layers + per_pair * sum(n * (n + 1) / 2 for n in ids)
    for i, r in enumerate(rows):
        known = sum(held) + n_ids + b * i                               # one token per sequence and forward at least
        by += (layers + head) * s + known * kv + b * r * (kv + d * s + cfg.vocab * 4)
        fl += 2.0 * b * r * (layers + head) + per_pair * r * (known + b * (r + 1) / 2)
    return {"bytes": float(by), "flops": float(fl)}


def tolerance(case):
    """About four times what the same pass shows with its sums in another order (one launch per projection, the
    feed-forward block in one piece, no CTA pairs).  Measured: logits behind a given cache 3e-5 (1b) to 1.7e-4 (13b), max
    3.4e-3; after a prompt, keys and values 1.6e-3 (7b) to 2.2e-3 (13b), max 2.5e-2 - they are rounded to bf16 where they
    are stored, and every layer inherits the flips of the one before.  A query rounded to bf16 shows 7e-3 to 1.4e-2."""
    if case["model"] == "tiny":
        return {"rel": 1e-5, "max": 1e-3}
    if case["kind"] == "step":
        return {"rel": 1e-3, "max": 2e-2}
    return {"rel": 8e-3, "max": 0.1}


def _weights(cfg, gen):
    dt, dev = cfg.torch_dtype, "cuda"
    d, qd, kvd, f, v = cfg.d_model, cfg.n_heads * cfg.head_dim, cfg.n_kv_heads * cfg.head_dim, cfg.d_ffn, cfg.vocab

    def mat(rows, cols):
        return torch.empty(rows, cols, dtype=dt, device=dev).normal_(0.0, 0.02, generator=gen)

    def gain():
        return torch.empty(d, dtype=torch.float32, device=dev).normal_(1.0, 0.1, generator=gen).to(dt)

    w = {"tok_emb": mat(v, d), "g_final": gain(), "lm_head": mat(v, d)}
    for name, (r, c) in {"wq": (qd, d), "wk": (kvd, d), "wv": (kvd, d), "wo": (d, qd), "w_gate": (f, d), "w_up": (f, d),
                         "w_down": (d, f)}.items():
        w[name] = [mat(r, c) for _ in range(cfg.n_layers)]
    for name in ("g_attn", "g_ffn"):
        w[name] = [gain() for _ in range(cfg.n_layers)]
    w["bias_perm"] = torch.randperm(v, generator=gen, device=dev).to(torch.int32)
    return w


def prepare(case, seed):
    import dataclasses
    cfg = dataclasses.replace(CONFIGS[case["model"]], bias_beta=BETA[case["model"]])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    b, c, lens = case["batch"], case["c"], _lengths(case)
    w = _weights(cfg, gen)
    more = {"step": c * case.get("steps", 0), "prefill": c, "generate": case.get("tokens", 0) + c,
            "request": (case.get("tokens", 0) + 1) * c + case.get("trigger", 0) + case.get("answer", 0)}[case["kind"]]
    dec = engine.Decoder(cfg, w, b, c, case["length"] + more + 8)
    state = {"case": case, "dec": dec, "weights": w, "logits": dec.fc_debug_logits(True)}

    def ids(*shape):
        return torch.randint(0, cfg.vocab, shape, generator=gen, device="cuda")

    if case["kind"] == "step":
        kv = dec.kv.view(cfg.torch_dtype)
        for i in range(0, kv.numel(), 1 << 30):
            kv[i:i + (1 << 30)].normal_(generator=gen)
        # the first window of every sequence: some right guesses (they follow the permutation), then wrong ones
        win = ids(b, c)
        right = torch.randint(0, c, (b,), generator=gen, device="cuda")
        for j in range(1, c):
            win[:, j] = torch.where(right >= j, w["bias_perm"][win[:, j - 1]].long(), win[:, j])
        state["window"] = win.to(torch.int32).cpu().numpy()
        state["lens"] = lens
    else:
        state["prompts"], state["lens"] = ids(b, case["length"]).to(torch.int32).cpu().numpy(), lens
        if case["kind"] == "request":
            state["trigger"] = ids(case["trigger"]).to(torch.int32).cpu().numpy()
    torch.cuda.synchronize()
    return state


def run(state):
    case, dec, out = state["case"], state["dec"], {}
    if case["kind"] == "step":
        window = state["window"]
        dec.fc_debug_set_state(state["lens"], window[:, 0], case["c"], pad_id=PAD)
        for i in range(case["steps"]):
            out["step%d" % i] = dec.fc_jacobi_step(window if i == 0 else None)
    else:
        dec.fc_prefill(state["prompts"], state["lens"], case["c"])
        if case["kind"] == "prefill":
            out["step"] = dec.fc_jacobi_step()
            out["kv"] = dec.kv_view()
        elif case["kind"] == "generate":
            out["tokens"], out["lens"], _ = dec.fc_generate(case["tokens"])
        else:
            out["tokens"], out["lens"], _ = dec.fc_generate(case["tokens"] * case["c"], max_iters=case["tokens"])
            out["answer"] = dec.fc_finish_with_trigger(state["trigger"], case["answer"])
    out["logits"] = state["logits"]
    return out

class _Exact:
    """The same model in 64 bits: K and V rounded to the model's type where they are stored, nothing else rounded."""

    def __init__(self, cfg, w, kv):
        self.cfg, self.w, self.kv = cfg, w, kv                       # kv [layers, 2, batch, kv heads, slots, head_dim]
        self.rope = cfg.rope_theta ** (-torch.arange(0, cfg.head_dim, 2, dtype=torch.float64, device="cuda") / cfg.head_dim)

    def _norm(self, x, gain):
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + self.cfg.rms_eps) * gain.double()

    def _turn(self, t, pos):                                         # [rows, heads, head_dim]
        a = (pos[:, None] * self.rope)[:, None]
        x, y = t.chunk(2, -1)
        return torch.cat([x * a.cos() - y * a.sin(), x * a.sin() + y * a.cos()], -1)

    def forward(self, tokens, lens, head=True):
        """tokens [n, c] behind lens[i] cached ones; the K/V of every row is stored; logits [n * c, vocab]."""
        cfg, w = self.cfg, self.w
        n, c = tokens.shape
        hd, g = cfg.head_dim, cfg.n_heads // cfg.n_kv_heads
        x = w["tok_emb"][tokens.reshape(-1)].double()
        pos = torch.cat([torch.arange(m, m + c, device="cuda") for m in lens]).double()
        for l in range(cfg.n_layers):
            h = self._norm(x, w["g_attn"][l])
            q, k, v = (h @ w[name][l].double().T for name in ("wq", "wk", "wv"))
            q, k = self._turn(q.view(n * c, -1, hd), pos), self._turn(k.view(n * c, -1, hd), pos)
            out = torch.empty_like(q)
            for i, m in enumerate(lens):
                at = slice(i * c, (i + 1) * c)
                for half, t in enumerate((k, v.view(n * c, -1, hd))):
                    self.kv[l, half, i, :, m:m + c] = t[at].transpose(0, 1).to(self.kv.dtype)
                seen = torch.arange(m + c, device="cuda") <= torch.arange(m, m + c, device="cuda")[:, None]
                for j in range(cfg.n_kv_heads):
                    keys, values = self.kv[l, 0, i, j, :m + c].double(), self.kv[l, 1, i, j, :m + c].double()
                    s = torch.einsum("rhd,kd->hrk", q[at, j * g:(j + 1) * g], keys) / math.sqrt(hd)
                    p = s.masked_fill(~seen, -math.inf).softmax(-1)
                    out[at, j * g:(j + 1) * g] = torch.einsum("hrk,kd->rhd", p, values)
            x = x + out.reshape(n * c, -1) @ w["wo"][l].double().T
            h = self._norm(x, w["g_ffn"][l])
            h = torch.nn.functional.silu(h @ w["w_gate"][l].double().T) * (h @ w["w_up"][l].double().T)
            x = x + h @ w["w_down"][l].double().T
        if not head:
            return None
        logits = self._norm(x, w["g_final"]) @ w["lm_head"].double().T
        logits[torch.arange(n * c, device="cuda"), w["bias_perm"].long()[tokens.reshape(-1)]] += cfg.bias_beta
        return logits


def exact(case, seed):
    """Logits, and for a prompt the stored keys and values; the tokens are whole numbers and have no such value."""
    if work(case)["flops"] > 1.2e14:                                 # over about 20 seconds in 64 bits
        return None
    state = prepare(case, seed)
    cfg, w, kv, c, lens = state["dec"].cfg, state["weights"], state["dec"].kv_view(), case["c"], list(state["lens"])
    n, model, logits = len(lens), _Exact(cfg, w, kv), state["logits"].double()
    step = case["kind"] == "step"

    def iterate(win, count):
        made = [0] * n
        for _ in range(count):
            got = model.forward(win, lens)
            logits[:len(got)] = got
            best, new = got.view(n, c, -1).argmax(-1), win.clone()
            for i in range(n):
                k = 1
                while k < c and int(win[i, k]) == int(best[i, k - 1]):
                    k += 1
                lens[i], made[i] = lens[i] + k, made[i] + k
                new[i, :c - k + 1] = best[i, k - 1:]
                for j in range(c - k + 1, c):
                    new[i, j] = PAD if step else int(ids[i, (made[i] + j - 1) % size[i]])
            win = new
        return win, max(made)

    if step:
        iterate(torch.from_numpy(state["window"]).long().cuda(), case["steps"])
        return {"logits": logits}
    ids, size = state["prompts"], list(lens)
    lens = [m - 1 for m in size]
    for i, m in enumerate(lens):
        sub = _Exact(cfg, w, kv[:, :, i:i + 1])
        if m:
            sub.forward(torch.from_numpy(ids[i:i + 1, :m]).long().cuda(), [0], head=False)
    win = torch.tensor([[int(ids[i, m])] + [int(ids[i, (j - 1) % (m + 1)]) for j in range(1, c)] for i, m in enumerate(lens)],
                       device="cuda")
    if case["kind"] == "prefill":
        iterate(win, 1)
        return {"logits": logits, "kv": kv}
    win, most = iterate(win, case["tokens"])
    if case["kind"] == "generate":                                   # a sequence that is ahead ends, and its rows go
        return {"logits": logits} if most == case["tokens"] else None
    rest = torch.cat([win, torch.from_numpy(state["trigger"]).long().cuda().expand(n, -1)], 1)
    if rest.shape[1] > 1:
        model.forward(rest[:, :-1], lens, head=False)
    lens = [m + rest.shape[1] - 1 for m in lens]
    win = rest[:, -1:]
    for _ in range(case["answer"]):
        got = model.forward(win, lens)
        logits[:n] = got
        win, lens = got.argmax(-1)[:, None], [m + 1 for m in lens]
    return {"logits": logits}
