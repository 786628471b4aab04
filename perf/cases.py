"""The calls that a user of this library makes, with the sizes they make them at.

Every case is one call (or, for a generation, the two calls) of ``WorldModel`` on device
arrays, as a training or planning loop would issue it.  The handle, the weights and the
inputs are in hand before; outputs are allocated by the call.  Weights, latents and masks
follow the distributions of ``synth`` (weights and biases ~ N(0, 0.05^2), latents ~ N(0, 1),
Bernoulli masks), drawn on the device.
"""
from __future__ import annotations

import math

import torch

import paper_2205_01435_gb300 as pkg

# The model sizes of the library's workloads, and sizes that are no multiple of anything (the
# number of graph substitutions, and so of actions, is whatever the rule set gives).
TINY = dict(Z=32, A=64, H=256, K=5)
SMALL = dict(Z=32, A=128, H=256, K=5)
MID = dict(Z=64, A=256, H=512, K=8)
SCORE = dict(Z=64, A=256, H=512, K=5)
LARGE = dict(Z=128, A=512, H=1024, K=8)
ODD = dict(Z=50, A=101, H=300, K=6)

# Live steps per episode when the done head ends episodes (random weights: few survive the
# first steps), for work() only.
LIVE_STEPS = 3.2


def _case(kind, model, precision, B, T, **flags):
    c = dict(kind=kind, precision=precision, B=B, T=T, sampled=False, done=False, xfers=0, density=0.3,
             ragged=False, seqs=False, carried=False, shaped=False, pop=0)
    c.update(model)
    c.update(flags)
    return c


def listed():
    out = []

    def add(name, *a, **k):
        out.append(dict(_case(*a, **k), name=name))

    # a handful of dreams for a look at the model, fp32: every launch and every step's latency counts
    add("tiny_rollout_fp32", "rollout", TINY, "fp32", 16, 20, density=0.5)
    # one environment step of a vectorised Gym-like wrapper: state in, state and heads out
    add("step_bf16", "rollout", MID, "bf16", 500, 1, seqs=True, carried=True)
    # a small batch of dreams in the low-latency regime
    add("small_rollout_bf16", "rollout", SMALL, "bf16", 1024, 50)
    # one generation of a controller search: 8 candidates x 256 episodes, and their fitness
    add("generation_bf16", "generation", SMALL, "bf16", 2048, 50, pop=8)
    # dreams that the done head ends: most episodes are over after a few steps
    add("mid_rollout_done_bf16", "rollout", MID, "bf16", 8192, 100, density=0.2, done=True)
    # the data-collection rollout: a large batch, actions drawn from the controller's softmax
    add("large_rollout_bf16", "rollout", LARGE, "bf16", 65536, 64, density=0.1, sampled=True)
    # the two-level (substitution, location) action on a large model
    add("hier_rollout_bf16", "rollout", LARGE, "bf16", 16384, 8, density=0.3, sampled=True, xfers=112)
    # a rule set of 101 actions and a model that is a multiple of nothing
    add("odd_rollout_bf16", "rollout", ODD, "bf16", 2000, 30, sampled=True)
    # scoring recorded trajectories, at both precisions; the fp32 ones end at different steps
    add("score_bf16", "score", SCORE, "bf16", 512, 128)
    add("score_fp32", "score", SCORE, "fp32", 512, 128, ragged=True)
    # the world model's training step on a minibatch of trajectories
    add("train_bf16", "train", SCORE, "bf16", 512, 128)
    add("train_fp32", "train", SCORE, "fp32", 200, 100, ragged=True)
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: batches from one to thousands, short and long horizons,
    both precisions, the library's model sizes and odd ones."""
    odd = dict(Z=rng.randint(5, 100), A=rng.randint(17, 300), H=rng.randint(33, 500), K=rng.randint(2, 8))
    model = rng.choice([TINY, SMALL, MID, SCORE, LARGE, odd, odd, odd])
    regular = model is not odd
    precision = rng.choice(["fp32", "bf16", "bf16"])
    kind = rng.choice(["rollout", "rollout", "rollout", "score", "score", "train", "train", "generation"])
    density = round(rng.uniform(0.1, 0.6), 2)
    if kind == "generation":
        pop = rng.choice([2, 4, 8])
        return _case(kind, rng.choice([TINY, SMALL, MID]), "bf16", 256 * pop, rng.randint(10, 60), pop=pop,
                     density=density, sampled=rng.random() < 0.5)
    if kind == "train":
        return _case(kind, model, precision, _log_int(rng, 8, 512), _log_int(rng, 8, 128), ragged=rng.random() < 0.5)
    if kind == "score":
        return _case(kind, model, precision, _log_int(rng, 8, 1024), _log_int(rng, 8, 200), ragged=rng.random() < 0.5,
                     seqs=rng.random() < 0.25)
    if regular and model["A"] >= 256 and precision == "bf16" and rng.random() < 0.25:
        return _case(kind, model, precision, _log_int(rng, 64, 8192), rng.randint(1, 12), density=density,
                     sampled=rng.random() < 0.5, xfers=rng.randint(20, 120))
    most = 16384 if regular and precision == "bf16" else 4096
    seqs = rng.random() < 0.2
    return _case(kind, model, precision, _log_int(rng, 1, most), 1 if seqs else _log_int(rng, 1, 64), density=density,
                 sampled=rng.random() < 0.5, done=regular and precision == "bf16" and rng.random() < 0.25, seqs=seqs,
                 carried=seqs, shaped=rng.random() < 0.2)


# ------------------------------------------------------------------ inputs
def _cfg(c):
    return dict(z_dim=c["Z"], a_dim=c["A"], h_dim=c["H"], k_mix=c["K"], precision=c["precision"],
                ctrl_sample=int(c["sampled"]), ctrl_tau=1.0, done_terminates=int(c["done"]), seed=7,
                reward_mode=int(c["shaped"]), n_xfers=c["xfers"])


def _normal(gen, *shape, std=1.0):
    return torch.randn(shape, generator=gen, device="cuda") * std


def _weights(c, gen):
    Z, A, H, K = c["Z"], c["A"], c["H"], c["K"]
    shapes = dict(W_lstm=(Z + A + H, 4 * H), b_lstm=(4 * H,), W_mdn=(H, 3 * K * Z), b_mdn=(3 * K * Z,), w_rew=(H,),
                  w_done=(H,), W_ctrl=(Z + H, A), b_ctrl=(A,), w_rt=(H,), w_mem=(H,))
    w = {n: _normal(gen, *s, std=0.05) for n, s in shapes.items()}
    scalars = _normal(gen, 4, std=0.05).tolist()
    w.update(zip(("b_rew", "b_done", "b_rt", "b_mem"), scalars))
    return w


def _pack_bits(valid):
    """bool [..., n] -> little-endian 32-bit words [..., ceil(n / 32)]."""
    n = valid.shape[-1]
    pad = -n % 32
    if pad:
        valid = torch.nn.functional.pad(valid, (0, pad))
    bits = valid.view(*valid.shape[:-1], -1, 32).long() << torch.arange(32, device=valid.device)
    words = bits.sum(-1)
    return torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32)


def _inputs(c, gen):
    Z, A, H, B, T = c["Z"], c["A"], c["H"], c["B"], c["T"]
    x = {}
    if c["kind"] in ("score", "train"):
        x["z_seq"] = _normal(gen, T + 1, B, Z)
        x["actions"] = torch.randint(0, A, (T, B), generator=gen, device="cuda", dtype=torch.int32)
        if c["ragged"]:
            x["lengths"] = torch.randint(1, T + 1, (B,), generator=gen, device="cuda", dtype=torch.int32)
        return x
    x["z0"] = _normal(gen, B, Z)
    if c["carried"]:
        x["h0"] = torch.tanh(_normal(gen, B, H, std=0.3))
        x["c0"] = _normal(gen, B, H, std=0.4)
    if c["shaped"]:
        x["rt0"], x["mem0"] = _normal(gen, B, std=0.5), _normal(gen, B, std=0.5)
    masks, loc = [], []
    NX = c["xfers"]
    L = A - NX
    for _ in range(T):
        if not NX:
            masks.append(_pack_bits(torch.rand((B, A), generator=gen, device="cuda") < c["density"]))
            continue
        # every substitution has some number of places in the graph (none: it is invalid); the
        # last one is the NO-OP, which is always valid and has no place
        n = torch.randint(1, L + 1, (B, NX), generator=gen, device="cuda")
        n *= torch.rand((B, NX), generator=gen, device="cuda") < c["density"]
        n[:, -1] = 0
        valid = torch.zeros((B, A), dtype=torch.bool, device="cuda")
        valid[:, :NX] = n > 0
        valid[:, NX - 1] = True
        masks.append(_pack_bits(valid))
        k = (n[..., None] - 32 * torch.arange((L + 31) // 32, device="cuda")).clamp(0, 32)
        words = (torch.ones_like(k) << k) - 1
        loc.append(torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32))
    x["mask"] = torch.stack(masks)
    if NX:
        x["loc_mask"] = torch.stack(loc)
    if c["pop"]:
        x["W_pop"] = _normal(gen, c["pop"], Z + H, A, std=0.05)
        x["b_pop"] = _normal(gen, c["pop"], A, std=0.05)
    return x


def _all(c, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return _weights(c, gen), _inputs(c, gen)


def prepare(case, seed):
    c = dict(case)
    w, x = _all(c, seed)
    model = pkg.load().WorldModel(_cfg(c), w)
    if c["pop"]:
        model.set_controllers(x.pop("W_pop"), x.pop("b_pop"), pop_group=c["B"] // c["pop"])
    return dict(case=c, model=model, x=x)


def run(state):
    c, m, x = state["case"], state["model"], state["x"]
    if c["kind"] == "train":
        return m.mdn_nll_backward(x["z_seq"], x["actions"], lengths=x.get("lengths"))
    if c["kind"] == "score":
        return m.mdn_nll(x["z_seq"], x["actions"], lengths=x.get("lengths"), want_seq=c["seqs"])
    out = m.rollout(x["z0"], c["T"], mask=x["mask"], loc_mask=x.get("loc_mask"), h0=x.get("h0"), c0=x.get("c0"),
                    rt0=x.get("rt0"), mem0=x.get("mem0"), want_seq=c["seqs"])
    if c["kind"] == "generation":
        out.update(m.returns(out["rewards"], out["done"], 0.99, stop_at_done=False, want_fitness=True))
    return out


# ------------------------------------------------------------------ work and tolerance
def work(case):
    c = case
    Z, A, H, K, B, T = (c[k] for k in ("Z", "A", "H", "K", "B", "T"))
    KX, M = Z + H, 3 * K * Z
    el = 2 if c["precision"] == "bf16" else 4
    gates, heads, ctrl = 2 * KX * 4 * H, 2 * H * (M + 2), 2 * KX * A
    weights = (KX + A) * 4 * H + H * M
    if c["kind"] in ("score", "train"):
        rows = B * T
        flops = rows * (gates + heads)
        nbytes = el * weights + 4 * ((T + 1) * B * Z + rows + B)
        if c["kind"] == "train":  # and both operands' gradients of every product
            flops *= 3
            nbytes += 4 * weights
        if c["seqs"]:
            nbytes += 4 * rows * (2 * H + M)
        return dict(bytes=float(nbytes), flops=float(flops))
    live = min(float(T), LIVE_STEPS) if c["done"] else float(T)
    words = (A + 31) // 32
    P = max(1, c["pop"])
    flops = B * live * (gates + heads + ctrl)
    nbytes = el * (weights + P * KX * A) + 4 * (B * Z + B * live * words)  # weights, z0, masks read
    nbytes += 4 * B * T * Z + 9 * B * T + 8 * B * H  # z, actions, rewards, done; the final h, c
    if c["xfers"]:
        nbytes += 4 * B * T * (1 + (A - c["xfers"] + 31) // 32)
    if c["carried"]:
        nbytes += 8 * B * H
    if c["seqs"]:
        nbytes += B * T * (4 * (2 * H + M) + Z)
    if c["kind"] == "generation":
        nbytes += 9 * B * T
    return dict(bytes=float(nbytes), flops=float(flops))


def tolerance(case):
    """About four times the distance between two kernel families on the same inputs.  Scoring and
    training are smooth (fp32 likelihoods 7e-8 apart, bf16 ones 1e-6, bf16 hidden states and head
    outputs 9e-4, gradients 7e-6 and 1e-3).  A rollout takes an action and Z mixture components
    per step by comparing floats: sums in another order flip a few of these and the flipped
    episode goes on from there (2e-4 to 8e-2 apart, with up to 2% of the choices of a sampled
    controller)."""
    c = case
    f32 = c["precision"] == "fp32"
    if c["kind"] == "score":
        return {"rel": (2e-5 if f32 else 4e-3) if c["seqs"] else (1e-6 if f32 else 1e-5)}
    if c["kind"] == "train":
        return {"rel": 4e-5 if f32 else 5e-3}
    return {"rel": 0.03, "max": 0.99, "differ": 0.01}


# ------------------------------------------------------------------ the same in 64 bits
def _philox(ep, step, purpose, block, seed):
    """Philox-4x32-10 words of the counter (ep lo, step, purpose << 24 | block, ep hi)."""
    low = 0xFFFFFFFF
    c = [ep & low, torch.full_like(ep, step & low), (block | (purpose << 24)) & low, (ep >> 32) & low]
    k0, k1 = seed & low, (seed >> 32) & low
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & low) ^ c[1] ^ k0, p1 & low, ((p0 >> 32) & low) ^ c[3] ^ k1, p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return c


def _uniform(word):
    return (word >> 8).double() * 2.0**-24


def _draws(c, t):
    """(component uniforms, normals) [B, Z] and the controller's two uniforms [B] of step t."""
    B, Z, seed = c["B"], c["Z"], _cfg(c)["seed"]
    nb = (Z + 3) // 4
    ep = torch.arange(B, device="cuda")[:, None].expand(B, nb).contiguous()
    block = torch.arange(nb, device="cuda")[None].expand(B, nb).contiguous()
    u = torch.stack([_uniform(w) for w in _philox(ep, t, 0, block, seed)], -1).view(B, -1)[:, :Z]
    n = [_uniform(w) for w in _philox(ep, t, 1, block, seed)]
    pairs = []
    for i in (0, 2):
        r, a = torch.sqrt(-2.0 * torch.log1p(-n[i])), 2.0 * math.pi * n[i + 1]
        pairs += [r * torch.cos(a), r * torch.sin(a)]
    eps = torch.stack(pairs, -1).view(B, -1)[:, :Z]
    e = torch.arange(B, device="cuda")
    v = _philox(e, t, 2, torch.zeros_like(e), seed)
    return u, eps, _uniform(v[0]), _uniform(v[1])


def _unpack_bits(words, n):
    w = words.long()[..., None] >> torch.arange(32, device=words.device)
    return (w & 1).bool().flatten(-2)[..., :n]


def _choose(logits, valid, u, sampled):
    """Masked argmax, or the inverse CDF of softmax over the valid ones; -1 where none is."""
    l = torch.where(valid, logits, -math.inf)
    top, a = l.max(-1)
    if sampled:
        p = torch.where(valid, torch.exp(l - top[:, None]), 0.0)
        hit = (torch.cumsum(p, -1) > (u * p.sum(-1))[:, None]) & valid
        a = hit.int().argmax(-1)
    return torch.where(valid.any(-1), a, -1)


def _cell(w, Z, A, H, z, h, c, acts):
    g = z @ w["W_lstm"][:Z] + h @ w["W_lstm"][Z + A:] + w["b_lstm"]
    for a in acts:
        g = g + torch.where(a[:, None] >= 0, w["W_lstm"][Z + a.clamp(min=0)], 0.0)
    i, f, g, o = g.split(H, -1)
    c = torch.sigmoid(f) * c + torch.sigmoid(i) * torch.tanh(g)
    return torch.sigmoid(o) * torch.tanh(c), c


def exact(case, seed):
    """What run() returns, in 64 bits throughout (a bf16 model's weight matrices are bf16 numbers)."""
    c = dict(case)
    Z, A, H, K, B, T, NX = (c[k] for k in ("Z", "A", "H", "K", "B", "T", "xfers"))
    # a done flag that flips replaces the rest of its episode; and the largest call takes minutes
    if c["done"] or work(c)["flops"] > 8e12:
        return None
    w, x = _all(c, seed)
    if c["precision"] == "bf16":
        for n in ("W_lstm", "W_mdn", "w_rew", "w_done", "W_ctrl", "w_rt", "w_mem"):
            w[n] = w[n].bfloat16()
        if c["pop"]:
            x["W_pop"] = x["W_pop"].bfloat16()
    f64 = lambda v: v.double() if torch.is_tensor(v) and v.is_floating_point() else v  # noqa: E731
    w, x = {n: f64(v) for n, v in w.items()}, {n: f64(v) for n, v in x.items()}
    h = x.get("h0", torch.zeros((B, H), dtype=torch.float64, device="cuda"))
    cc = x.get("c0", torch.zeros_like(h))
    if c["kind"] in ("score", "train"):
        names = ("W_lstm", "b_lstm", "W_mdn", "b_mdn")
        train = c["kind"] == "train"
        for n in names:
            w[n].requires_grad_(train)
        seqs = dict(h_seq=[], c_seq=[], mdn_seq=[])
        nll = torch.zeros(B, dtype=torch.float64, device="cuda")
        lengths = x.get("lengths", torch.full((B,), T, device="cuda"))
        for t in range(T):
            h, cc = _cell(w, Z, A, H, x["z_seq"][t], h, cc, [x["actions"][t].long()])
            md = h @ w["W_mdn"] + w["b_mdn"]
            lg, mu, ls = (v.view(B, Z, K) for v in md.split(K * Z, -1))
            zs = (x["z_seq"][t + 1][..., None] - mu) * torch.exp(-ls)
            lp = torch.log_softmax(lg, -1) - 0.5 * zs * zs - ls - 0.5 * math.log(2.0 * math.pi)
            nll = nll - torch.where(t < lengths, torch.logsumexp(lp, -1).sum(-1), 0.0)
            if c["seqs"]:
                for n, v in zip(("h_seq", "c_seq", "mdn_seq"), (h, cc, md)):
                    seqs[n].append(v)
        if train:
            grads = torch.autograd.grad(nll.sum(), [w[n] for n in names])
            return dict(zip(names, grads), nll=nll.detach())
        return dict({n: torch.stack(v) for n, v in seqs.items() if v}, nll=nll)
    out = {n: [] for n in ("z", "rewards", "h_seq", "c_seq", "mdn_seq", "rt_seq", "mem_seq")}
    z = x["z0"]
    out["z"].append(z)
    rt, mem = x.get("rt0"), x.get("mem0")
    per = B // max(1, c["pop"])
    for t in range(T):
        u, eps, ua, ul = _draws(c, t)
        if c["pop"]:
            zh = torch.cat([z, h], -1).view(c["pop"], per, -1)
            logits = (zh @ x["W_pop"] + x["b_pop"][:, None]).view(B, A)
        else:
            logits = torch.cat([z, h], -1) @ w["W_ctrl"] + w["b_ctrl"]
        valid = _unpack_bits(x["mask"][t], A)
        acts = [_choose(logits[:, :NX] if NX else logits, valid[:, :NX] if NX else valid, ua, c["sampled"])]
        taken = acts[0] >= 0
        if NX:
            lm = x["loc_mask"][t][torch.arange(B, device="cuda"), acts[0].clamp(min=0)]
            loc = _choose(logits[:, NX:], _unpack_bits(lm, A - NX), ul, c["sampled"])
            loc = torch.where((acts[0] < 0) | (acts[0] == NX - 1), -1, loc)
            taken &= (acts[0] == NX - 1) | (loc >= 0)
            acts.append(torch.where(loc >= 0, NX + loc, -1))
        h, cc = _cell(w, Z, A, H, z, h, cc, acts)
        md = h @ w["W_mdn"] + w["b_mdn"]
        lg, mu, ls = (v.view(B, Z, K) for v in md.split(K * Z, -1))
        cum = torch.cumsum(torch.softmax(lg, -1), -1)[..., :-1]
        k = (cum <= u[..., None]).sum(-1, keepdim=True)
        z = (mu.gather(-1, k) + torch.exp(ls.gather(-1, k)) * eps[..., None]).squeeze(-1)
        r = h @ w["w_rew"] + w["b_rew"]
        if c["shaped"]:
            rt1, mem1 = h @ w["w_rt"] + w["b_rt"], h @ w["w_mem"] + w["b_mem"]
            r = torch.where(taken, 0.8 * (rt - rt1) + 0.2 * (mem - mem1), -100.0)
            rt, mem = rt1, mem1
            out["rt_seq"].append(rt)
            out["mem_seq"].append(mem)
        out["z"].append(z)
        out["rewards"].append(r)
        if c["seqs"]:
            for n, v in zip(("h_seq", "c_seq", "mdn_seq"), (h, cc, md)):
                out[n].append(v)
    out = {n: torch.stack(v) for n, v in out.items() if v}
    out.update(h_final=h, c_final=cc)
    if c["kind"] == "generation":
        g, ret = torch.zeros(B, dtype=torch.float64, device="cuda"), []
        for t in reversed(range(T)):
            g = out["rewards"][t] + 0.99 * g
            ret.append(g)
        out["returns"] = torch.stack(ret[::-1])
        out["fitness"] = out["returns"][0].view(c["pop"], per).mean(-1)
    return out
