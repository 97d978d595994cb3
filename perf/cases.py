"""What the performance of this library is measured on: optimizer steps over whole parameter sets.

A pass is one call of the step a trainer makes: ``SkewAdam.step`` over a handle that owns a
model's tensors, or ``skew_step_tensor_noalloc`` over one tensor. Every case starts where a
trainer resumes from a checkpoint: bf16 weights, this step's gradients, and optimizer state
(M, v, R, C) of the size that such gradients leave after 1000 steps. Rows and columns of a
gradient differ in scale, and so do experts (their loads do).

A case is a parameter set built from a few numbers (``_specs``), hyper-parameters (``policy``,
``eps``, ``clip``) and the entry point:

* ``eps = 1e-30`` is the benchmark's; ``1e-8`` is the paper's and the binding's default;
* ``clip``: the trainer's global gradient-norm clip at 1.0, its factor handed to the step as a
  device scalar;
* ``fp32``: router and vectors kept in fp32, as the paper keeps them;
* ``stack``: an expert weight of all experts kept as one (E, n, m) array.
"""
import math

import numpy as np
import torch

from paper_2607_19058_gb300 import skewadam as S

BACKBONE, EXPERT, ROUTER = 0, 1, 2
TIERED, EXPERT_MOMENTUM, FACTORED_ROUTER, UNIFORM, ADAFACTOR = 0, 1, 2, 3, 4

T0 = 1000            # steps taken before the measured ones
BETA1, BETA2, CLIP_D = 0.9, 0.999, 1.0
SIGMA_W, SIGMA_G = 0.02, 1e-3
SPREAD = 0.3         # log-deviation of the row and column scales of a gradient
DITHER_SEED = 1234
ALIGN = 256          # elements: every tensor starts as an allocation of its own would

_MODEL = {"family": "model", "vocab": 0, "pos": 0, "d": 4096, "kv": 4096, "dense": 0, "blocks": 1, "experts": 0,
          "ffn": 4096, "router": 128, "odd": False, "fp32": False, "stack": False, "loads": "even",
          "policy": TIERED, "eps": 1e-30, "lr": 1e-3, "decay": 0.1, "clip": False}


def _model(name, **kw):
    return {"name": name, **_MODEL, **kw}


def listed():
    return [
        # a toy MoE, the smallest thing that is trained: latency and launches
        _model("toy", vocab=512, d=64, kv=64, dense=256, experts=8, ffn=128, router=8),
        # a set of ragged and odd tensors, from 3 x 5 to 4095 x 1000: tails, one-row matrices, odd
        # widths and vector lengths, some of them fp32
        {"name": "ragged", "family": "ragged", "tensors": 24, "largest": 1 << 22, "layout": 5, "policy": TIERED,
         "eps": 1e-30, "lr": 1e-3, "decay": 0.1, "clip": False},
        # a small MoE model as the paper trains (eps 1e-8, lr 3e-4, decay 0.05, gradient norm
        # clipped at 1.0, router and norms fp32), of width 768 with a 50257-word vocabulary
        _model("model_768", vocab=50257, pos=1024, d=768, kv=768, dense=3072, blocks=4, experts=8, ffn=1536, router=8,
               fp32=True, eps=1e-8, lr=3e-4, decay=0.05, clip=True),
        # one MoE layer of the full model: 128 experts of 4096 x 1024 under uneven loads
        _model("layer_4096x1024", experts=128, ffn=1024, loads="dirichlet"),
        # the full 6.78B-parameter set, the benchmark's workload
        _model("full_6780m", vocab=50304, pos=256, kv=1024, dense=4096, blocks=2, experts=128, ffn=4096),
        # 16 experts of 3 matrices of 4096 x 4096 at the paper's hyper-parameters under the norm clip, a third
        # of the experts without tokens in this step
        _model("paper_hp_850m", kv=1024, experts=16, ffn=4096, loads="zipf", fp32=True, eps=1e-8, lr=3e-4, decay=0.05,
               clip=True),
        # momentum on the experts too, beside awkward backbone shapes
        _model("expert_momentum", vocab=50257, experts=8, ffn=4096, router=127, odd=True, policy=EXPERT_MOMENTUM),
        # fine-grained experts kept as (E, n, m) stacks, widths that are not powers of two
        _model("stacked_3072x1536", d=3072, kv=768, experts=64, ffn=1536, router=64, stack=True, loads="zipf"),
        # the Adafactor comparator over a mid-sized set
        _model("adafactor_2048", vocab=32000, d=2048, kv=512, dense=5632, blocks=2, experts=16, ffn=1408, router=16,
               policy=ADAFACTOR),
        # one tensor without allocations: the paper's embedding (momentum), and an ordinary expert
        {"name": "noalloc_embedding", "family": "noalloc", "rows": 50304, "cols": 4096, "tier": BACKBONE,
         "policy": TIERED, "eps": 1e-8, "lr": 3e-4, "decay": 0.05, "clip": False},
        {"name": "noalloc_expert", "family": "noalloc", "rows": 2048, "cols": 1408, "tier": EXPERT,
         "policy": TIERED, "eps": 1e-8, "lr": 3e-4, "decay": 0.05, "clip": False},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    hp = {"eps": 1e-8, "lr": 3e-4, "decay": 0.05} if rng.random() < 0.5 else {"eps": 1e-30, "lr": 1e-3, "decay": 0.1}
    kind = rng.random()
    if kind < 0.2:
        return {"family": "ragged", "tensors": _log(rng, 4, 60), "largest": _log(rng, 1 << 12, 1 << 24),
                "layout": rng.randrange(1 << 20), "policy": rng.choice((TIERED, UNIFORM, ADAFACTOR)), **hp, "clip": False}
    if kind < 0.35:
        cols = _log(rng, 64, 8192)
        cols = cols if rng.random() < 0.2 else -(-cols // 8) * 8
        rows = min(_log(rng, 64, 60000), (1 << 28) // cols)
        # within the fixed scratch of that entry point, on any path
        rows = min(rows, (3 << 20) // (4 * (-(-cols // 256))), 60000)
        return {"family": "noalloc", "rows": rows, "cols": cols, "tier": rng.choice((BACKBONE, EXPERT)),
                "policy": TIERED, **hp, "clip": False}
    d = 8 * _log(rng, 8, 900)
    if rng.random() < 0.5:
        d = max(64, -(-d // 256) * 256)
    ffn = 8 * max(1, int(d * rng.uniform(0.25, 1.5)) // 8)
    E = _log(rng, 4, 128)
    E = max(2, min(E, (3 << 29) // (3 * d * ffn)))
    policy = rng.choice((TIERED, TIERED, TIERED, EXPERT_MOMENTUM, UNIFORM, ADAFACTOR))
    if policy in (EXPERT_MOMENTUM, UNIFORM):
        E = max(2, E // 3)
    return {**_MODEL, "vocab": rng.choice((0, 8000, 32000, 50257)) if d <= 4096 else 0, "d": d,
            "kv": max(8, d // rng.choice((1, 2, 4)) // 8 * 8), "dense": rng.choice((0, 8 * (d * 3 // 8))), "blocks": rng.choice((1, 2)),
            "experts": E, "ffn": ffn, "router": rng.choice((E, 64, 127)), "odd": rng.random() < 0.2,
            "fp32": rng.random() < 0.5, "stack": rng.random() < 0.5, "loads": rng.choice(("even", "dirichlet", "zipf")),
            "policy": policy, **hp, "clip": hp["eps"] == 1e-8}


# ---------------------------------------------------------------------------
# The parameter sets
# ---------------------------------------------------------------------------
def _specs(c):
    """[(shape, tier, fp32, expert)]: expert is an index, -1 for other tensors, -2 for a stack."""
    f = c["family"]
    if f == "noalloc":
        return [((c["rows"], c["cols"]), c["tier"], False, -1)]
    out = []
    if f == "ragged":
        r = np.random.RandomState(c["layout"])
        for k in range(c["tensors"]):
            n_el = math.exp(r.uniform(math.log(8), math.log(c["largest"]))) if k else c["largest"] * 0.98
            kind, fp32 = r.randint(0, 8), bool(r.randint(0, 5) == 0)
            m = int(round(math.exp(r.uniform(0.0, math.log(min(n_el, 5000))))))
            m = max(1, m - m % 8) if r.randint(0, 2) and m >= 8 else m
            if k == 0:
                m, kind, fp32 = 1000, 0, False
            n = max(1, int(n_el / m))
            if kind < 5:
                out.append(((n, m), (EXPERT, BACKBONE)[kind % 2], fp32, -1))
            elif kind == 5:
                out.append(((n, m), ROUTER, fp32, -1))
            elif kind == 6:
                out.append(((min(int(n_el), 200000),), BACKBONE, fp32, -1))
            else:
                out.append(((3, max(1, n // 3), m), EXPERT, fp32, -2))
        return out
    d, kv, F, E = c["d"], c["kv"], c["ffn"], c["experts"]
    v32 = c["fp32"]
    if c["vocab"]:
        out.append(((c["vocab"], d), BACKBONE, False, -1))
    if c["pos"]:
        out.append(((c["pos"], d), BACKBONE, False, -1))
    for b in range(c["blocks"]):
        out += [((d, d), BACKBONE, False, -1), ((kv, d), BACKBONE, False, -1), ((kv, d), BACKBONE, False, -1),
                ((d, d), BACKBONE, False, -1)]
        out += [((d,), BACKBONE, v32, -1)] * 4  # two norms, weight and bias
        if c["dense"] and (b == 0 or c["blocks"] > 2):
            out += [((c["dense"], d), BACKBONE, False, -1), ((c["dense"], d), BACKBONE, False, -1),
                    ((d, c["dense"]), BACKBONE, False, -1)]
        if E and (b == c["blocks"] - 1 or c["blocks"] > 2):  # a two-block set: one dense, one MoE block
            out.append(((d, c["router"]), ROUTER, v32, -1))
            if c["stack"]:
                out += [((E,) + s, EXPERT, False, -2) for s in ((d, F), (F, d), (d, F))]
            else:
                out += [(s, EXPERT, False, e) for e in range(E) for s in ((d, F), (F, d), (d, F))]
    if c["odd"]:
        out += [((4095, 1000), BACKBONE, False, -1), ((1, 4096), BACKBONE, False, -1)]
    out += [((d,), BACKBONE, v32, -1)] * 2
    return out


def _numel(shape):
    return math.prod(shape)


def _policy(shape, tier, policy):
    """(factored, momentum, decay) of a tensor under an allocation policy (the paper's Sec. 3 and Table 3)."""
    factored = len(shape) > 1 and (tier != ROUTER or policy in (FACTORED_ROUTER, UNIFORM, ADAFACTOR))
    momentum = policy != ADAFACTOR and (tier == BACKBONE or policy == UNIFORM or (tier == EXPERT and policy == EXPERT_MOMENTUM))
    return factored, momentum, tier != ROUTER


def _loads(c, seed, E):
    """Scale of each expert's gradient: 0 for an expert that saw no tokens in this step."""
    kind = c.get("loads", "even")
    r = np.random.RandomState(seed % (1 << 31))
    if kind == "dirichlet":
        e = r.exponential(size=E)
        return np.sqrt(0.5 * E * e / e.sum())
    if kind == "zipf":  # the 40 least loaded of 128 get none
        rank = r.permutation(E)
        return np.where(rank >= E - (40 * E) // 128, 0.0, 1.0)
    return np.ones(E)


def _inputs(c, seed):
    """Weights, gradients and state as plain tensors, from the seed alone."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    specs = _specs(c)
    off, end = [], {False: 0, True: 0}
    for shape, _, f32, _ in specs:
        off.append(end[f32])
        end[f32] += -(-_numel(shape) // ALIGN) * ALIGN
    flat = {}
    for f32, dt in ((False, torch.bfloat16), (True, torch.float32)):
        w = torch.zeros(end[f32], dtype=dt, device=dev)
        g = torch.zeros(end[f32], dtype=dt, device=dev)
        if end[f32]:
            w.normal_(0.0, SIGMA_W, generator=gen)
            g.normal_(0.0, SIGMA_G, generator=gen)
        flat[f32] = (w, g)
    loads = _loads(c, seed, max(1, c.get("experts", 1)))
    policy = c["policy"]
    grown = 1.0 if policy == ADAFACTOR else 1.0 - BETA2 ** T0  # how much of its limit a second moment has
    one = torch.ones((), device=dev)

    def scales(*shape):
        return torch.exp(SPREAD * torch.randn(shape, generator=gen, device=dev))

    ts, gss = [], torch.zeros((), dtype=torch.float64, device=dev)
    for (shape, tier, f32, expert), o in zip(specs, off):
        n_el = _numel(shape)
        w, g = (t[o: o + n_el].view(shape) for t in flat[f32])
        t = {"shape": shape, "tier": tier, "f32": f32, "w": w, "g": g, "M": None, "v": None, "R": None, "C": None}
        factored, momentum, _ = _policy(shape, tier, policy)
        size = one
        if expert == -2 and c["family"] == "model":
            size = torch.tensor(loads, dtype=torch.float32, device=dev).view(-1, 1, 1)
        elif expert >= 0:
            size = torch.tensor(float(loads[expert]), dtype=torch.float32, device=dev)
        if len(shape) > 1:
            r, q = scales(*shape[:-2], shape[-2], 1), scales(*shape[:-2], 1, shape[-1])
            g.mul_((r * size).to(g.dtype)).mul_(q.to(g.dtype))
            # the state of an expert without tokens comes from the steps in which it had some
            past = torch.where(size == 0, one, size) * SIGMA_G
            if factored:
                t["R"] = ((past * r).square() * q.square().mean(-1, keepdim=True)).reshape(-1) * grown
                t["C"] = ((past * q).square() * r.square().mean(-2, keepdim=True)).reshape(-1) * grown
        else:
            past = one * SIGMA_G
        if not factored:
            t["v"] = (past * past * grown * (0.5 + torch.rand(shape, generator=gen, device=dev))).reshape(-1)
        if momentum:
            M = torch.empty(shape, dtype=torch.float32, device=dev).normal_(0.0, 0.23, generator=gen)
            M.mul_(past)
            if len(shape) > 1:
                M.mul_(r).mul_(q)
            t["M"] = M.reshape(-1)
        if c["clip"]:
            gss += torch.linalg.vector_norm(g, dtype=torch.float32).double() ** 2
        ts.append(t)
    gamma = None
    if c["clip"]:  # the trainer's factor, and a past that was clipped as well
        gamma = torch.clamp(1.0 / (gss.sqrt() + 1e-6), max=1.0).float().reshape(1)
        for t in ts:
            for k, p in (("M", 1), ("v", 2), ("R", 2), ("C", 2)):
                if t[k] is not None:
                    t[k].mul_(gamma ** p)
    return ts, flat, gamma


def _state_order(ts):
    """The order of the state buffer: all M, all v (lengths that are multiples of 4 first in each), all R, all C."""
    out = {}
    for k in ("M", "v", "R", "C"):
        have = [(t, e) for t in ts if t[k] is not None for e in range(t["shape"][0] if len(t["shape"]) == 3 else 1)]
        if k in ("M", "v"):
            per = lambda t: _numel(t["shape"][-2:] if len(t["shape"]) == 3 else t["shape"])  # noqa: E731
            have = [x for x in have if per(x[0]) % 4 == 0] + [x for x in have if per(x[0]) % 4]
        out[k] = have
    return out


def _piece(t, k, e):
    E = t["shape"][0] if len(t["shape"]) == 3 else 1
    n = t[k].numel() // E
    return t[k][e * n: (e + 1) * n]


def _state_of(ts):
    """{key: the state arrays of that kind, one after another}."""
    return {k: torch.cat([_piece(t, k, e) for t, e in have]) for k, have in _state_order(ts).items() if have}


class _Run:
    pass


def prepare(case, seed):
    c = case
    ts, flat, gamma = _inputs(c, seed)
    s = _Run()
    s.t, s.lr, s.gamma, s.flat, s.ts = T0, c["lr"], gamma, flat, ts
    s.hp = S.hparams(BETA1, BETA2, c["eps"], CLIP_D, c["decay"], c["policy"])
    parts = _state_of(ts)
    if c["family"] == "noalloc":
        s.opt = None
        state = torch.cat([parts[k] for k in ("M", "v", "R", "C") if k in parts])
    else:
        s.opt = S.SkewAdam([(t["w"], t["g"], t["tier"]) for t in ts], s.hp)
        state = s.opt.state[: s.opt.state_bytes].view(torch.float32)
        state.copy_(torch.cat([parts[k] for k in ("M", "v", "R", "C") if k in parts]))
    s.state = state
    s.out, at = {}, 0
    for k in ("M", "v", "R", "C"):
        if k in parts:
            s.out[k] = state[at: at + parts[k].numel()]
            at += parts[k].numel()
    for f32, key in ((False, "weights"), (True, "weights_fp32")):
        if flat[f32][0].numel():
            s.out[key] = flat[f32][0]
    for t in ts:  # the library's copy is the state now
        t["M"] = t["v"] = t["R"] = t["C"] = None
    return s


def run(state):
    s = state
    s.t += 1
    if s.opt is not None:
        s.opt.step(s.t, s.lr, DITHER_SEED, grad_scale=s.gamma)
    else:
        t = s.ts[0]
        n, m = t["shape"]
        S.skew_step_tensor_noalloc(t["w"].data_ptr(), t["g"].data_ptr(), 2, n, m, t["tier"], 0, s.hp, s.state.data_ptr(),
                                   4 * s.state.numel(), 0, s.t, s.lr, DITHER_SEED,
                                   torch.cuda.current_stream().cuda_stream)
    return s.out


def work(case):
    """Weights read and written, gradients read, state read and written, each once."""
    by = fl = 0
    for shape, tier, f32, _ in _specs(case):
        factored, momentum, _ = _policy(shape, tier, case["policy"])
        n = _numel(shape)
        by += n * (12 if f32 else 6) + (8 * n if momentum else 0)
        E = shape[0] if len(shape) == 3 else 1
        by += 8 * E * (shape[-2] + shape[-1]) if factored else 8 * n
        fl += n * (13 if momentum else 10)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    """Two correct fp32 evaluations differ by a few 1e-8 in the state and, in bf16 weights, by one
    unit in the last place (2^-7 of the value) wherever x is that close to a rounding threshold:
    about one element in 1e5. Measured against ``exact``: 1e-5 to 1.8e-5 on the bf16 weights."""
    return {"rel": 8e-5, "max": 0.02}


# ---------------------------------------------------------------------------
# The step in 64 bits
# ---------------------------------------------------------------------------
def _dither(idx0, count, tid, step, seed):
    """16-bit draws of elements idx0 .. idx0 + count - 1: halves of the words of Philox-4x32-10
    (Salmon et al., SC'11) keyed by the seed and counted by (element / 8, tensor, step)."""
    dev, low = torch.device("cuda"), 0xFFFFFFFF
    b0, b1 = idx0 >> 3, (idx0 + count + 7) >> 3
    blk = torch.arange(b0, b1, dtype=torch.int64, device=dev)
    c = [blk & low, blk >> 32, torch.full_like(blk, tid), torch.full_like(blk, step & low)]
    k0, k1 = seed & low, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # the low 64 bits; the shift is masked
        c = [((p1 >> 32) & low) ^ c[1] ^ k0, p1 & low, ((p0 >> 32) & low) ^ c[3] ^ k1, p0 & low]
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    halves = torch.stack([h for w in c for h in (w & 0xFFFF, w >> 16)], dim=1).reshape(-1)
    return halves[idx0 - 8 * b0: idx0 - 8 * b0 + count]


def exact(case, seed):
    c = case
    total = sum(_numel(s[0]) for s in _specs(c))
    if total > 2_000_000_000:
        return None
    ts, flat, gamma = _inputs(c, seed)
    f = lambda x: float(np.float32(x))  # noqa: E731  # the hyper-parameters are C floats
    t = T0 + 1
    b1, b2, eps, d, lr, lam = f(BETA1), f(BETA2), f(c["eps"]), f(CLIP_D), f(c["lr"]), f(c["decay"])
    bias_m, bias = math.sqrt(1 - b2 ** t) / (1 - b1 ** t), math.sqrt(1 - b2 ** t)
    if c["policy"] == ADAFACTOR:
        b2, bias_m, bias = f(1.0 - t ** -0.8), 1.0, 1.0
    gam = 1.0 if gamma is None else float(gamma)
    # few bf16 weights: the number that rounds the other way is a matter of luck, so x itself stands for them
    rounded = sum(_numel(s[0]) for s in _specs(c) if not s[2]) >= 1 << 24
    new = {False: torch.zeros(flat[False][0].numel(), dtype=torch.float64, device="cuda"),
           True: torch.zeros(flat[True][0].numel(), dtype=torch.float64, device="cuda")}
    for f32 in (False, True):  # what lies between the tensors stays as it was
        new[f32].copy_(flat[f32][0])
    state = [{"shape": x["shape"], **{k: None if x[k] is None else torch.empty(x[k].numel(), dtype=torch.float64, device="cuda")
                                      for k in ("M", "v", "R", "C")}} for x in ts]
    for tid, (x, y) in enumerate(zip(ts, state)):
        shape = x["shape"]
        factored, momentum, decay = _policy(shape, x["tier"], c["policy"])
        E = shape[0] if len(shape) == 3 else 1
        n_el = _numel(shape) // E
        sub = shape[1:] if len(shape) == 3 else shape
        w0 = flat[x["f32"]][0]
        start = (x["w"].data_ptr() - w0.data_ptr()) // w0.element_size()
        for e in range(E):
            w = x["w"].reshape(E, *sub)[e].double()
            g = x["g"].reshape(E, *sub)[e].double().mul_(gam)
            g2 = g * g
            if factored:
                R = b2 * _piece(x, "R", e).double() + (1 - b2) * g2.mean(1)
                C = b2 * _piece(x, "C", e).double() + (1 - b2) * g2.mean(0)
                _piece(y, "R", e).copy_(R)
                _piece(y, "C", e).copy_(C)
                V = torch.outer(R, C / R.mean())
            else:
                V = (b2 * _piece(x, "v", e).double() + (1 - b2) * g2.reshape(-1)).view(sub)
                _piece(y, "v", e).copy_(V.reshape(-1))
            del g2
            if momentum:
                M = b1 * _piece(x, "M", e).double().view(sub) + (1 - b1) * g
                _piece(y, "M", e).copy_(M.reshape(-1))
                U = bias_m * M / V.clamp_(min=eps).sqrt_()
            else:
                U = bias * g / V.clamp_(min=eps).sqrt_()
            rms = U.square().mean().sqrt()
            U /= torch.clamp(rms / d, min=1.0)
            w = w * (1 - lr * lam if decay else 1.0) - lr * U
            w = w.reshape(-1)
            if not x["f32"] and rounded:
                r = _dither(e * n_el, n_el, tid, t, DITHER_SEED)
                bits = w.float().view(torch.int32)
                w = ((bits + r.to(torch.int32)) & -65536).view(torch.float32).double()
            new[x["f32"]][start + e * n_el: start + (e + 1) * n_el] = w
    out = _state_of(state)
    if new[False].numel():
        out["weights"] = new[False]
    if new[True].numel():
        out["weights_fp32"] = new[True]
    return out
