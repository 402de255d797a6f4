"""The optimizer steps whose speed and results are measured.

A case is one call (or one training step's calls) of the package's public
entry points on a parameter set in the middle of a run: weights, optimizer
state and update history are populated, the step counter stands at ``K0``, so
Error Feedback is active and no bias correction is degenerate. ``run`` steps
and returns every arena the step writes. Sizes are those of the repository's
own parameter sets (a flat 2^20 vector, GPT-2 small, Llama-1B and Llama-7B
shapes) and of its tests, with generic ragged ones beside them.

Three kinds of case:
  "step"  one DelayedAdamW step (any rule, correction, dtype and stash mode)
  "muon"  one DelayedMuon step; with ``vectors`` the whole training step of a
          model whose other tensors take AdamW, both clipped from one norm
  "norm"  dpo_grad_norm_noalloc, the gradient norm without allocation
"""
import math

import numpy as np
import torch

from paper_2606_30634_gb300 import dpo, muon

K0 = 100           # gradients consumed before the measured call
ALIGN = 128        # arena alignment of every tensor, in elements
LR, MUON_LR = 3e-4, 2e-3
BETA1, BETA2, BETA3, EPS, WD, PSI = 0.9, 0.95, 0.99, 1e-8, 0.1, 0.004
MU, NS_EPS, RMS, NS = 0.95, 1e-7, 0.2, (3.4445, -4.7750, 2.0315)
RULES = {"adamw": 0, "nadam": 1, "lion": 2, "adan": 3}
CORR = {"ef": 0, "sapipe-same": 1, "sapipe-updated": 2}   # "none": no history buffer
DT = {"f32": dpo.DPO_F32, "bf16": dpo.DPO_BF16}
TDT = {"f32": torch.float32, "bf16": torch.bfloat16}


# ------------------------------------------------------------------ sets ----

def _gpt2(layers=12):
    d, ffn, t = 768, 3072, [50257 * 768, 1024 * 768]
    for _ in range(layers):
        t += [d, d, d * 3 * d, 3 * d, d * d, d, d, d, d * ffn, ffn, ffn * d, d]
    return t + [d, d]


def _llama(d, ffn, n_kv, layers, vocab=0):
    t = [vocab * d] if vocab else []
    for _ in range(layers):
        t += [d * d, n_kv * d, n_kv * d, d * d, ffn * d, ffn * d, d * ffn, d, d]
    return t + ([d] if vocab else [])


def _ragged(total, n, salt):
    """n tensor sizes that sum to about total, spread over two decades."""
    g = np.random.RandomState(salt)
    w = 10.0 ** g.uniform(-2, 0, n)
    return [max(1, int(total * x / w.sum())) | 1 for x in w]


def _numels(case):
    s = case["set"]
    if s == "flat":
        return [case["n"]]
    if s == "odd-few":       # a handful of tiny and odd tensors
        return [1, 8, 4099, 70_001, 13]
    if s == "gpt2":
        return _gpt2()
    if s == "llama-1b":
        return _llama(2048, 8192, 512, 16, 128256)
    if s == "llama-7b-layer":
        return _llama(4096, 11008, 4096, 1)
    return _ragged(case["n"], case["tensors"], case["salt"])


def _shapes(case):
    s = case["set"]
    if s == "pair":          # one wide and one tall matrix
        return [(256, 768), (768, 256)]
    if s == "gpt2":
        return [(768, 2304), (768, 768), (768, 3072), (3072, 768)] * 12
    if s == "odd-few":
        return [(300, 700), (64, 96), (777, 1555), (1000, 3001), (2050, 517)]
    if s == "llama-1b-4layers":
        return [(2048, 2048), (512, 2048), (512, 2048), (2048, 2048), (8192, 2048),
                (8192, 2048), (2048, 8192)] * 4
    if s == "llama-7b-layer":
        return [(4096, 4096)] * 4 + [(11008, 4096)] * 2 + [(4096, 11008)]
    d, f = case["d"], case["ffn"]   # "block": attention and MLP matrices of width d
    return [(d, 3 * d), (d, d), (d, f), (f, d)] * case["layers"]


def _vectors(case):
    """The tensors beside a model's matrices: embedding, norms and biases."""
    return [50257 * 768, 1024 * 768] + [768, 768, 2304, 768, 768, 768, 3072, 768] * 12 + [768, 768]


def listed():
    return [
        # the smallest calls: a few odd tensors, clipped; launches and latency count
        dict(name="adamw-odd-few", kind="step", set="odd-few", rule="adamw", corr="ef",
             param="bf16", stash="bf16", grad="bf16", clip=0.03, mode="copy"),
        # one flat fp32 vector, all state fp32
        dict(name="adamw-flat-1m", kind="step", set="flat", n=1 << 20, rule="adamw", corr="ef",
             param="f32", stash="f32", grad="f32", clip=0.0, mode="copy"),
        # many small and odd tensors, SAPipe-WP, half of them synchronous (WPipe)
        dict(name="nadam-ragged-6m-wpipe", kind="step", set="ragged", n=6_000_000, tensors=60,
             salt=7, rule="nadam", corr="sapipe-same", param="bf16", stash="bf16", grad="f32",
             clip=1.0, mode="copy", half_sync=True),
        # GPT-2 small, fp32 stash: the ordinary step of a small model
        dict(name="adamw-gpt2", kind="step", set="gpt2", rule="adamw", corr="ef", param="bf16",
             stash="f32", grad="bf16", clip=0.0, mode="copy"),
        # one 7B decoder layer (a pipeline stage's share), Adan, ping-pong stash
        dict(name="adan-7b-layer-pingpong", kind="step", set="llama-7b-layer", rule="adan",
             corr="ef", param="bf16", stash="bf16", grad="bf16", clip=0.0, mode="pingpong"),
        # Llama-1B with global-norm clipping: the largest step
        dict(name="adamw-llama-1b-clip", kind="step", set="llama-1b", rule="adamw", corr="ef",
             param="bf16", stash="f32", grad="bf16", clip=1.0, mode="copy"),
        # the allocation-free norm on a 4M-element fp32 gradient
        dict(name="norm-4m", kind="norm", n=(1 << 22) + 5, grad="f32", clip=1.0),
        # delayed Muon, from two small matrices to a 7B decoder layer
        dict(name="muon-pair", kind="muon", set="pair", corr="ef", stash="bf16", grad="bf16",
             clip=0.0, vectors=False),
        dict(name="muon-odd-few", kind="muon", set="odd-few", corr="ef", stash="f32",
             grad="f32", clip=0.0, vectors=False),
        # GPT-2's whole training step: Muon on the matrices, AdamW on the rest, one norm
        dict(name="muon-gpt2-whole", kind="muon", set="gpt2", corr="ef", stash="bf16",
             grad="bf16", clip=1.0, vectors=True),
        dict(name="muon-1b-4layers", kind="muon", set="llama-1b-4layers", corr="none",
             stash="bf16", grad="bf16", clip=1.0, vectors=False),
        dict(name="muon-7b-layer", kind="muon", set="llama-7b-layer", corr="ef", stash="bf16",
             grad="bf16", clip=0.0, vectors=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "muon", "muon", "muon", "norm"])
    grad = rng.choice(["bf16", "bf16", "f32"])
    if kind == "norm":
        return dict(kind="norm", n=_log(rng, 1000, 1 << 28), grad=grad, clip=1.0)
    if kind == "step":
        corr = rng.choice(["ef", "ef", "none", "sapipe-same", "sapipe-updated"])
        param = rng.choice(["bf16", "bf16", "f32"])
        stash = rng.choice(["bf16", "f32"])
        pp = param == stash == "bf16" and corr in ("ef", "none")
        n = _log(rng, 50_000, 250_000_000)
        return dict(kind="step", set="ragged", n=n, tensors=rng.randint(1, 150),
                    salt=rng.randint(0, 1 << 20), rule=rng.choice(["adamw", "adamw", *RULES]),
                    corr=corr, param=param, stash=stash, grad=grad,
                    clip=rng.choice([0.0, 1.0]),
                    mode=rng.choice(["copy", "pingpong"]) if pp else "copy",
                    half_sync=rng.random() < 0.2)
    d = _log(rng, 128, 2560)
    if rng.random() < 0.6:
        d = -(-d // 64) * 64          # most models' widths are round
    ffn = rng.choice([4 * d, (8 * d // 3 + 63) // 64 * 64, 3 * d + rng.randint(1, 63)])
    per = 4 * d * d + 2 * d * ffn     # parameters of one layer
    most = max(1, min(24, 200_000_000 // per, int(6e12 / (6 * d * per))))
    return dict(kind="muon", set="block", d=d, ffn=ffn, layers=rng.randint(1, most),
                corr=rng.choice(["ef", "ef", "none", "sapipe-same"]),
                stash=rng.choice(["bf16", "f32"]), grad=grad, clip=rng.choice([0.0, 1.0]),
                vectors=False)


# ---------------------------------------------------------------- inputs ----

def _offsets(numels):
    offs, o = [], 0
    for n in numels:
        offs.append(o)
        o += -(-n // ALIGN) * ALIGN
    return offs, max(o, ALIGN)


NAMES = ("master", "m", "v", "n", "grad_prev", "ef", "grad", "stash", "vector")


def _draw(total, seed, name, scale):
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 16 + NAMES.index(name)) % (1 << 62))
    return torch.randn(total, device="cuda", generator=g).mul_(scale)


def _input(name, total, seed, lr, grad):
    """One arena of a run's state: N(0, 0.02^2) weights, N(0, 1e-3^2) gradients
    in the gradient dtype, moments and history of their steady size."""
    if name in ("v", "n"):
        return _draw(total, seed, name, 0.3).add_(1.0).mul_(1e-3).square_()
    if name in ("grad", "grad_prev"):
        return _draw(total, seed, name, 1e-3).to(TDT[grad if name == "grad" else "f32"])
    return _draw(total, seed, name, {"master": 0.02, "m": 2.3e-4, "ef": 0.5 * lr}[name])


def _adam(numels, case, seed, **kw):
    """A DelayedAdamW context K0 steps into a run."""
    corr = case["corr"]
    sync = [case.get("half_sync", False) and i >= len(numels) // 2 for i in range(len(numels))]
    opt = dpo.DelayedAdamW(
        numels, param_dtype=DT[case["param"]], stash_dtype=DT[case["stash"]],
        grad_dtype=DT[case["grad"]], lr=LR, beta1=BETA1, beta2=BETA2, eps=EPS, weight_decay=WD,
        ef=corr != "none", max_grad_norm=case["clip"], correction=CORR.get(corr, 0), sync=sync,
        optimizer=RULES[case["rule"]], beta3=BETA3, momentum_decay=PSI,
        stash_mode=dpo.DPO_STASH_PINGPONG if case["mode"] == "pingpong" else dpo.DPO_STASH_COPY,
        init_mode=dpo.DPO_INIT_RESUME, **kw)
    total = opt.layout.total
    for name in ("master", "m", "v", "n", "grad_prev", "ef", "grad"):
        if getattr(opt, name) is not None:
            src = "v" if name == "v" and case["rule"] == "adan" else name
            a = _input(src, total, seed, LR, case["grad"])
            getattr(opt, name).copy_(a.sqrt_().mul_(0.1) if src == "v" and
                                     case["rule"] == "adan" else a)
    if opt.param is not None:
        opt.param.copy_(opt.master)
    opt.stash.copy_(opt.master)
    dpo.dpo_set_step(opt.ctx, K0)
    return opt


def _muon(case, seed):
    shapes = _shapes(case)
    m = muon.DelayedMuon(
        shapes, stash_dtype=DT[case["stash"]], grad_dtype=DT[case["grad"]], lr=MUON_LR,
        momentum=MU, weight_decay=WD, ef=case["corr"] != "none", max_grad_norm=case["clip"],
        coeffs=NS, ns_eps=NS_EPS, rms_scale=RMS, ns_steps=5, init_mode=dpo.DPO_INIT_RESUME,
        correction=CORR.get(case["corr"], 0))
    total = m.master.numel()
    for name, arena in (("master", m.master), ("m", m.mom), ("ef", m.ef), ("grad", m.grad)):
        if arena is not None:
            arena.copy_(_input(name, total, seed, MUON_LR, case["grad"]))
    m.param.copy_(m.master)
    m.stash.copy_(m.master)
    m.set_step(K0)
    return m


def _vector_case(case):
    return dict(rule="adamw", corr="ef", param="bf16", stash="bf16", grad="bf16",
                clip=case["clip"], mode="copy")


def prepare(case, seed):
    if case["kind"] == "norm":
        return dict(kind="norm", n=case["n"], dt=DT[case["grad"]], clip=case["clip"],
                    grad=_input("grad", case["n"], seed, LR, case["grad"]),
                    norm=torch.zeros(1, dtype=torch.float64, device="cuda"),
                    coef=torch.zeros(1, dtype=torch.float32, device="cuda"))
    if case["kind"] == "step":
        return dict(kind="step", opt=_adam(_numels(case), case, seed))
    s = dict(kind="muon", m=_muon(case, seed), opt=None)
    if case["vectors"]:
        s["opt"] = _adam(_vectors(case), _vector_case(case), seed + 1_000_003)
        s["acc"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["m"].set_clip_source(s["acc"])
        s["opt"].set_clip_source(s["acc"])
    return s


def _adam_out(opt):
    return {n: getattr(opt, n) for n in ("master", "m", "v", "n", "grad_prev", "ef", "param",
                                         "stash") if getattr(opt, n) is not None}


def run(state):
    if state["kind"] == "norm":
        dpo.dpo_grad_norm_noalloc(state["grad"], state["n"], state["dt"], state["clip"],
                                  state["norm"], state["coef"])
        return {"norm": state["norm"], "coef": state["coef"]}
    if state["kind"] == "step":
        state["opt"].step()
        return _adam_out(state["opt"])
    m, opt = state["m"], state["opt"]
    if opt is not None:
        dpo.global_sqnorm([opt, m], state["acc"])
        opt.step()
    m.step()
    out = {n: getattr(m, n) for n in ("master", "mom", "ef", "param", "stash")
           if getattr(m, n) is not None}
    return {"muon": out, "vectors": _adam_out(opt)} if opt is not None else out


# ------------------------------------------------------------------ work ----

def _size(dt):
    return 2 if dt == "bf16" else 4


def _adam_bytes(numels, case):
    """Each input read once and each output written once, per element."""
    n = sum(numels)
    sync = sum(numels[len(numels) // 2:]) if case.get("half_sync") else 0
    states = {"adamw": 2, "nadam": 2, "lion": 1, "adan": 4}[case["rule"]]
    per = 8 * (1 + states) + _size(case["grad"]) + (2 if case["param"] == "bf16" else 0)
    late = ((0 if case["mode"] == "pingpong" else _size(case["stash"])) +
            (8 if case["corr"] != "none" else 0))
    return n * per + (n - sync) * late


def work(case):
    if case["kind"] == "norm":
        return {"bytes": case["n"] * _size(case["grad"]), "flops": 2 * case["n"]}
    if case["kind"] == "step":
        n = _numels(case)
        return {"bytes": _adam_bytes(n, case), "flops": 20 * sum(n)}
    b = f = 0
    for r, c in _shapes(case):
        per = 8 + 8 + _size(case["grad"]) + 2 + _size(case["stash"])
        b += r * c * (per + (8 if case["corr"] != "none" else 0))
        r, c = min(r, c), max(r, c)
        # the unique entries of X X^T and A A, and all of B X
        f += 5 * (r * (r + 1) * c + r * (r + 1) * r + 2 * r * r * c)
    if case["vectors"]:
        b += _adam_bytes(_vectors(case), _vector_case(case))
    return {"bytes": b, "flops": f}


def tolerance(case):
    if case["kind"] == "norm":
        return {"rel": 1e-6, "max": 1e-6}     # fp32 sums of squares, fp64 beyond a thread
    if case["kind"] == "step":
        # fp32 state: a few roundings of 2^-24. A bf16 output may round the
        # other way where the fp32 value is off by one ulp: 2^-8 of the
        # element, on about one element in 10^4.
        bf16 = "bf16" in (case["param"], case["stash"])
        return {"rel": 1e-4, "max": 1e-2} if bf16 else {"rel": 1e-6, "max": 1e-5}
    # Newton-Schulz holds every iterate in bf16: a product within an fp32
    # accumulation error of a rounding boundary rounds the other way, and the
    # flips cascade over five steps. Two correct fp32 accumulations differ by
    # 4e-3 to 6e-3 normwise in O, which the history U = lr (r O + wd X) shows
    # in full; the weights show it scaled by lr.
    return {"rel": 2.4e-2, "max": 0.25}


# ----------------------------------------------------------------- exact ----

def _f32(x):
    return float(np.float32(x))


def _adam_scalars(k):
    b1, b2, b3, lr = _f32(BETA1), _f32(BETA2), _f32(BETA3), _f32(LR)
    mu = lambda i: b1 * (1.0 - 0.5 * 0.96 ** (i * _f32(PSI)))
    prod = math.prod(mu(i) for i in range(1, k + 1))
    return dict(b1=b1, b2=b2, b3=b3, lr=lr, eps=_f32(EPS), wd=_f32(WD), k=k,
                cg=lr * (1 - mu(k)) / (1 - prod), cm=lr * mu(k + 1) / (1 - prod * mu(k + 1)))


def _rule(rule, s, g, x, m, v, n, gp):
    """(update, m, v, n, grad_prev) of one element-wise rule."""
    b1, b2, b3, k, lr = s["b1"], s["b2"], s["b3"], s["k"], s["lr"]
    decay = lr * s["wd"] * x
    if rule == "lion":
        return lr * torch.sign(b1 * m + (1 - b1) * g) + decay, b2 * m + (1 - b2) * g, v, n, gp
    if rule == "adan":
        diff = g - gp
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * diff
        n = b3 * n + (1 - b3) * (g + b2 * diff).square()
        den = (n / (1 - b3 ** k)).sqrt() + s["eps"]
        return lr * (m / (1 - b1 ** k) + b2 * v / (1 - b2 ** k)) / den + decay, m, v, n, g
    m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
    den = (v / (1 - b2 ** k)).sqrt() + s["eps"]
    if rule == "adamw":
        return lr * (m / (1 - b1 ** k)) / den + decay, m, v, n, gp
    return (s["cg"] * g + s["cm"] * m) / den + decay, m, v, n, gp


def _exact_adam(numels, case, seed, coef):
    rule, corr = case["rule"], case["corr"]
    offs, total = _offsets(numels)
    names = ["master", "m", "grad"] + (["v"] if rule != "lion" else [])
    names += (["n", "grad_prev"] if rule == "adan" else []) + (["ef"] if corr != "none" else [])
    a = {n: _input(n, total, seed, LR, case["grad"]).double() for n in names}
    if rule == "adan":
        a["v"] = _input("v", total, seed, LR, case["grad"]).sqrt_().mul_(0.1).double()
    g = a.pop("grad")
    if coef is None:
        sq = sum(float(g[o:o + n].square().sum()) for o, n in zip(offs, numels))
        coef = min(1.0, _f32(case["clip"]) / (math.sqrt(sq) + 1e-6)) if case["clip"] > 0 else 1.0
    w16 = a["master"].float().to(torch.bfloat16).double()
    out = dict(a)
    if case["param"] == "bf16":
        out["param"] = w16.clone()
    out["stash"] = w16 if case["stash"] == "bf16" else a["master"].clone()
    s, s2 = _adam_scalars(K0 + 1), _adam_scalars(K0 + 2)
    half = len(numels) // 2 if case.get("half_sync") else len(numels)
    for i, (o, n) in enumerate(zip(offs, numels)):
        late = i < half
        for lo in range(o, o + n, 1 << 26):
            q = slice(lo, min(lo + (1 << 26), o + n))
            at = lambda name: a[name][q] if name in a else None
            x, gc = at("master"), g[q] * coef
            u, m, v, nn, gp = _rule(rule, s, gc, x, at("m"), at("v"), at("n"), at("grad_prev"))
            x1 = x - u
            if late and corr == "ef":
                x1 = x - (2.0 * u - at("ef"))
            if late and case["mode"] != "pingpong":
                out["stash"][q] = x - at("ef") if corr.startswith("sapipe") else x
            if late and corr == "sapipe-updated":
                u = _rule(rule, s2, gc, x1, m, v, nn, gp)[0]
            for name, val in (("m", m), ("v", v), ("n", nn), ("grad_prev", gp)):
                if name in a:
                    out[name][q] = val
            if late and corr != "none":
                out["ef"][q] = u
            if case["param"] == "bf16":
                # ping-pong: an odd call writes delayed tensors' weights to the stash buffer
                out["stash" if late and case["mode"] == "pingpong" else "param"][q] = x1
            out["master"][q] = x1
    return out


def _newton_schulz(x):
    x = x / (torch.linalg.norm(x) + _f32(NS_EPS))
    tall = x.shape[0] > x.shape[1]
    x = x.T if tall else x
    a, b, c = (_f32(v) for v in NS)
    for _ in range(5):
        g = x @ x.T
        x = a * x + (b * g + c * (g @ g)) @ x
    return x.T if tall else x


def _exact_muon(case, seed, coef):
    shapes = _shapes(case)
    offs, total = _offsets([r * c for r, c in shapes])
    get = lambda n: _input(n, total, seed, MUON_LR, case["grad"]).double()
    x, m, g = get("master"), get("m"), get("grad")
    ef = get("ef") if case["corr"] != "none" else None
    if coef is None:
        sq = sum(float(g[o:o + r * c].square().sum()) for o, (r, c) in zip(offs, shapes))
        coef = min(1.0, _f32(case["clip"]) / (math.sqrt(sq) + 1e-6)) if case["clip"] > 0 else 1.0
    mu, lr, wd, rms = _f32(MU), _f32(MUON_LR), _f32(WD), _f32(RMS)
    w16 = x.float().to(torch.bfloat16).double()
    out = {"param": w16.clone(), "stash": w16 if case["stash"] == "bf16" else x.clone()}
    for o, (r, c) in zip(offs, shapes):
        q = slice(o, o + r * c)
        m[q] = mu * m[q] + (1 - mu) * (coef * g[q])
        ns = _newton_schulz(m[q].view(r, c)).reshape(-1)
        x0 = x[q].clone()
        u = lr * (rms * math.sqrt(max(r, c)) * ns + wd * x0)
        out["stash"][q] = x0 - ef[q] if case["corr"].startswith("sapipe") else x0
        x[q] = x0 - (2.0 * u - ef[q]) if case["corr"] == "ef" else x0 - u
        out["param"][q] = x[q]
        if ef is not None:
            ef[q] = u
    out.update(master=x, mom=m)
    return out if ef is None else dict(out, ef=ef)


def exact(case, seed):
    if case["kind"] == "norm":
        g = _input("grad", case["n"], seed, LR, case["grad"]).double()
        norm = g.square().sum().sqrt().reshape(1)
        return {"norm": norm, "coef": (case["clip"] / (norm + 1e-6)).clamp(max=1.0)}
    if case["kind"] == "step":
        return _exact_adam(_numels(case), case, seed, None)
    # fp64 matrix products run at about 1 TFLOP/s
    if sum(5 * (4 * min(s) ** 2 * max(s) + 2 * min(s) ** 3) for s in _shapes(case)) > 1.2e13:
        return None
    if not case["vectors"]:
        return _exact_muon(case, seed, None)
    shapes, vec = _shapes(case), _vectors(case)
    sq = 0.0
    for numels, sd in (([r * c for r, c in shapes], seed), (vec, seed + 1_000_003)):
        offs, total = _offsets(numels)
        g = _input("grad", total, sd, LR, "bf16").double()
        sq += sum(float(g[o:o + n].square().sum()) for o, n in zip(offs, numels))
    coef = min(1.0, _f32(case["clip"]) / (math.sqrt(sq) + 1e-6))
    return {"muon": _exact_muon(case, seed, coef),
            "vectors": _exact_adam(vec, _vector_case(case), seed + 1_000_003, coef)}
