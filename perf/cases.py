"""The timed work of this framework: rounds of Efficient-Adam as a training program has them run.

A program holds one `EARound` (n workers and the server as buffers on one GPU), fills the n workers'
gradients and calls `step(grads, x)` every round -- or, where the gradients become ready one after
another, `worker_compress`, `server_step` and `apply` one by one.  A program that may not allocate
calls `ea_worker_compress_noalloc` with its own buffers.  Every case is one such round (or one such
compress) and returns everything it writes that lives in a buffer of its own: x, the broadcast and
the workers' messages (codes and scales) and the Adam moments; the residuals show in the round after
it.  Sizes run from a 500-dimensional problem, where a round is all latency, to hundreds of millions
of parameters, where it is all memory traffic.
"""
import math

import torch

import paper_2205_14473_gb300 as ea
from paper_2205_14473_gb300 import workloads as W

BETA1, EPS, X_STD = 0.9, 1e-8, 0.02

# A case: api (step | calls | noalloc), d, n, placement (0: Adam at the workers, 1: at the server), the
# quantizers qw / qs of the messages and their scale groups gw / gs (0: one scale for the vector,
# > 0: blocks of that length, -1: one per tensor), ef (error feedback), form (0: the paper's Adam, 1:
# the textbook form), alpha, beta2, and the gradients' distribution and size (grad, std).
# tensors: "" or the shape of the model behind the vector: "resnet18", or "LxW" for L layers of a
# W x W matrix, a bias and two vectors of W (the last layer's matrix cut so that d need not be round).


def _case(name, **kw):
    c = dict(api="step", d=0, n=8, placement=0, qw="sign", gw=4096, qs="sign", gs=4096, ef=True, form=0, alpha=1e-3,
             beta2=0.999, grad="normal", std=1.0, tensors="")
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    r18 = sum(W.resnet18_tensor_sizes())
    return [
        # the paper's convex toy (Section 5.1): 500 dimensions, ten workers, Example 2's quantizer
        _case("toy_500_pow2", d=500, n=10, qw="pow2", qs="pow2", gw=0, gs=0, alpha=1e-4, beta2=0.99, std=1e-3),
        # a small model or one layer of it: one sign scale for the whole vector
        _case("small_65k_sign", d=65_536, n=4, gw=0, gs=0),
        # the quadratic problem at a million parameters, the gradients handed over one by one
        _case("quadratic_1m_sign_calls", api="calls", d=1_000_000, n=8, gw=0, gs=0, alpha=1e-2),
        # ResNet-18: 62 tensors with a sign scale each, sixteen workers, heavy-tailed gradients
        _case("resnet18_16w_sign", d=r18, n=16, gw=-1, gs=-1, tensors="resnet18", grad="student"),
        # the same model with the Adam moments on the server, call by call
        _case("resnet18_16w_sign_server_calls", api="calls", d=r18, n=16, gw=-1, gs=-1, tensors="resnet18",
              grad="student", placement=1),
        # the grid quantizers (4 bits stochastic up, 8 bits down) in short buckets
        _case("buckets512_grid", d=15_000_001, n=8, qw="grid4s", gw=512, qs="grid8", gs=512, grad="outlier", std=1e-3,
              alpha=1e-4),
        # the grid with one largest-magnitude scale for the whole vector, both ways
        _case("whole_30m_grid8", d=30_000_000, n=4, qw="grid8", gw=0, qs="grid8", gs=0, grad="outlier", std=1e-3,
              alpha=1e-4),
        # a caller without allocations: one worker's message of a 40-million vector
        _case("noalloc_40m_sign", api="noalloc", d=40_000_001, n=1, gw=0, gs=0),
        # sixteen workers, the textbook Adam on the server, 4096-blocks
        _case("blocks_20m_16w_sign_server", d=20_000_003, n=16, placement=1, form=1, std=1e-2),
        # an odd size and worker count, grid quantizers, Adam on the server, call by call
        _case("grid_27m_5w_server_calls", api="calls", d=27_000_001, n=5, placement=1, qw="grid4s", qs="grid8",
              grad="outlier", std=1e-3, alpha=1e-4),
        # BERT-base sized: 4-bit stochastic grid up, 8-bit grid down, 4096-blocks
        _case("bert_110m_grid", d=110_000_000, n=8, qw="grid4s", qs="grid8", grad="outlier", std=1e-3, alpha=1e-4),
        # the large end: sign messages in 4096-blocks, a ragged size
        _case("large_400m_sign", d=400_000_007, n=8, std=1e-4, alpha=1e-4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["whole", "whole", "tensors", "blocks", "blocks", "tiles", "tiles", "noalloc"])
    grad = rng.choice(["normal", "outlier", "student"])
    kw = dict(api=rng.choice(["step", "step", "calls"]), placement=rng.randrange(2), form=int(rng.random() < 0.25),
              ef=rng.random() < 0.85, grad=grad, std=10.0 ** rng.randint(-4, 0), alpha=10.0 ** rng.randint(-4, -2))
    signs, grids = ("sign", "sign"), rng.choice([("grid4s", "grid8"), ("grid8", "grid8"), ("grid2", "grid4s"),
                                                  ("grid16", "grid16"), ("sign", "grid8"), ("grid4s", "sign")])
    if kind == "whole":
        d = _log_int(rng, 500, 30_000_000)
        qw, qs = rng.choice([signs, signs, grids, ("pow2", "pow2"), ("full", "full")])
        kw.update(gw=0, gs=0)
    elif kind == "tensors":
        layers, width = rng.randint(1, 40), _log_int(rng, 16, 700)
        kw.update(tensors="%dx%d" % (layers, width), gw=-1, gs=-1)
        d = layers * (width * width + 3 * width) - rng.randrange(width)
        qw, qs = rng.choice([signs, signs, grids])
    elif kind == "blocks":
        g = rng.choice([128, 256, 512, 1000, 1024, 2048, 6000, 8192])
        d = _log_int(rng, 4 * g, 16_000_000)
        qw, qs = rng.choice([signs, grids])
        kw.update(gw=g, gs=g)
    elif kind == "noalloc":
        d = _log_int(rng, 2000, 40_000_000)
        qw = qs = rng.choice(["sign", "grid4s", "grid8"])
        kw.update(api="noalloc", gw=0, gs=0)
    else:
        d = _log_int(rng, 5000, 120_000_000)
        qw, qs = rng.choice([signs, signs, grids])
    n = 1 if kind == "noalloc" else rng.choice([1, 2, 3, 4, 5, 8, 8, 10, 16])
    if d * n > 800_000_000:
        n = 4
    return _case("", d=d, n=n, qw=qw, qs=qs, **kw)


# ------------------------------------------------------------------------------------ a case's parts

def _segments(case):
    if not case["tensors"]:
        return ()
    if case["tensors"] == "resnet18":
        return tuple(W.resnet18_tensor_sizes())
    layers, width = (int(v) for v in case["tensors"].split("x"))
    sizes = [width * width, width, width, width] * layers
    sizes[-4] -= sum(sizes) - case["d"]
    return tuple(sizes)


_KINDS = {"sign": (1, False), "grid2": (2, False), "grid4s": (4, True), "grid8": (8, False), "grid16": (16, False),
          "pow2": (4, False), "full": (32, False)}


def _spec(case, q, group):
    bits, stochastic = _KINDS[q]
    if q == "sign":
        return W.sign_q(group, _segments(case) if group < 0 else ())
    if q == "pow2":
        return W.pow2_q(-17, -11, 4)
    if q == "full":
        return W.identity_q()
    return W.QuantSpec(W.Q_UNIFORM_MAX, bits, group, _segments(case) if group < 0 else (), stochastic)


def _scales(case, q, group):
    """Scale words of a message."""
    if q in ("pow2", "full"):
        return 0
    return 1 if group == 0 else (-(-case["d"] // group) if group > 0 else len(_segments(case)))


def _generator(case, seed, what):
    return torch.Generator(device="cuda").manual_seed(1 + 4096 * (int(seed) % (1 << 40)) + what)


def _x0(case, seed):
    return torch.randn(case["d"], generator=_generator(case, seed, 4000), device="cuda").mul_(X_STD)


def _gradient(case, seed, i):
    """Worker i's gradient: Gaussian; with 1% of the coordinates 100 times larger; or Student-t(3), every
    tensor (or 1/16th of the vector) with a magnitude of its own, log-uniform over four decades."""
    d, gen = case["d"], _generator(case, seed, i)
    g = torch.randn(d, generator=gen, device="cuda")
    if case["grad"] == "outlier":
        g.mul_(torch.where(torch.rand(d, generator=gen, device="cuda") < 0.01, 100.0, 1.0))
    elif case["grad"] == "student":
        chi = torch.randn(d, generator=gen, device="cuda").square_()
        for _ in range(2):
            chi.add_(torch.randn(d, generator=gen, device="cuda").square_())
        g.div_(chi.div_(3.0).sqrt_().clamp_(min=1e-3))
        sizes = _segments(case) or tuple(d * (k + 1) // 16 - d * k // 16 for k in range(16))
        at = 0
        for k, size in enumerate(sizes):  # the magnitudes belong to the model: the same for every worker
            g[at:at + size].mul_(10.0 ** (-4.0 + 4.0 * ((k * 0.6180339887) % 1.0)))
            at += size
    return g.mul_(case["std"])


def _config(case, seed):
    return ea.EAConfig(d=case["d"], n=case["n"], qw=_spec(case, case["qw"], case["gw"]),
                       qs=_spec(case, case["qs"], case["gs"]), alpha=case["alpha"], beta1=BETA1, beta2=case["beta2"],
                       eps=EPS, placement=case["placement"], error_feedback=case["ef"], seed=int(seed),
                       adam_form=case["form"])


def _workers(first, second, n):
    """The n workers' buffers as one [n, ...] view, from the views of the first two."""
    if n == 1:
        return first[None]
    step = (second.data_ptr() - first.data_ptr()) // first.element_size()
    return first.as_strided((n, first.numel()), (step, 1), first.storage_offset())


def prepare(case, seed):
    cfg = _config(case, seed)
    d, n, at_worker = case["d"], case["n"], case["placement"] == 0
    grads = [_gradient(case, seed, i) for i in range(n)]
    if case["api"] == "noalloc":
        dev = grads[0].device
        c, keep = cfg.to_c()
        s = dict(api="noalloc", c=c, keep=keep, g=grads[0], t=0, e=torch.zeros(d, device=dev),
                 codes=torch.zeros(4 * -(-d * cfg.qw.bits // 128), dtype=torch.int32, device=dev),
                 scales=torch.zeros(1, device=dev), stream=torch.cuda.current_stream())
        s["m"] = torch.zeros(d if at_worker else 4, device=dev)
        s["v"] = torch.full((d if at_worker else 4,), EPS if case["form"] == 0 else 0.0, device=dev)
        return s
    rnd = ea.EARound(cfg)
    x = _x0(case, seed)
    out = {"x": x, "codes": rnd.view(ea.EA_VIEW_CODES_SERVER), "scales": rnd.view(ea.EA_VIEW_SCALES_SERVER)}

    def workers(which):
        return _workers(rnd.view(which, 0), rnd.view(which, 1) if n > 1 else None, n)

    out["worker_codes"] = workers(ea.EA_VIEW_CODES_WORKER)
    if _scales(case, case["qw"], case["gw"]):
        out["worker_scales"] = workers(ea.EA_VIEW_SCALES_WORKER)
    if not _scales(case, case["qs"], case["gs"]):
        del out["scales"]
    if at_worker:
        out["m"], out["v"] = workers(ea.EA_VIEW_M), workers(ea.EA_VIEW_V)
    else:
        out["m"], out["v"] = rnd.view(ea.EA_VIEW_M_SERVER), rnd.view(ea.EA_VIEW_V_SERVER)
    return dict(api=case["api"], rnd=rnd, grads=grads, x=x, out=out)


def run(state):
    if state["api"] == "noalloc":
        s = state
        ea.ea_worker_compress_noalloc(s["c"], 0, s["t"], s["g"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(),
                                      s["e"].data_ptr(), s["codes"].data_ptr(), s["scales"].data_ptr(),
                                      s["stream"].cuda_stream)
        s["t"] += 1
        return {k: s[k] for k in ("e", "codes", "scales", "m", "v")}
    rnd, grads, x = state["rnd"], state["grads"], state["x"]
    if state["api"] == "step":
        rnd.step(grads, x)
    else:
        for i, g in enumerate(grads):
            rnd.worker_compress(i, g)
        rnd.server_step()
        rnd.apply(x)
    return state["out"]


def work(case):
    d, n = case["d"], case["n"]
    bw, bs = _KINDS[case["qw"]][0] / 8, _KINDS[case["qs"]][0] / 8
    at_worker = case["placement"] == 0
    # a worker: the gradient read, the residual (and the moments) read and written, the message written
    worker = d * (4 + 8 + (16 if at_worker else 0) + bw) + 4 * _scales(case, case["qw"], case["gw"])
    flops = d * (13 if at_worker else 4)
    if case["api"] == "noalloc":
        return {"bytes": worker, "flops": flops}
    # the server: its residual (and the moments), x and the broadcast
    server = d * (8 + 8 + (0 if at_worker else 16) + bs) + 4 * _scales(case, case["qs"], case["gs"])
    return {"bytes": n * worker + server, "flops": n * flops + d * (n + 14)}


# Largest differences that another correct evaluation in 32 bits may show, by quantizer: (relative, and the
# share of code words that differ).  About four times what one pass shows against the same in 64 bits.  Moments
# agree to 2e-7; what is larger comes from single codes that fall on the other side of a threshold (a sum of
# sixteen signs near zero, a grid point's midpoint) and then move x, or a residual, by a whole step there.
_TOLERANCE = {"sign": (1e-3, 2e-3), "grid2": (1e-5, 4e-4), "grid4s": (1e-5, 4e-4), "grid8": (1e-5, 4e-4),
              "grid16": (1e-5, 0.01), "pow2": (1e-5, 4e-4), "full": (1e-6, 0.01)}


def tolerance(case):
    rel, differ = (max(v) for v in zip(_TOLERANCE[case["qw"]], _TOLERANCE[case["qs"]]))
    if case["api"] == "noalloc":
        rel = max(rel, 5e-3)  # the residual is returned, whose outliers' steps are its largest values
    return {"rel": rel, "max": 0.9, "differ": differ}


# --------------------------------------------------------------------------------- the same in 64 bits

def _philox(seed, who, t, j):
    """The 24-bit uniform variates of coordinates j: Philox4x32-10 (Salmon et al., SC'11), key = seed,
    counter = (j / 4, who, t), word j mod 4."""
    mask, blk = 0xFFFFFFFF, j >> 2
    c = [blk & mask, blk >> 32, torch.full_like(j, who), torch.full_like(j, t)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    w = j & 3
    word = torch.where(w == 0, c[0], torch.where(w == 1, c[1], torch.where(w == 2, c[2], c[3])))
    return (word >> 8).double() * 2.0 ** -24


def _quantize64(case, u, q, group, seed, who):
    """(codes, scales or None, decoded) of one message."""
    bits, stochastic = _KINDS[q]
    d = u.numel()
    if q == "full":
        return None, None, u
    if q == "pow2":
        lo, hi = -17, -11
        fraction, e = torch.frexp(u.abs())  # |u| = fraction 2^e, fraction in [0.5, 1)
        e = (e.long() - 1 + (fraction >= 0.75).long()).clamp(lo, hi)
        power = torch.tensor([2.0 ** k for k in range(lo, hi + 1)], dtype=torch.float64, device=u.device)
        code = torch.where(u == 0, 7, e - lo + torch.where(u < 0, 8, 0))
        return code, None, torch.where(u == 0, 0.0, torch.sign(u) * power[e - lo])
    a = u.abs()
    lengths = [d] if group == 0 else list(_segments(case)) if group < 0 else None
    if lengths is None:
        k = -(-d // group)
        b = torch.nn.functional.pad(a, (0, k * group - d)).view(k, group)
        size = torch.full((k,), group, device=u.device)
        size[-1] = d - (k - 1) * group
        s = b.sum(1) / size if q == "sign" else b.amax(1)
        su = s.repeat_interleave(group)[:d]
    else:
        parts = a.split(lengths)
        s = torch.stack([p.mean() if q == "sign" else p.max() for p in parts])
        su = torch.cat([v.expand(m) for v, m in zip(s, lengths)])
    if q == "sign":
        return (u >= 0).long(), s, torch.where(u >= 0, su, -su)
    L = 2 ** (bits - 1) - 1
    y = torch.where(su > 0, u / su.clamp(min=1e-300), 0.0) * L
    if stochastic:
        i = torch.floor(y)
        for at in range(0, d, 1 << 25):
            part = slice(at, min(d, at + (1 << 25)))
            U = _philox(int(seed), who, 0, torch.arange(part.start, part.stop, device=u.device))
            i[part] += (U < y[part] - i[part]).double()
    else:
        i = torch.round(y)
    return i.long() + L, s, su * (i / L)


def _pack(codes, bits):
    if codes is None:
        return None
    per = 32 // bits
    c = torch.nn.functional.pad(codes, (0, -codes.numel() % per)).view(-1, per)
    w = torch.zeros(c.shape[0], dtype=torch.int64, device=c.device)
    for k in range(per):
        w |= c[:, k] << (k * bits)
    return w.to(torch.int32)  # the low 32 bits


def _adam64(case, g):
    """The first round's moments and step of a gradient (or average) g."""
    def f32(v):
        return torch.tensor(v, dtype=torch.float32).double().item()

    b1, b2, alpha, eps = f32(BETA1), f32(case["beta2"]), f32(case["alpha"]), f32(EPS)
    m = (1 - b1) * g
    if case["form"] == 0:
        v = b2 * eps + (1 - b2) * g * g
        return m, v, alpha * m / v.sqrt()
    v = (1 - b2) * g * g
    return m, v, alpha * (m / (1 - b1)) / ((v / (1 - b2)).sqrt() + eps)


def exact(case, seed):
    d, n, at_worker = case["d"], case["n"], case["placement"] == 0
    codes, scales, ms, vs = [], [], [], []
    total = torch.zeros(d, dtype=torch.float64, device="cuda")
    for i in range(n):
        u = _gradient(case, seed, i).double()
        if at_worker:
            m, v, u = _adam64(case, u)
            ms.append(m)
            vs.append(v)
        c, s, dec = _quantize64(case, u, case["qw"], case["gw"], seed, i)
        codes.append(_pack(c, _KINDS[case["qw"]][0]))
        scales.append(s)
        if case["api"] == "noalloc":
            four = torch.zeros(4, dtype=torch.float64, device="cuda")
            pad = 4 * -(-d * _KINDS[case["qw"]][0] // 128) - codes[0].numel()
            return {"e": u - dec if case["ef"] else torch.zeros_like(u),
                    "codes": torch.nn.functional.pad(codes[0], (0, pad)), "scales": s,
                    "m": ms[0] if at_worker else four,
                    "v": vs[0] if at_worker else (four + EPS if case["form"] == 0 else four)}
        total += dec
        del u, dec, c
    w = total.div_(n)
    if not at_worker:
        m, v, w = _adam64(case, w)
        ms, vs = [m], [v]
    c, s, dec = _quantize64(case, w, case["qs"], case["gs"], seed, n)
    out = {"x": _x0(case, seed).double() - dec, "codes": _pack(c, _KINDS[case["qs"]][0]),
           "worker_codes": None if codes[0] is None else torch.stack(codes)}
    if s is not None:
        out["scales"] = s
    if scales[0] is not None:
        out["worker_scales"] = torch.stack(scales)
    out["m"], out["v"] = (torch.stack(ms), torch.stack(vs)) if at_worker else (ms[0], vs[0])
    return out
