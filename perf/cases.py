"""What this library's callers have it do, as cases that can be timed and checked.

A training loop calls it once per simulated-loss step: the forward (theta~ from
theta and theta0), the storage switch, and the gradient map, by itself or fused
with the AdamW update. An evaluation merges experts. The cases go through the
public binding (`SmatParameters`, `SmatSession`, `merge`) on the parameter lists
of `paper_2609_33437_gb300.workloads` and on flat and ragged lists, from some ten
thousand elements (a set of adapters) to a whole 7B model.

Every tensor of a list is a view of one flat buffer per array (each starting on a
128-byte boundary), as a trainer with flat parameter storage has them, so that a
call's whole result is a few tensors.

`exact` restates the library's definitions (Philox-4x32 draws keyed by seed, step,
tensor and element; Scale, Mask, Perturb; the gradient map; AdamW; the merging
methods) in plain torch with 64-bit integers and floats.
"""

import math

import torch

from paper_2609_33437_gb300 import smat as S
from paper_2609_33437_gb300 import workloads as W

STEP = 7          # the SMAT step of every case (a key of the random draws)
ADAM = dict(lr=1e-5, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.01, adam_step=20)
DEVICE = "cuda"


# ----------------------------------------------------------------- the cases ---
def listed():
    return [
        # Adapter matrices of odd sizes trained in fp32 with the paper's own settings (uniform Perturb, one
        # Scale for all, half of the coordinates kept): the smallest call, where launches and latency count.
        _case("step_adapters_f32", "step", "ragged", n=70001, count=24, dtype="f32", gdtype="f32", keep=0.5,
              alpha="global", noise="uniform", sigma=2e-3),
        # A vision tower with its projector in bf16, the paper's settings: an ordinary step over many small
        # tensors (biases and norms among them).
        _case("step_vision_bf16", "step", "vision", dtype="bf16", gdtype="bf16", alpha="global", noise="uniform",
              sigma=5e-5),
        # The forward of a 0.5B decoder: Gaussian Perturb of a given RMS, Scale per tensor.
        _case("forward_0p5b", "forward", "dec_0p5b", layers=24, dtype="bf16", alpha="tensor", noise="gaussian",
              sigma=1e-4),
        # The forward of a whole 7B decoder with Perturb relative to each tensor's std(theta - theta0): the
        # largest call.
        _case("forward_7b_relative", "forward", "llama_7b", layers=32, dtype="bf16", alpha="tensor",
              noise="gaussian", sigma_rel=0.1),
        # A vision-language model (8 language layers): two keep rates, a given RMS, so no statistics.
        _case("forward_vl", "forward", "vl_7b", layers=8, dtype="bf16", alpha="tensor", noise="gaussian",
              sigma=5e-5),
        # Scale drawn per element on one flat tensor of odd size (the flat-tensor sweep's setting).
        _case("forward_elem_alpha", "forward", "flat", n=100000007, dtype="bf16", keep=0.9, alpha="element",
              noise="gaussian", sigma=1e-4),
        # Gradient accumulation: a further micro-batch's fp32 gradient mapped onto the sum.
        _case("grad_accumulate_0p5b", "grad", "dec_0p5b", layers=24, dtype="bf16", gdtype="f32", alpha="tensor",
              noise="gaussian", sigma=1e-4, accumulate=True),
        # The gradient map in place, as the parameter-switching classes call it, on half of the 7B decoder.
        _case("grad_in_place_7b", "grad", "llama_7b", layers=16, dtype="bf16", gdtype="bf16", alpha="tensor",
              noise="gaussian", sigma=2e-5, accumulate=False),
        # Gradient map and AdamW in one pass on fp32 parameters, gradients and moments (a vision tower).
        _case("adamw_vision_f32", "adamw", "vision", dtype="f32", gdtype="f32", alpha="tensor", noise="gaussian",
              sigma=5e-5),
        # Evaluation: Task Arithmetic over four vision-tower experts.
        _case("merge_ta_vision", "merge", "vision", dtype="bf16", method="ta", experts=4, gamma=0.4),
        # DARE + Task Arithmetic over eight experts of the 0.5B decoder.
        _case("merge_dare_0p5b", "merge", "dec_0p5b", layers=24, dtype="bf16", method="dare", experts=8, gamma=0.3,
              p_drop=0.9),
        # TIES over eight experts of the 7B decoder's first four layers, embedding and head.
        _case("merge_ties_7b", "merge", "llama_7b", layers=4, dtype="bf16", method="ties", experts=8, gamma=0.3,
              retention=0.5),
    ]


# Every key that a case can have, with the value that stands for "not said".
_DEFAULTS = dict(layers=0, n=0, count=0, dtype="bf16", gdtype="f32", keep=-1.0, alpha="tensor", noise="gaussian",
                 sigma=0.0, sigma_rel=0.0, alpha_min=0.3, draw_bits=32, rounds=10, inplace=False, shard=0,
                 accumulate=False, method="", experts=0, gamma=1.0, p_drop=0.0, retention=1.0)


def _case(name, kind, params, **more):
    c = dict(_DEFAULTS, kind=kind, list=params, **more)
    if name:
        c["name"] = name
    return c


def _log(rng, lo, hi):
    """A size spread over the logarithm of [lo, hi], odd as often as not."""
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    """One more case: any path, over list shapes, sizes, types and options that a trainer or an evaluation sets."""
    kind = rng.choice(["step", "step", "forward", "forward", "grad", "adamw", "merge", "merge"])
    more = {"dtype": rng.choice(["bf16", "bf16", "f32"])}
    params = rng.choice(["flat", "ragged", "ragged", "dec_0p5b", "llama_7b", "vision"])
    top = 1 << 28 if kind != "merge" else 1 << 27
    if params == "flat":
        more["n"] = _log(rng, 1 << 16, top)
    elif params == "ragged":
        more["n"], more["count"] = _log(rng, 1 << 14, top), rng.randint(3, 24)
    elif params == "dec_0p5b":
        more["layers"] = rng.randint(1, 24)
    elif params == "llama_7b":
        more["layers"] = rng.randint(1, 2)
    if kind == "merge":
        more["method"] = rng.choice(["wa", "ta", "dare", "ties", "ties"])
        more["experts"] = rng.randint(2, 8) if params in ("dec_0p5b", "llama_7b", "vision") else rng.randint(2, 16)
        more["gamma"] = round(rng.uniform(0.2, 1.0), 2)
        if more["method"] == "dare":
            more["p_drop"] = rng.choice([0.5, 0.8, 0.9])
            more["rounds"] = rng.choice([10, 10, 7])
        if more["method"] == "ties":
            more["retention"] = rng.choice([0.1, 0.2, 0.3, 0.5, 0.7])
        return _case("", kind, params, **more)
    more["gdtype"] = rng.choice(["f32", "bf16"])
    more["keep"] = rng.choice([0.3, 0.5, 0.7, 0.9, round(rng.uniform(0.1, 0.99), 3)])
    more["alpha"] = rng.choice(["global", "tensor", "tensor", "element"])
    more["alpha_min"] = rng.choice([0.0, 0.2, 0.3])
    more["noise"] = rng.choice(["uniform", "uniform", "gaussian", "gaussian", "laplace"])
    more["draw_bits"] = rng.choice([32, 32, 32, 16])
    more["rounds"] = rng.choice([10, 10, 7]) if more["noise"] != "laplace" else 10
    if rng.random() < 0.35 and kind in ("step", "forward"):
        more["sigma_rel"] = rng.choice([0.05, 0.1, 0.3])
    else:
        more["sigma"] = rng.choice([5e-5, 1e-4, 2e-3])
    if rng.random() < 0.2:
        more["shard"] = 16 * rng.randint(1, 1 << 30)
    if kind == "forward" and params in ("flat", "ragged") and more["n"] <= 1 << 24 and rng.random() < 0.5:
        more["inplace"] = True
    if kind == "grad":
        more["accumulate"] = rng.random() < 0.5
    return _case("", kind, params, **more)


def _shapes(c):
    """[(elements, keep probability)] of the case's parameter list."""
    if c["list"] == "flat":
        got = [(c["n"], "linear", 0.5)]
    elif c["list"] == "ragged":
        # odd sizes whose ratios run over about a factor of sixteen
        w = [2.0 ** (4 * ((k * 7) % c["count"]) / c["count"]) for k in range(c["count"])]
        got = [(max(1, int(c["n"] * x / sum(w))) | 1, "linear" if k % 4 else "other", 0.5) for k, x in enumerate(w)]
    else:
        name = "vl_7b" if c["list"] == "vision" else c["list"]
        got = []
        for t in W.WORKLOADS[name]().tensors:
            parts = t.name.split("layers.")
            vision = t.name.startswith(("vit.", "proj."))
            if c["list"] == "vision" and not vision:
                continue
            if not vision and len(parts) > 1 and int(parts[1].split(".")[0]) >= c["layers"]:
                continue
            got.append((t.numel, t.kind, t.keep_prob))
    return [(n, (c["keep"] if c["keep"] >= 0 else keep) if kind == "linear" else 1.0) for n, kind, keep in got]


_DT = {"f32": torch.float32, "bf16": torch.bfloat16}
_ALPHA = {"global": S.SMAT_ALPHA_GLOBAL, "tensor": S.SMAT_ALPHA_PER_TENSOR, "element": S.SMAT_ALPHA_PER_ELEMENT}
_NOISE = {"uniform": S.SMAT_NOISE_UNIFORM, "gaussian": S.SMAT_NOISE_GAUSSIAN, "laplace": S.SMAT_NOISE_LAPLACE}
_METHOD = {"wa": S.SMAT_MERGE_WA, "ta": S.SMAT_MERGE_TA, "dare": S.SMAT_MERGE_DARE_TA, "ties": S.SMAT_MERGE_TIES}


# ------------------------------------------------------------------- inputs ---
def _places(c):
    """[(first, numel)] of each tensor in a flat buffer, and the buffer's length."""
    at, got = 0, []
    for n, _ in _shapes(c):
        got.append((at, n))
        at += (n + 63) // 64 * 64
    return got, at


def _views(flat, places):
    return [flat[a:a + n] for a, n in places]


def _normal(gen, n, std, dtype, plus=None):
    """A flat buffer of N(0, std^2) (plus another buffer), drawn in fp32 a part at a time."""
    out = torch.empty(n, dtype=dtype, device=DEVICE)
    part = 1 << 27
    for a in range(0, n, part):
        x = torch.randn(min(part, n - a), generator=gen, device=DEVICE)
        x.mul_(std)
        if plus is not None:
            x += plus[a:a + part]
        out[a:a + part] = x
    return out


def _inputs(c, seed):
    """The arrays that the call reads, from the seed alone."""
    places, total = _places(c)
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(int(seed) * 1000003 + 17)
    dt, x = _DT[c["dtype"]], {"places": places, "total": total}
    x["theta0"] = _normal(gen, total, 0.02, dt)
    if c["kind"] == "merge":
        x["experts"] = [_normal(gen, total, 3e-4, dt, x["theta0"]) for _ in range(c["experts"])]
        return x
    x["theta"] = _normal(gen, total, 3e-4, dt, x["theta0"])
    if c["kind"] in ("step", "grad", "adamw"):
        x["g"] = _normal(gen, total, 1.0, _DT[c["gdtype"]])
    if c["kind"] == "grad" and c["accumulate"]:
        x["acc"] = _normal(gen, total, 1.0, _DT[c["gdtype"]])
    if c["kind"] == "adamw":
        x["m1"] = _normal(gen, total, 0.1, torch.float32)
        x["m2"] = _normal(gen, total, 0.1, torch.float32).square_().add_(1e-3)
    return x


def _rng_seed(seed):
    return 1000 + int(seed)


def _f32(v):
    """A setting as the library receives it: 32-bit."""
    return torch.tensor(float(v), dtype=torch.float32).item()


def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    places, total = x["places"], x["total"]
    s = dict(case=c, **x)
    if c["kind"] == "merge":
        s["out"] = torch.zeros(total, dtype=_DT[c["dtype"]], device=DEVICE)
        t0, out = _views(x["theta0"], places), _views(s["out"], places)
        ex = [_views(e, places) for e in x["experts"]]
        s["call"] = dict(theta0s=t0, experts=[[e[k] for e in ex] for k in range(len(places))], outs=out,
                         method=_METHOD[c["method"]], gamma=c["gamma"], p_drop=c["p_drop"],
                         retention=c["retention"], seed=_rng_seed(seed), philox_rounds=c["rounds"])
        return s
    keeps = [k for _, k in _shapes(c)]
    n = len(keeps)
    options = dict(sigma_rels=[c["sigma_rel"]] * n, seed=_rng_seed(seed), alpha_min=c["alpha_min"], alpha_max=1.0,
                   alpha_mode=_ALPHA[c["alpha"]], noise=_NOISE[c["noise"]], philox_rounds=c["rounds"],
                   draw_bits=c["draw_bits"], elem_offsets=[c["shard"]] * n)
    theta, theta0 = _views(x["theta"], places), _views(x["theta0"], places)
    if c["kind"] == "step" and n <= 24 and c["dtype"] == c["gdtype"]:
        # the parameter-switching class, as a training loop holds it (its theta~ buffers are its own)
        params = [torch.nn.Parameter(t) for t in theta]
        for p, g in zip(params, _views(x["g"], places)):
            p.grad = g
        s["params"] = S.SmatParameters(params, theta0, keeps, [c["sigma"]] * n, **options)
        return s
    if c["inplace"]:
        # the paper's memory mode: theta~ takes theta0's buffer, theta0 comes back from pinned host memory
        host = torch.empty(total, dtype=_DT[c["dtype"]], pin_memory=True)
        host.copy_(x["theta0"])
        s["host"], s["sim"] = _views(host, places), x["theta0"]
    else:
        s["sim"] = torch.zeros(total, dtype=_DT[c["dtype"]], device=DEVICE)
    s["session"] = S.SmatSession(theta, theta0, _views(s["sim"], places), keeps, [c["sigma"]] * n, **options)
    if c["kind"] in ("step", "grad", "adamw"):
        s["gs"] = _views(x["g"], places)
    if c["kind"] == "grad":
        s["out"] = x["acc"] if c["accumulate"] else x["g"]
        s["gouts"] = _views(s["out"], places)
    if c["kind"] == "adamw":
        s["m1s"], s["m2s"] = _views(x["m1"], places), _views(x["m2"], places)
    if c["kind"] in ("grad", "adamw"):
        s["session"].simulate_multi(STEP)  # the forward whose mask the call maps through
    return s


# ---------------------------------------------------------------------- run ---
def run(s):
    c = s["case"]
    if c["kind"] == "merge":
        S.merge(**s["call"])
        return s["out"]
    if "params" in s:
        p = s["params"]
        p.simulate(STEP)
        p.swap()
        p.grad_map(STEP)
        p.swap()
        return {"sim": p.sims, "grad": s["g"]}
    sess = s["session"]
    if c["kind"] == "step":
        sess.simulate_multi(STEP)
        sess.swap()
        sess.grad_map_multi(STEP, s["gs"])
        sess.swap()
        return {"sim": s["sim"], "grad": s["g"]}
    if c["kind"] == "forward":
        if c["inplace"]:
            sess.refill_theta0(s["host"])
        sess.simulate_multi(STEP)
        return s["sim"]
    if c["kind"] == "grad":
        sess.grad_map_multi(STEP, s["gs"], s["gouts"], accumulate=c["accumulate"])
        return s["out"]
    sess.grad_map_adamw_multi(STEP, s["gs"], s["m1s"], s["m2s"], **ADAM)
    return {"theta": s["theta"], "m1": s["m1"], "m2": s["m2"]}


def work(case):
    """Bytes: each input read once, each output written once. Operations: the arithmetic of the definitions
    (differences, products, sums, the noise law), the integer work of the draws not counted."""
    n = sum(k for k, _ in _shapes(case))
    b = 2 if case["dtype"] == "bf16" else 4
    gb = 2 if case["gdtype"] == "bf16" else 4
    kind = case["kind"]
    if kind == "merge":
        k = case["experts"]
        return {"bytes": (k + 2) * b * n, "flops": (3 if case["method"] != "ties" else 5) * k * n}
    forward = {"bytes": 3 * b * n, "flops": 6 * n}
    if kind == "forward":
        return forward
    grad = {"bytes": 2 * gb * n + (gb * n if case["accumulate"] else 0), "flops": 2 * n}
    if kind == "step":
        return {m: forward[m] + grad[m] for m in forward}
    if kind == "grad":
        return grad
    return {"bytes": (gb + 2 * b + 16) * n, "flops": 14 * n}


def tolerance(case):
    """About four times the distance from `exact` that a correct run at the case's types shows: half an ulp of
    the stored type on each value (bf16: up to 2^-9, 1.7e-3 in the 2-norm; fp32: up to 2^-24), and for fp32 the
    few roundings before it, which count where theta0 + delta + eps cancels."""
    stored = [case["dtype"]]
    if case["kind"] == "step":
        stored.append(case["gdtype"])
    if case["kind"] == "grad":
        stored = [case["gdtype"]]
    if "bf16" in stored or (case["kind"] == "adamw" and case["gdtype"] == "bf16"):
        return {"rel": 7e-3, "max": 1.6e-2}
    return {"rel": 5e-7, "max": 1e-5}


# -------------------------------------------------- the definitions, 64 bits ---
_MASK, _PERTURB, _SCALE_E, _SCALE_T, _MASK_LO = range(5)
_M32 = 0xFFFFFFFF
_PART = 1 << 24  # elements per part


def _philox(j, stream, tid, step, seed, rounds):
    """Blocks j (int64 tensor) of a stream as [len(j), 4] words: Philox-4x32, counter (j, stream | tensor, step)."""
    c = [j & _M32, j >> 32, torch.full_like(j, (stream << 28) | tid), torch.full_like(j, step)]
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(rounds):
        a, b = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((b >> 32) & _M32) ^ c[1] ^ k0, b & _M32, ((a >> 32) & _M32) ^ c[3] ^ k1, a & _M32]
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return torch.stack(c, 1)


class _Draws:
    """The draws of elements [lo, hi) of one tensor (lo a multiple of 16; the shard offset too)."""

    def __init__(self, tid, lo, hi, shard, step, seed, rounds, bits):
        self.tid, self.n, self.step, self.seed, self.rounds, self.bits = tid, hi - lo, step, seed, rounds, bits
        self.g0, self.groups = shard + lo, (hi - lo + 15) // 16

    def _blocks(self, stream, per_group):
        first = self.g0 // 16 * per_group
        j = torch.arange(first, first + self.groups * per_group, dtype=torch.int64, device=DEVICE)
        return _philox(j, stream, self.tid, self.step, self.seed, self.rounds)

    def _halves(self, stream):
        w = self._blocks(stream, 2)
        return torch.stack([w & 0xFFFF, w >> 16], 2).reshape(-1)[:self.n]

    def kept(self, keep):
        t = math.floor(_f32(keep) * 2.0 ** self.bits)
        if t >= 1 << self.bits:
            return torch.ones(self.n, dtype=torch.bool, device=DEVICE)
        if self.bits == 16:
            return self._halves(_MASK) < t
        w = self._blocks(_MASK, 1)
        high = torch.stack([(w >> s) & 255 for s in (0, 8, 16, 24)], 2).reshape(-1)[:self.n]
        low = (self._blocks(_MASK_LO, 4) >> 8).reshape(-1)[:self.n]
        return ((high << 24) | low) < t

    def unit(self, stream):
        """The stream's field of each element, as the midpoint of its cell in (0, 1) and the cell's left end."""
        if self.bits == 16:
            u, one = self._halves(stream), 1 << 16
        else:
            w = self._blocks(stream, 3).reshape(-1, 3)  # three words serve four elements
            last = (w[:, 0] & 255) | ((w[:, 1] & 255) << 8) | ((w[:, 2] & 255) << 16)
            u, one = torch.cat([w >> 8, last[:, None]], 1).reshape(-1)[:self.n], 1 << 24
        u = u.to(torch.float64)
        return (u + 0.5) / one, u / one


def _scale(c, tid, seed):
    """alpha of a tensor (global: one for all)."""
    t = 0x0FFFFFFF if c["alpha"] == "global" else tid
    u = int(_philox(torch.zeros(1, dtype=torch.int64), _SCALE_T, t, STEP, seed, c["rounds"])[0, 0]) >> 8
    return _f32(c["alpha_min"]) + (1.0 - _f32(c["alpha_min"])) * u * 2.0 ** -24


def _noise(law, mid):
    v = 2 * mid - 1
    if law == "uniform":
        return math.sqrt(3.0) * v
    if law == "gaussian":
        return math.sqrt(2.0) * torch.erfinv(v)
    return -torch.sign(v) * torch.log1p(-v.abs()) / math.sqrt(2.0)


def _parts(places):
    for k, (a, n) in enumerate(places):
        for lo in range(0, n, _PART):
            yield k, a, lo, min(n, lo + _PART)


def _exact_merge(c, x, seed):
    out = torch.zeros(x["total"], dtype=torch.float64, device=DEVICE)
    K, method = c["experts"], c["method"]
    keep, gamma = _f32(1.0 - _f32(c["p_drop"])), _f32(c["gamma"])
    thr = {}
    if method == "ties":  # the r-th largest magnitude of each tensor's fp32 differences
        for k, (a, n) in enumerate(x["places"]):
            r = min(n, max(1, math.ceil(_f32(c["retention"]) * n)))
            for e, y in enumerate(x["experts"]):
                d = (y[a:a + n].float() - x["theta0"][a:a + n].float()).abs_()
                thr[k, e] = torch.sort(d).values[n - r].item()
    for k, a, lo, hi in _parts(x["places"]):
        at = slice(a + lo, a + hi)
        t0 = x["theta0"][at].double()
        acc = torch.zeros_like(t0)
        if method == "ties":
            d = torch.stack([y[at].double() - t0 for y in x["experts"]])
            mag = torch.stack([(y[at].float() - x["theta0"][at].float()).abs() for y in x["experts"]])
            held = mag >= torch.tensor([thr[k, e] for e in range(K)], device=DEVICE)[:, None]
            sign = torch.sign((d * held).sum(0))
            held &= torch.sign(d) == sign
            held &= sign != 0
            acc = gamma * (d * held).sum(0) / held.sum(0).clamp(min=1)
        else:
            for e, y in enumerate(x["experts"]):
                d = y[at].double() - t0
                if method == "dare":
                    d = d * _Draws(k, lo, hi, 0, e, _rng_seed(seed), c["rounds"], 32).kept(keep) / keep
                acc += d * (1.0 / K if method == "wa" else gamma)
        out[at] = t0 + acc
    return out


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    if c["kind"] == "merge":
        return _exact_merge(c, x, seed)
    places, total, key = x["places"], x["total"], _rng_seed(seed)
    keeps = [k for _, k in _shapes(c)]
    alphas = [_scale(c, k, key) for k in range(len(places))]
    kind, f64 = c["kind"], torch.float64
    sim = torch.zeros(total, dtype=f64, device=DEVICE) if kind in ("step", "forward") else None
    # padding between tensors keeps what the inputs hold there
    new = {m: x[m].double() for m in ("g", "acc", "theta", "m1", "m2")
           if m in x and (kind in ("step", "grad") and m in ("g", "acc") or kind == "adamw" and m != "g")}
    if kind == "forward" and c["inplace"]:
        sim.copy_(x["theta0"])
    sigma = [_f32(c["sigma"])] * len(places)
    if c["sigma_rel"] > 0 and sim is not None:
        for k, (a, n) in enumerate(places):
            s1 = s2 = 0.0
            for lo in range(0, n, _PART):
                at = slice(a + lo, a + min(n, lo + _PART))
                d = (x["theta"][at].float() - x["theta0"][at].float()).double()
                s1, s2 = s1 + d.sum().item(), s2 + d.square().sum().item()
            sigma[k] = _f32(c["sigma_rel"]) * math.sqrt(max(0.0, s2 / n - (s1 / n) ** 2))
    for k, a, lo, hi in _parts(places):
        at = slice(a + lo, a + hi)
        r = _Draws(k, lo, hi, c["shard"], STEP, key, c["rounds"], c["draw_bits"])
        alpha = alphas[k]
        if c["alpha"] == "element":
            alpha = _f32(c["alpha_min"]) + (1.0 - _f32(c["alpha_min"])) * r.unit(_SCALE_E)[1]
        m = r.kept(keeps[k]) * (alpha / _f32(keeps[k]))
        if sim is not None:
            t0 = x["theta0"][at].double()
            v = t0 + m * (x["theta"][at].double() - t0)
            if sigma[k] > 0:
                v += sigma[k] * _noise(c["noise"], r.unit(_PERTURB)[0])
            sim[at] = v
        if kind in ("step", "grad", "adamw"):
            g = m * x["g"][at].double()
        if kind == "step" or kind == "grad" and not c["accumulate"]:
            new["g"][at] = g
        elif kind == "grad":
            new["acc"][at] += g
        elif kind == "adamw":
            g = g.to(_DT[c["gdtype"]]).double()
            b1, b2, lr, decay, eps = (_f32(ADAM[m]) for m in ("beta1", "beta2", "lr", "weight_decay", "eps"))
            t = ADAM["adam_step"]
            m1 = b1 * new["m1"][at] + (1 - b1) * g
            m2 = b2 * new["m2"][at] + (1 - b2) * g * g
            new["theta"][at] *= 1 - lr * decay
            new["theta"][at] -= lr / (1 - b1 ** t) * m1 / (m2.sqrt() / math.sqrt(1 - b2 ** t) + eps)
            new["m1"][at], new["m2"][at] = m1, m2
    if kind == "forward":
        return sim
    if kind == "step":
        if len(places) <= 24 and c["dtype"] == c["gdtype"]:
            return {"sim": _views(sim, places), "grad": new["g"]}
        return {"sim": sim, "grad": new["g"]}
    if kind == "grad":
        return new["acc"] if c["accumulate"] else new["g"]
    return new
