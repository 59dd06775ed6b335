"""The sharded weight update as a training program calls it: the cases that its speed is measured on.

A case names a model's tensor list (a family and its sizes), the optimizer, the number of replicas and of
gradient copies, the data types, the shard layout and the route a program takes through the public entry
points:

  fused     ws_fused_update over all shards: gradients read from the replicas' tensors, weights written to
            the weight tensors (fp32 weight tensors are the master copy, bf16 ones a copy of the fp32 state)
  separate  ws_pack_sets of all gradient lists, ws_shard_update of all shards, ws_unpack of the weights
  replica   what one replica does around its two collectives: ws_pack of its own gradients, ws_shard_update
            of its shard from the reduce-scatter's receive buffer, ws_unpack of the gathered weights
  slices    ws_shard_update of one shard from the slices of all replicas

Everything is resident in device memory, the weights and slots keep advancing from pass to pass, and the
step number that the bias corrections use advances with them.
"""
from __future__ import annotations

import math

import torch

from paper_2004_13336_b200 import binding as ws
from paper_2004_13336_b200 import workloads as W

_DTYPE = {"f32": torch.float32, "bf16": torch.bfloat16}
_HYPER = {
    "sgdm": dict(lr=0.1, momentum=0.9, weight_decay=5e-5),
    "adam": dict(),
    "lamb": dict(eps=1e-6, weight_decay=0.01),
    "lars": dict(lr=10.0, momentum=0.9, weight_decay=5e-5, trust_coeff=0.001),
    "adafactor": dict(lr=1e-2, eps=1e-30, eps2=1e-3, clip_threshold=1.0, decay_exponent=0.8),
}
_SLOTS = {"sgdm": 1, "adam": 2, "lamb": 2, "lars": 1, "adafactor": 0}


def _case(name, family, opt, copies, **kw):
    c = dict(name=name, family=family, opt=opt, copies=copies, width=0, layers=0, vocab=0, grad="f32", out="f32",
             route="fused", layout="per_tensor", align=32, outliers=False)
    c.update(kw)
    return c


def listed():
    return [
        # a few tensors, 45 792 parameters: nothing but latency and launches
        _case("tiny adam 4", "tiny", "adam", 4, width=128),
        # a small model whose norms need two phases: launches again, 1.7 M parameters
        _case("small lamb 8", "encdec", "lamb", 8, width=128, layers=2, vocab=6000),
        # the image network under its two optimizers: many small tensors, 25.6 M parameters
        _case("image sgdm 8", "conv", "sgdm", 8, width=64, vocab=1000),
        _case("image lars 8", "conv", "lars", 8, width=64, vocab=1000),
        # one of eight replicas around its collectives, bf16 gradients on the wire and bf16 weights gathered
        _case("image replica sgdm 8", "conv", "sgdm", 8, width=64, vocab=1000, route="replica", grad="bf16", out="bf16"),
        # the translation network, 211 M parameters: the ordinary step
        _case("translation adam 8", "encdec", "adam", 8, width=1024, layers=6, vocab=33708),
        # ... under the factored optimizer, with few copies
        _case("translation adafactor 4", "encdec", "adafactor", 4, width=1024, layers=6, vocab=33708),
        # ... under LAMB through the separate kernels, weights emitted in bf16
        _case("translation lamb separate 4", "encdec", "lamb", 4, width=1024, layers=6, vocab=33708, route="separate", out="bf16"),
        # ... sharded 128 ways: one replica pulls its slice of 128 gradient buffers
        _case("translation adam slices 128", "encdec", "adam", 128, width=1024, layers=6, vocab=33708, route="slices"),
        # sizes that divide nothing (odd rows, vectors, scalars, empty tensors), the concatenated layout
        _case("ragged adafactor 2", "ragged", "adafactor", 2, width=611, layers=7, vocab=9973, layout="concat"),
        # the large encoder under its optimizer, 335 M parameters, 16 copies
        _case("encoder lamb 16", "encoder", "lamb", 16, width=1024, layers=24, vocab=30522),
        # the largest: 1.56 G parameters, bf16 gradients with outliers, fp32 state, bf16 weights
        _case("decoder adam 4", "decoder", "adam", 4, width=1600, layers=48, vocab=50257, grad="bf16", out="bf16", outliers=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        route = rng.choice(["fused", "fused", "fused", "separate", "replica", "slices"])
        one_kernel = route in ("replica", "slices")          # a single shard: the elementwise optimizers
        opt = rng.choice(["sgdm", "adam"] if one_kernel else ["sgdm", "adam", "lamb", "lars", "adafactor"])
        family = rng.choice(["tiny", "conv", "encdec", "encoder", "decoder", "ragged"])
        width, layers, vocab = {
            "tiny": lambda: (_log_int(rng, 32, 1024), 0, 0),
            "conv": lambda: (_log_int(rng, 12, 96), 0, _log_int(rng, 10, 2000)),
            "encdec": lambda: (16 * _log_int(rng, 4, 64), rng.randint(1, 6), _log_int(rng, 1000, 34000)),
            "encoder": lambda: (16 * _log_int(rng, 4, 64), rng.randint(2, 24), _log_int(rng, 1000, 31000)),
            "decoder": lambda: (16 * _log_int(rng, 4, 100), rng.randint(2, 24), _log_int(rng, 1000, 51000)),
            "ragged": lambda: (_log_int(rng, 17, 1200), rng.randint(1, 8), _log_int(rng, 100, 20000)),
        }[family]()
        copies = rng.choice({"fused": [1, 2, 3, 4, 6, 8, 12, 16, 32], "separate": [1, 2, 3, 4, 8],
                             "replica": [2, 3, 8, 16, 64], "slices": [2, 8, 16, 64, 128, 512, 1024]}[route])
        c = _case("", family, opt, copies, width=width, layers=layers, vocab=vocab, route=route,
                  grad=rng.choice(["f32", "bf16"]), out=rng.choice(["f32", "bf16"]),
                  layout=rng.choice(["per_tensor", "per_tensor", "concat"]), align=rng.choice([32, 32, 8]))
        del c["name"]
        n = sum(_numels(c))
        if n <= 500e6 and 2 * copies * n <= 8e9 * (copies if one_kernel else 1) and work(c)["bytes"] <= 25e9:
            return c


# ------------------------------------------------------------------ tensor lists
def _conv(width, classes):
    """Bottleneck image network; width 64 and 1000 classes is the 25.6 M parameter one."""
    s = [(7, 7, 3, width), (width,), (width,)]
    cin = width
    for w, blocks in ((width, 3), (2 * width, 4), (4 * width, 6), (8 * width, 3)):
        for b in range(blocks):
            s += [(1, 1, cin, w), (w,), (w,), (3, 3, w, w), (w,), (w,), (1, 1, w, 4 * w), (4 * w,), (4 * w,)]
            if b == 0:
                s += [(1, 1, cin, 4 * w), (4 * w,), (4 * w,)]
            cin = 4 * w
    return s + [(cin, classes), (classes,)]


def _ragged(width, layers, vocab):
    s = [(vocab, width), (), (0, width)]
    for k in range(layers):
        s += [(width, 3 * width + k), (3 * width + k,), (width + 1, width), (width,), (3, 5, k + 1, width // 4 + 1), (k + 1,)]
    return s + [(width, vocab + 2), (vocab + 2,)]


def _shapes(c):
    d = c["width"]
    return {
        "tiny": lambda: [(64, d), (d,), (3, 3, 16, max(1, d // 4)), (max(1, d // 4),), (4 * d, 64), (64,)],
        "conv": lambda: _conv(d, c["vocab"]),
        "encdec": lambda: W.transformer_shapes(d, 4 * d, c["vocab"], c["layers"]),
        "encoder": lambda: W.bert_large_shapes(d, 4 * d, c["vocab"], 512, c["layers"]),
        "decoder": lambda: W.decoder_1p5b_shapes(d, 4 * d, c["vocab"], 1024, c["layers"]),
        "ragged": lambda: _ragged(d, c["layers"], c["vocab"]),
    }[c["family"]]()


def _numels(c):
    return [math.prod(s) for s in _shapes(c)]


def _offsets(numels):
    """Starts of the tensors in a flat arena (each rounded up to 8 elements) and its length."""
    offs, at = [], 0
    for n in numels:
        offs.append(at)
        at += (n + 7) // 8 * 8
    return offs, at


def _hyper(c):
    return dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8, weight_decay=0.0, momentum=0.0, grad_scale=1.0, step=10) | _HYPER[c["opt"]]


# ------------------------------------------------------------------------ inputs
def _normal(n, std, gen, dtype=torch.float32, outliers=False):
    t = torch.empty(n, device="cuda").normal_(0.0, std, generator=gen)
    if outliers:            # 1 % of the entries are a hundred times larger
        t[torch.empty(n, device="cuda").uniform_(generator=gen) < 0.01] *= 100.0
    return t.to(dtype)


def _gen(seed, k):
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1_000_003 + k * 10_007 + 17) & 0x7FFFFFFF)
    return g


def _state(c, seed, length):
    """Weights and slots of the whole model, in an arena."""
    w = _normal(length, 0.02, _gen(seed, 1))
    m = _normal(length, 1e-3, _gen(seed, 2)) if _SLOTS[c["opt"]] else None
    v = _normal(length, 1e-5, _gen(seed, 3)).abs_() if _SLOTS[c["opt"]] == 2 else None
    return w, m, v


def _factored(n, seed):
    return torch.empty(n, device="cuda").uniform_(1e-6, 1e-3, generator=_gen(seed, 4))


def _grads(c, seed, n, k):
    return _normal(n, 1e-3, _gen(seed, 10 + k), _DTYPE[c["grad"]], c["outliers"])


def prepare(case, seed):
    c, s = case, {"case": case}
    numels = _numels(c)
    offs, length = _offsets(numels)
    views = lambda t: [t[o:o + n] for o, n in zip(offs, numels)]  # noqa: E731
    plan = s["plan"] = ws.Plan(_shapes(c), c["copies"], c["align"], layout=c["layout"])
    r = s["r"] = c["copies"] // 2
    s["hyper"] = _hyper(c)
    out = _DTYPE[c["out"]]
    w, m, v = _state(c, seed, length)
    s["weights"] = w.to(out, copy=True)

    def packed(t):
        if t is None:
            return None
        flat = torch.empty(plan.G, device="cuda")
        ws.ws_pack(plan, views(t), flat)
        return flat

    s["w"], s["m"], s["v"] = packed(w), packed(m), packed(v)
    if c["opt"] == "adafactor":
        s["v"] = _factored(plan.factored_elems, seed)
    if c["opt"] in ("lamb", "lars", "adafactor"):
        s["workspace"] = torch.zeros(plan.workspace_bytes(c["opt"]), dtype=torch.uint8, device="cuda")
    else:
        s["workspace"] = None
    if c["route"] == "fused":
        if c["out"] == "f32":
            s["w"] = None
        s["grads"] = ws.TensorTable(plan, [views(_grads(c, seed, length, k)) for k in range(c["copies"])])
        s["table"] = ws.TensorTable(plan, [views(s["weights"])])
        return s
    s["weight_list"] = ws.PtrList(views(s["weights"]))
    s["gathered"] = s["w"].to(out, copy=True)
    if c["route"] == "separate":
        s["grads"] = ws.TensorTable(plan, [views(_grads(c, seed, length, k)) for k in range(c["copies"])])
        s["packed"] = torch.empty(c["copies"], plan.G, dtype=_DTYPE[c["grad"]], device="cuda")
        s["packed_list"] = ws.PtrList(list(s["packed"]))
        if c["out"] == "f32":
            s["gathered"] = None
        return s
    lo, hi = r * plan.S, (r + 1) * plan.S            # the replica holds one shard of the state
    s["w"], s["m"], s["v"] = (None if t is None else t[lo:hi].clone() for t in (s["w"], s["m"], s["v"]))
    if c["route"] == "replica":
        s["grads"] = ws.PtrList(views(_grads(c, seed, length, 0)))
        s["packed"] = torch.empty(plan.G, dtype=_DTYPE[c["grad"]], device="cuda")
        s["received"] = [_grads(c, seed, plan.S, 1)]
    else:
        s["slices"] = ws.PtrList([_grads(c, seed, plan.S, k) for k in range(c["copies"])])
    return s


# -------------------------------------------------------------------------- a pass
def run(s):
    c, plan, r = s["case"], s["plan"], s["r"]
    hyper = ws.make_hyper(c["opt"], s["hyper"])
    s["hyper"]["step"] += 1
    w, m, v = s["w"], s["m"], s["v"]
    if c["route"] == "fused":
        ws.ws_fused_update(plan, -1, s["grads"], w, m, v, hyper, s["table"], s["workspace"])
        return {"weights": s["weights"], "w": w, "m": m, "v": v}
    if c["route"] == "separate":
        ws.ws_pack_sets(plan, s["grads"], s["packed_list"])
        ws.ws_shard_update(plan, -1, s["packed_list"], w, m, v, hyper, s["gathered"], s["workspace"])
        ws.ws_unpack(plan, w if s["gathered"] is None else s["gathered"], s["weight_list"])
        return {"packed": s["packed"], "gathered": s["gathered"], "weights": s["weights"], "w": w, "m": m, "v": v}
    if c["route"] == "replica":
        ws.ws_pack(plan, s["grads"], s["packed"])
        ws.ws_shard_update(plan, r, s["received"], w, m, v, hyper, s["gathered"], None, slice_mode=1)
        ws.ws_unpack(plan, s["gathered"], s["weight_list"])
        return {"packed": s["packed"], "gathered": s["gathered"], "weights": s["weights"], "w": w, "m": m, "v": v}
    ws.ws_shard_update(plan, r, s["slices"], w, m, v, hyper, s["gathered"], None, slice_mode=1)
    return {"gathered": s["gathered"], "w": w, "m": m, "v": v}


def work(case):
    """Bytes: what every call of the route has to read and write, once."""
    c = case
    n, k = sum(_numels(c)), c["copies"]
    g, o = (4 if c["grad"] == "f32" else 2), (4 if c["out"] == "f32" else 2)
    state = 8 * (1 + _SLOTS[c["opt"]])
    extra = 8 * sum(_factored_sizes(c)) if c["opt"] == "adafactor" else 0
    emitted = 2 if c["out"] == "bf16" else 0           # next to the fp32 state
    flops = n * (k + 12)
    if c["route"] == "fused":
        nbytes = n * (g * k + state + emitted)
    elif c["route"] == "separate":
        nbytes = n * (2 * g * k + g * k + state + emitted + 2 * o)
    elif c["route"] == "replica":
        nbytes, flops = n * (2 * g + 2 * o) + n / k * (g + state + o), n / k * 12
    else:
        nbytes, flops = n / k * (g * k + state + o), n / k * (k + 12)
    return {"bytes": nbytes + extra, "flops": flops}


def tolerance(case):
    """Four times what the outputs are off the same update in 64 bits: 3e-8 to 6e-8 where every output is one
    rounding of a short fp32 expression, 6.5e-7 for the factored moments (fp32 sums over rows and columns,
    added in no fixed order), 1.7e-3 for weights rounded to bf16.  Norms may be summed in another order.  A
    single element under Adam or LAMB is off by more where its gradient copies cancel and its second moment
    is almost zero: the step divides by its root."""
    if case["out"] == "bf16":
        return {"rel": 7e-3}
    rel = {"sgdm": 2.5e-7, "adam": 2.5e-7, "lamb": 5e-7, "lars": 5e-7, "adafactor": 3e-6}[case["opt"]]
    return {"rel": rel, "max": 1e-4}


# ------------------------------------------------------------------ in 64 bits
def _factored_sizes(c):
    return [n if len(s) < 2 or n == 0 else n // s[-1] + s[-1] for s, n in zip(_shapes(c), _numels(c))]


def _layout(c, numels):
    """(start of every tensor in a shard or in the concatenation, piece sizes, shard length)."""
    R, A = c["copies"], c["align"]
    up = lambda x: (x + A - 1) // A * A  # noqa: E731
    offs, at = [], 0
    if c["layout"] == "concat":
        for n in numels:
            offs.append(at)
            at = up(at + n)
        return offs, None, up(-(-at // R))
    pieces = [up(-(-n // R)) for n in numels]
    for p in pieces:
        offs.append(at)
        at += p
    return offs, pieces, at


class _Packed:
    """A shard-major [R][S] buffer in 64 bits."""

    def __init__(self, c, numels):
        self.R = c["copies"]
        self.offs, self.pieces, self.S = _layout(c, numels)
        self.flat = torch.zeros(self.R * self.S, dtype=torch.float64, device="cuda")

    def put(self, t, x):
        if self.pieces is None:
            self.flat[self.offs[t]:self.offs[t] + x.numel()] = x
        elif x.numel():
            p = self.pieces[t]
            full = torch.zeros(self.R * p, dtype=torch.float64, device="cuda")
            full[:x.numel()] = x
            self.flat.view(self.R, self.S)[:, self.offs[t]:self.offs[t] + p] = full.view(self.R, p)

    def shard(self, r):
        return self.flat[r * self.S:(r + 1) * self.S]


def _step64(h, opt, shape, g, w, m, v):
    """One update of one tensor: (w', m', v'); v is the factored state under Adafactor."""
    g = g * h["grad_scale"]
    if opt == "sgdm":
        m = h["momentum"] * m + g + h["weight_decay"] * w
        return w - h["lr"] * m, m, None
    if opt == "lars":
        a, b = w.norm(), g.norm()
        rate = h["trust_coeff"] * a / (b + h["weight_decay"] * a) if a > 0 and b > 0 else 1.0
        m = h["momentum"] * m + h["lr"] * rate * (g + h["weight_decay"] * w)
        return w - m, m, None
    t = h["step"]
    if opt == "adafactor":
        if g.numel() == 0:
            return w, None, v
        beta = 1.0 - t ** -h["decay_exponent"]
        q = g * g + h["eps"]
        if len(shape) < 2:
            v = beta * v + (1 - beta) * q
            u = g / v.sqrt()
        else:
            cols = shape[-1]
            rows = g.numel() // cols
            q = q.view(rows, cols)
            v = torch.cat([beta * v[:rows] + (1 - beta) * q.sum(1), beta * v[rows:] + (1 - beta) * q.sum(0)])
            u = (g.view(rows, cols) * (v[:rows].sum() / v[:rows]).sqrt()[:, None] / v[rows:].sqrt()).view(-1)
        rms = lambda x: float(x.square().mean().sqrt())  # noqa: E731
        rate = max(h["eps2"], rms(w)) * min(h["lr"], t ** -0.5) / max(1.0, rms(u) / h["clip_threshold"])
        return w - rate * u, None, v
    m = h["beta1"] * m + (1 - h["beta1"]) * g
    v = h["beta2"] * v + (1 - h["beta2"]) * g * g
    u = (m / (1 - h["beta1"] ** t)) / ((v / (1 - h["beta2"] ** t)).sqrt() + h["eps"])
    if opt == "adam":
        return w - h["lr"] * u, m, v
    u = u + h["weight_decay"] * w
    a, b = w.norm(), u.norm()
    return w - h["lr"] * (a / b if a > 0 and b > 0 else 1.0) * u, m, v


def exact(case, seed):
    c, h = case, _hyper(case)
    opt, numels, shapes = c["opt"], _numels(c), _shapes(c)
    offs, length = _offsets(numels)
    w, m, v = _state(c, seed, length)
    slots = _SLOTS[opt]
    if c["route"] in ("replica", "slices"):
        return _exact_shard(c, h, seed, numels, offs, length, w, m, v)
    grads = [_grads(c, seed, length, k) for k in range(c["copies"])]
    fsizes = _factored_sizes(c)
    fac = _factored(sum(fsizes), seed).double() if opt == "adafactor" else None
    master = c["route"] == "fused" and c["out"] == "f32"
    pw = None if master else _Packed(c, numels)
    pm = _Packed(c, numels) if slots else None
    pv = _Packed(c, numels) if slots == 2 else None
    weights = w.to(_DTYPE[c["out"]]).double()
    at = 0
    for t, (shape, n, o) in enumerate(zip(shapes, numels, offs)):
        g = torch.zeros(n, dtype=torch.float64, device="cuda")
        for a in grads:
            g += a[o:o + n]
        vt = fac[at:at + fsizes[t]] if fac is not None else v[o:o + n].double() if v is not None else None
        wt, mt, vt = _step64(h, opt, shape, g, w[o:o + n].double(), m[o:o + n].double() if slots else None, vt)
        weights[o:o + n] = wt
        if pw:
            pw.put(t, wt)
        if pm:
            pm.put(t, mt)
        if pv:
            pv.put(t, vt)
        if fac is not None:
            fac[at:at + fsizes[t]] = vt
            at += fsizes[t]
    got = {"weights": weights, "w": pw and pw.flat, "m": pm and pm.flat, "v": fac if fac is not None else pv and pv.flat}
    if c["route"] == "separate":
        got["gathered"] = pw.flat if c["out"] == "bf16" else None
        rows = []
        for a in grads:
            p = _Packed(c, numels)
            for t, (n, o) in enumerate(zip(numels, offs)):
                p.put(t, a[o:o + n].double())
            rows.append(p.flat)
        got["packed"] = torch.stack(rows)
    return got


def _exact_shard(c, h, seed, numels, offs, length, w, m, v):
    """One shard: elementwise on the packed state, its padding zero."""
    r, out = c["copies"] // 2, _DTYPE[c["out"]]

    def packed(a):
        if a is None:
            return None
        p = _Packed(c, numels)
        for t, (n, o) in enumerate(zip(numels, offs)):
            p.put(t, a[o:o + n].double())
        return p

    there = packed(torch.ones(length, device="cuda")).shard(r)      # 0 where the shard is padded
    pw, pm, pv = packed(w), packed(m), packed(v)
    ks = range(1, 2) if c["route"] == "replica" else range(c["copies"])
    g = torch.zeros(pw.S, dtype=torch.float64, device="cuda")
    for k in ks:
        g += _grads(c, seed, pw.S, k)
    sw, sm, sv = (None if p is None else p.shard(r).clone() for p in (pw, pm, pv))
    sw, sm, sv = (None if x is None else x * there for x in _step64(h, c["opt"], (pw.S,), g, sw, sm, sv))
    pw.flat = pw.flat.to(torch.float32).to(out).double()            # the other slots: the initial weights, narrowed
    pw.shard(r)[:] = sw
    got = {"gathered": pw.flat, "w": sw, "m": sm, "v": sv}
    if c["route"] == "replica":
        got["packed"] = packed(_grads(c, seed, length, 0)).flat
        weights = w.to(out).double()
        for t, (n, o) in enumerate(zip(numels, offs)):
            if pw.pieces is None:
                weights[o:o + n] = pw.flat[pw.offs[t]:pw.offs[t] + n]
            elif n:
                p = pw.pieces[t]
                weights[o:o + n] = pw.flat.view(pw.R, pw.S)[:, pw.offs[t]:pw.offs[t] + p].reshape(-1)[:n]
        got["weights"] = weights
    return got
