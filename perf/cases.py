"""The calls whose speed is tracked, each through the package's public entry points.

Four kinds of call, after what a program that serves or calibrates a compressed
Mixtral-style model does with this library:

  layer       ``moe_forward`` on a workspace that the program keeps: one MoE block
              of a decode step (a few tokens) or of a prefill (thousands)
  static      ``moe_forward_static``, for programs that may not hold a workspace
  stack       ``stack_forward``: several pre-norm residual blocks in one call
  importance  ``token_importance``: the Eq. 6 importance of a prompt's tokens and
              the protect mask, from the block's attention map

Shapes are the ones of the benchmark and of the tests: the Mixtral-8x7b block
(H 4096, F 14336, 8 experts), the 8x22b block (H 6144, F 16384), the tiny layer
(H 256, F 512, group 64), and a half-size block for unquantised fp16 experts.

The weights of a seed are one model: cases of the same shape and bit table share
them (a program packs a model once and calls it at many batch sizes), and packed
host buffers are kept for the next preparation, at most ``KEPT`` of them.
"""
import math
from collections import OrderedDict

import numpy as np
import torch

import paper_2410_06270_gb300 as mc

DEV = "cuda"
B20 = "2,2,3,3,1,3,3,3"   # mean 2.50 bits, the benchmark's decode table
B16 = "2,3,1,2,3,2,1,2"   # mean 2.00
B13 = "1,2,1,3,1,2,2,1"   # mean 1.63
KEPT = 8                  # packed host buffers kept

M7 = {"H": 4096, "F": 14336, "E": 8}
M22 = {"H": 6144, "F": 16384, "E": 8}
TINY = {"H": 256, "F": 512, "E": 8}
HALF = {"H": 2048, "F": 7168, "E": 8}


def _layer(T, shape, bits=B20, group=128, mu=0.0, protect=0.0, drop=0.0, skew=0.0, routing=False, kind="layer"):
    return {"kind": kind, "T": T, **shape, "group": group, "bits": bits, "mu": mu, "protect": protect, "drop": drop,
            "skew": skew, "routing": routing}


def listed():
    return [
        # the smallest layer, all options on: launch count and host time decide
        {"name": "tiny64", **_layer(64, TINY, "3,2,2,1,3,2,2,3", group=64, mu=0.3, protect=0.25, routing=True)},
        # one token of one user: decode latency of a block
        {"name": "decode1", **_layer(1, M7)},
        # a small batch where no workspace may be held
        {"name": "decode5_static", **_layer(5, M7, kind="static")},
        # the decode batch that the benchmark's headline is quoted on
        {"name": "decode16", **_layer(16, M7)},
        # a decode batch of many users, ODP on, an odd size
        {"name": "decode45_odp", **_layer(45, M7, mu=0.3, protect=0.1)},
        # a short prompt with ODP, protected tokens and the routing handed back
        {"name": "odp256", **_layer(256, M7, mu=0.3, protect=0.1, routing=True)},
        # the benchmark's prefill: a long prompt, skewed expert loads
        {"name": "prefill4096", **_layer(4096, M7, skew=0.9)},
        # an odd prompt length, groups of 64, a smaller bit budget, 2% of tokens dropped
        {"name": "prefill1019_g64", **_layer(1019, M7, B16, group=64, mu=0.3, protect=0.1, drop=0.02)},
        # the larger model of the paper at the decode batch
        {"name": "decode16_8x22b", **_layer(16, M22)},
        # unquantised experts: the baseline that a user compares the compressed layer with
        {"name": "decode16_fp16", **_layer(16, HALF, "16")},
        # eight residual blocks of a decode step in one call, ODP on
        {"name": "stack8_32", **_layer(32, M7, mu=0.165, protect=0.1, kind="stack"), "layers": 8},
        # the protect mask of a 2048-token prompt from its 32-head attention map
        {"name": "importance2048", "kind": "importance", "L": 2048, "H": 4096, "heads": 32, "protect": 0.02},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _table(rng):
    b = rng.choice([B20, B20, B16, B13]).split(",")
    rng.shuffle(b)
    return ",".join(b)


def draw(rng):
    what = rng.choice(["layer"] * 6 + ["static", "stack", "fp16", "importance"])
    if what == "importance":
        return {"kind": "importance", "L": _log_int(rng, 48, 2048), "H": rng.choice([2048, 4096]),
                "heads": rng.choice([8, 16, 32]), "protect": rng.choice([0.02, 0.1])}
    odp = rng.random() < 0.5
    opts = {"mu": 0.3 if odp else 0.0, "protect": 0.1 if odp else 0.0}
    if what == "fp16":
        return _layer(_log_int(rng, 1, 40), rng.choice([TINY, HALF]), "16", **opts)
    if what == "static":
        return _layer(_log_int(rng, 1, 90), rng.choice([TINY, HALF, M7]), _table(rng), rng.choice([64, 128]),
                      kind="static", **opts)
    if what == "stack":
        return {**_layer(_log_int(rng, 1, 48), rng.choice([HALF, M7]), _table(rng), mu=0.165, protect=0.1,
                         kind="stack"), "layers": rng.randint(2, 8)}
    skew = rng.choice([0.0, 0.9])
    return _layer(_log_int(rng, 1, 4096), rng.choice([TINY, HALF, M7, M7]), _table(rng), rng.choice([64, 128, 128]),
                  drop=0.02 if odp and rng.random() < 0.3 else 0.0, skew=skew, routing=rng.random() < 0.3, **opts)


# ------------------------------------------------------------------ inputs --

def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + stream) % (1 << 62))


def _bits(case):
    b = [int(v) for v in case["bits"].split(",")]
    return b * case["E"] if len(b) == 1 else b


def _std_scale(m):
    return 1.0 if m < 2 else 0.2  # a block adds to the residual without drowning it


class _Weights:
    """The canonical experts of a seed, on the device.  One draw of rows serves
    every matrix, each from another place of it: codes of N(0, 0.02) weights under a
    min-max scale, fractional zero points around the middle of the range (HQQ
    storage), 1-bit signs with z = 1/2.  Values only, any expert on request."""

    def __init__(self, case, seed):
        self.case, self.bits = case, _bits(case)
        H, F = case["H"], case["F"]
        g = _gen(seed, 1)
        self.place = torch.randint(0, 4096, (case["E"], 3), generator=g, device=DEV).cpu().numpy() * 64
        n = H * F + 4096 * 64
        self.w = torch.randn(n, generator=g, device=DEV)
        if self.bits[0] == 16:
            self.w = (self.w * 0.02).half()
            return
        ng = H * F // case["group"] + 4096 * 64
        self.jitter = torch.rand(ng, generator=g, device=DEV) * 0.45 + 0.8
        self.shift = torch.randn(ng, generator=g, device=DEV) * 0.25
        self.codes = {}
        for b in sorted(set(self.bits)):
            top = (1 << b) - 1
            q = (self.w >= 0) if b == 1 else (self.w * (top / 5.2) + top / 2).round().clamp(0, top)
            self.codes[b] = q.to(torch.uint8)
        del self.w

    def shape(self, m):
        c = self.case
        return (c["F"], c["H"]) if m < 2 else (c["H"], c["F"])

    def matrix(self, e, m):
        """(codes, scale, zero) of a quantised matrix, or (fp16 weights, None, None)."""
        rows, cols = self.shape(m)
        at, b = int(self.place[e, m]), self.bits[e]
        if b == 16:
            return self.w[at:at + rows * cols].view(rows, cols) * _std_scale(m), None, None
        ng, top = cols // self.case["group"], (1 << b) - 1
        jitter = self.jitter[at:at + rows * ng].view(rows, ng)
        scale = (jitter * (2 * 0.8 * 0.02 if b == 1 else 5.2 * 0.02 / top) * _std_scale(m)).half()
        zero = torch.full_like(scale, 0.5) if b == 1 else \
            (self.shift[at:at + rows * ng].view(rows, ng) + top / 2).half()
        return self.codes[b][at:at + rows * cols].view(rows, cols), scale, zero

    def exact(self, e, m):
        """The dequantised matrix in 64 bits."""
        q, s, z = self.matrix(e, m)
        if s is None:
            return q.double()
        rows, cols = self.shape(m)
        return ((q.view(rows, -1, self.case["group"]).double() - z.double()[..., None]) *
                s.double()[..., None]).view(rows, cols)


_kept = OrderedDict()


def _packed(case, seed):
    """This seed's experts, packed and on the device."""
    key = (seed, case["H"], case["F"], case["E"], case["group"], case["bits"])
    shape = mc.Shape(case["E"], case["H"], case["F"], case["group"])
    if key not in _kept:
        W = _Weights(case, seed)
        host = {b: c.cpu() for b, c in W.codes.items()} if W.bits[0] != 16 else {}
        codes, scales, zeros = [], [], []
        for e in range(case["E"]):
            for m in range(3):
                q, s, z = W.matrix(e, m)
                if s is None:
                    codes.append(q.cpu().numpy())
                else:
                    at = int(W.place[e, m])
                    codes.append(host[W.bits[e]][at:at + q.numel()].view(q.shape).numpy())
                scales.append(None if s is None else s.cpu().numpy())
                zeros.append(None if z is None else z.cpu().numpy())
        _kept[key] = mc.pack_experts_host(shape, W.bits, codes, scales, zeros)
        while len(_kept) > KEPT:
            _kept.popitem(last=False)
    _kept.move_to_end(key)
    return shape, mc.upload_packed(_kept[key], DEV)


def _tokens(case, seed):
    """(x, gates [layers, E, H], protect) of a layer or a stack."""
    T, H, E = case["T"], case["H"], case["E"]
    g = _gen(seed, 2)
    x = torch.randn(T, H, generator=g, device=DEV)
    if case["kind"] == "stack":
        # tokens that belong to two experts' directions, as a trained router's do:
        # the gates read them clearly through every block of the residual stream
        u = torch.linalg.qr(torch.randn(H, E, generator=g, device=DEV))[0].T
        pick = torch.rand(T, E, generator=g, device=DEV).argsort(dim=1)
        r = math.sqrt(H / 4096)
        first = torch.where(torch.rand(T, 1, generator=g, device=DEV) < 0.25, 70.0 * r, 40.0 * r)
        x += first * u[pick[:, 0]] + 25.0 * r * u[pick[:, 1]]
        noise = torch.randn(case["layers"], E, H, generator=g, device=DEV)
        gates = (0.1 / r) * u[None] + 0.02 / H ** 0.5 * noise
    else:
        gates = torch.randn(1, E, H, generator=g, device=DEV) * (1.28 / H ** 0.5)
        if case["skew"]:
            u = torch.randn(H, generator=g, device=DEV)
            u /= u.norm()
            x += 3.0 * u
            gates += (case["skew"] * torch.linspace(-1, 1, E, device=DEV))[:, None] * u
    protect = None
    if case["protect"] or case["drop"]:
        order = torch.rand(T, generator=g, device=DEV).argsort()
        protect = torch.zeros(T, dtype=torch.uint8, device=DEV)
        protect[order[:math.ceil(case["protect"] * T)]] = 1
        if case["drop"]:
            protect[order[T - math.ceil(case["drop"] * T):]] = 2
    return x.bfloat16(), gates.bfloat16(), protect


def _attention(case, seed):
    L, nh = case["L"], case["heads"]
    g = _gen(seed, 3)
    t = torch.randn(L, case["H"], generator=g, device=DEV).bfloat16()
    attn = torch.empty(nh, L, L, device=DEV)
    above = torch.ones(L, L, dtype=torch.bool, device=DEV).triu(1)
    for h in range(nh):
        s = torch.randn(L, L, generator=g, device=DEV).masked_fill_(above, -math.inf)
        torch.softmax(s, dim=1, out=attn[h])
    return t, attn


def prepare(case, seed):
    if case["kind"] == "importance":
        t, attn = _attention(case, seed)
        n = mc.load().mc_token_importance_workspace_size(case["L"])
        return {"case": case, "t": t, "attn": attn, "ws": torch.empty(n, dtype=torch.uint8, device=DEV)}
    shape, packed = _packed(case, seed)
    x, gates, protect = _tokens(case, seed)
    s = {"case": case, "shape": shape, "x": x, "gate": gates[0].contiguous(), "protect": protect,
         "bits": np.asarray(_bits(case), np.int8), "packed": packed}
    if case["kind"] == "layer":
        s["ws"] = mc.alloc_workspace(shape, case["T"])
    elif case["kind"] == "stack":
        n = case["layers"]
        # one device copy of the experts per block, so that every block streams its own
        s["args"] = mc.StackArgs([g.contiguous() for g in gates], [s["bits"]] * n,
                                 [packed] + [packed.clone() for _ in range(n - 1)], [case["mu"]] * n)
        s["gamma"] = torch.ones(n, case["H"], dtype=torch.bfloat16, device=DEV)
        s["ws"] = mc.stack_workspace(shape, case["T"])
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "importance":
        importance, mask = mc.token_importance(s["t"], s["attn"], c["protect"], workspace=s["ws"])
        return {"importance": importance, "mask": mask}
    if c["kind"] == "static":
        return {"y": mc.moe_forward_static(s["x"], s["gate"], s["shape"], s["bits"], s["packed"], c["mu"],
                                           s["protect"])}
    if c["kind"] == "stack":
        h = s["x"].clone()  # updated in place
        return {"y": mc.stack_forward(h, s["shape"], s["args"], s["gamma"], s["ws"], s["protect"])}
    if c["routing"]:
        y, r = mc.moe_forward(s["x"], s["gate"], s["shape"], s["bits"], s["packed"], c["mu"], s["protect"],
                              workspace=s["ws"], routing=True)
        return {"y": y, **r}
    return {"y": mc.moe_forward(s["x"], s["gate"], s["shape"], s["bits"], s["packed"], c["mu"], s["protect"],
                                workspace=s["ws"])}


# ------------------------------------------------------ what a pass costs --

def _kept_pairs(case):
    """Expected (token, slot) pairs: ODP drops a secondary whose weight is below mu
    of the primary's, for gate logits ~ N(0, 1.28)."""
    T = case["T"]
    if not case["mu"]:
        return 2.0 * T
    if case["kind"] == "stack":
        cut = 0.25
    else:
        l = np.sort(np.random.default_rng(0).standard_normal((20000, case["E"])) * 1.28, axis=1)
        cut = float(np.mean(l[:, -1] - l[:, -2] > -math.log(case["mu"])))
    return T * (2.0 - cut * (1.0 - case["protect"])) * (1.0 - case["drop"])


def work(case):
    if case["kind"] == "importance":
        L = case["L"]
        return {"bytes": case["heads"] * L * (L + 1) / 2 * 4 + L * case["H"] * 2 + L * 5,
                "flops": case["heads"] * L * (L + 1) / 2}
    T, H, F, E = case["T"], case["H"], case["F"], case["E"]
    per = np.mean([H * F * b / 8 + (0 if b == 16 else H * F / case["group"] * 4) for b in _bits(case)])
    pairs = _kept_pairs(case)
    touched = E * (1.0 - (1.0 - 2.0 / E) ** (pairs / 2.0))
    n = case.get("layers", 1)
    return {"bytes": n * (touched * 3 * per + E * H * 2) + 4 * T * H, "flops": n * (pairs * 6 * H * F + 2 * T * E * H)}


def tolerance(case):
    if case["kind"] == "importance":
        # fp32 sums of up to 2048 x 32 probabilities; the mask flips at a near-tie
        return {"rel": 2e-6, "max": 2e-5, "differ": 0.002}
    if case["kind"] == "stack":
        # the blocks' bf16 roundings add up: about 6e-3 off the 64-bit result after eight
        return {"rel": 2e-2, "max": 0.2}
    # bf16 output over fp16 inputs of both contractions: about 2e-3 off the 64-bit result
    return {"rel": 7e-3, "max": 0.05, "differ": 0.001}


# ---------------------------------------------------------- the same, 64 bits --

def _exact_block(x, gate, W, mu, protect):
    """(y, idx, w, pruned) of one block: x and gate in 64 bits."""
    T = x.shape[0]
    top, idx = (x @ gate.T).sort(dim=1, descending=True, stable=True)
    top, idx = top[:, :2], idx[:, :2]
    w = torch.softmax(top, dim=1)
    mask = torch.zeros(T, dtype=torch.uint8, device=DEV) if protect is None else protect
    pruned = ((mask == 0) & (w[:, 1] < mu * w[:, 0])).to(torch.uint8)
    w = torch.where(pruned[:, None] == 1, w.new_tensor([1.0, 0.0]), w)
    w = torch.where(mask[:, None] == 2, torch.zeros_like(w), w)
    pruned[mask == 2] = 2
    y = torch.zeros_like(x)
    for e in range(W.case["E"]):
        share = torch.where(idx == e, w, torch.zeros_like(w)).sum(dim=1)
        at = share.nonzero()[:, 0]
        if at.numel():
            xe = x[at]
            a = xe @ W.exact(e, 0).T
            h = a * torch.sigmoid(a) * (xe @ W.exact(e, 1).T)
            y[at] += share[at, None] * (h @ W.exact(e, 2).T)
    return y, idx.int(), w, pruned


def exact(case, seed):
    if case["kind"] == "importance":
        t, attn = _attention(case, seed)
        L = case["L"]
        col = torch.zeros(L, dtype=torch.float64, device=DEV)
        for a in attn:
            col += a.double().sum(dim=0)
        seen = torch.arange(L, 0, -1, dtype=torch.float64, device=DEV)
        imp = t.double().abs().sum(dim=1) * col / case["heads"] / seen
        mask = torch.zeros(L, dtype=torch.uint8, device=DEV)
        mask[imp.sort(descending=True, stable=True)[1][:math.ceil(case["protect"] * L - 1e-6)]] = 1
        return {"importance": imp, "mask": mask}
    W = _Weights(case, seed)
    x, gates, protect = _tokens(case, seed)
    if case["kind"] == "stack":
        h = x.double()
        for g in gates:
            n = h / (h.square().mean(dim=1, keepdim=True) + 1e-5).sqrt()
            h = h + _exact_block(n, g.double(), W, case["mu"], protect)[0]
        return {"y": h}
    y, idx, w, pruned = _exact_block(x.double(), gates[0].double(), W, case["mu"], protect)
    return {"y": y, "idx": idx, "w": w, "pruned": pruned} if case["routing"] else {"y": y}
