"""Performance cases of the representative-token selection library.

Each case is one piece of work that a program using the library has it do, through the
public calls of `paper_2605_03110_b200.binding`: the selection of one layer, the selection
chain over the layers of a model, one representative set per attention head, what consumes the
set (nearest-representative map and attention on the representatives), and the calls that take
host buffers.  Sizes are those of the repository's own workloads (`workloads.CONFIGS`, the
crossover sweep and their head splits) plus lengths and widths that fit no tile.

Inputs follow the recipe of `workloads.py` -- prototypes, noise around them, drift, re-drawn and
fresh rows from layer to layer -- drawn on the GPU from the seed alone.

  op       full    ada_select_full on one layer (Definition 1)
           step    ada_cascade_step on one layer (Algorithm 1) with an inherited set
           heads   ada_cascade_step_heads: one set per head
           pipe    full selection at layer 0, then a cascade step per later layer; `adaptive`:
                   the steps carry the device-resident threshold (Section 8.1)
           attend  ada_nearest_rep, then ada_attention_reps with the expansion to every token
           host    ada_cascade_step_host on pinned host buffers
  q        share of the tokens that are representatives of the set at hand (prototypes / T)
  causal   ADA_CROSS_CAUSAL in the steps (ADA_ATTN_CAUSAL in the attention)
"""
import math

import torch

from paper_2605_03110_b200 import binding as ada

TAU = 0.3
SIGMA = 0.05                     # noise of a token around its prototype
DELTA, RHO, PHI = 0.02, 0.02, 0.003   # drift, re-drawn share and fresh share per layer


def _case(name, op, dtype, T, d, q, B=1, h=1, L=1, causal=False, adaptive=False):
    c = {"op": op, "dtype": dtype, "B": B, "T": T, "d": d, "h": h, "L": L, "q": q,
         "causal": causal, "adaptive": adaptive}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: layer 0 of a GPT-2-sized model on a 512-token text, fp32 activations
        _case("full-f32-512", "full", "f32", 512, 768, 0.2),
        # the whole selection of that model, twelve layers: launches and host time count
        _case("pipe-f32-512", "pipe", "f32", 512, 768, 0.2, L=12),
        # a batch of mid-length texts through the same width in bf16
        _case("pipe-bf16-8x2048", "pipe", "bf16", 2048, 768, 0.065, B=8, L=12),
        # layer 0 of a GPT-J-sized model on a 2048-token prompt
        _case("full-bf16-2048", "full", "bf16", 2048, 4096, 0.2),
        # the selection of that model on a prompt whose length fits no tile, causal cross check
        # and adaptive threshold on
        _case("pipe-bf16-2005-adaptive", "pipe", "bf16", 2005, 4096, 0.2, L=28, causal=True, adaptive=True),
        # layer 0 (and, without the cascade, every layer) of a long prompt of a 6.7B-sized model
        _case("full-bf16-8192", "full", "bf16", 8192, 4096, 0.05),
        # the selection of that model, 32 layers: the repository's headline workload
        _case("pipe-bf16-8192", "pipe", "bf16", 8192, 4096, 0.05, L=32),
        # the ends of the crossover sweep at its greatest length: few representatives (a stream
        # over the activations) and half of all tokens
        _case("step-bf16-16384-sparse", "step", "bf16", 16384, 4096, 0.01),
        _case("step-bf16-16384-dense", "step", "bf16", 16384, 4096, 0.5),
        # one set per attention head, 32 heads of 128
        _case("heads-bf16-2048", "heads", "bf16", 2048, 128, 0.2, h=32),
        # what a layer's attention does with its set: 32 heads of 128, a long prompt and the few
        # hundred representatives of its first layers
        _case("attend-bf16-8192", "attend", "bf16", 8192, 128, 0.05, h=32),
        # activations that live in host memory: copies and the step in one call
        _case("host-bf16-2048", "host", "bf16", 2048, 4096, 0.2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _log_width(rng, lo, hi, step):
    return max(step, _log_int(rng, lo, hi) // step * step)


def draw(rng):
    """A case of the ranges above: lengths of 256..16384 tokens (fp32: ..2048), widths of
    256..5120 (any width whose rows are whole 16-byte units), sets of 1 %..50 % of the tokens.
    No more work than the 32-layer chain of the headline workload."""
    while True:
        op = rng.choice(["full", "full", "step", "step", "step", "pipe", "pipe", "heads", "attend", "host"])
        q = round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4)
        causal = rng.random() < 0.3
        if op == "heads":
            c = _case(None, op, "bf16", _log_int(rng, 256, 8192), rng.choice([32, 64, 80, 96, 128]), q,
                      h=rng.choice([8, 12, 16, 25, 32]), causal=causal)
        elif op == "attend":
            c = _case(None, op, "bf16", _log_int(rng, 256, 8192), rng.choice([32, 64, 80, 96, 128]), q,
                      h=rng.choice([8, 12, 16, 25, 32]), causal=causal)
            # sets of a few hundred representatives: at most 148 tiles of 128 query rows over the heads
            if -(-_protos(c["T"], q) // 128) * c["h"] > 148:
                continue
        else:
            f32 = op != "host" and rng.random() < 0.25
            T = _log_int(rng, 256, 2048 if f32 else 16384)
            d = _log_width(rng, 256, 1600 if f32 else 5120, 4 if f32 else 8)
            B = rng.choice([1, 1, 1, 2, 5, 8])
            c = _case(None, op, "f32" if f32 else "bf16", T, d, q, B=B, L=rng.randint(3, 16) if op == "pipe" else 1,
                      causal=causal, adaptive=op == "pipe" and rng.random() < 0.3)
        w = work(c)
        if w["bytes"] <= 2.0e9 and w["flops"] <= 1.2e12 and (op != "host" or w["bytes"] <= 7e7):
            return c


# ---------------------------------------------------------------- inputs
class _Activations:
    """fp32 activations of B sequences (B, T, d), layer by layer."""

    def __init__(self, gen, B, T, d, P):
        dev = gen.device
        self.gen, self.B, self.T, self.d, self.P = gen, B, T, d, P
        self.protos = torch.randn((B, P, d), generator=gen, device=dev)
        # every prototype has at least one token
        perm = torch.rand((B, T), generator=gen, device=dev).argsort(1)
        lab = torch.randint(P, (B, T), generator=gen, device=dev)
        lab[:, :P] = torch.arange(P, device=dev)
        self.labels = torch.empty_like(lab).scatter_(1, perm, lab)
        self.fresh = P                                    # next label of a token of its own
        self.X = torch.randn((B, T, d), generator=gen, device=dev).mul_(SIGMA)
        for b in range(B):
            self.X[b] += self.protos[b, self.labels[b]]

    def advance(self):
        g, dev = self.gen, self.gen.device
        self.X.add_(torch.randn(self.X.shape, generator=g, device=dev), alpha=DELTA)
        n_re, n_fr = int(RHO * self.T), int(PHI * self.T)
        for b in range(self.B):
            pos = torch.randperm(self.T, generator=g, device=dev)
            re, fr = pos[:n_re], pos[n_re:n_re + n_fr]
            if n_re:
                j = torch.randint(self.P, (n_re,), generator=g, device=dev)
                self.X[b, re] = self.protos[b, j] + SIGMA * torch.randn((n_re, self.d), generator=g, device=dev)
                self.labels[b, re] = j
            if n_fr:
                self.X[b, fr] = torch.randn((n_fr, self.d), generator=g, device=dev)
                self.labels[b, fr] = self.fresh + torch.arange(n_fr, device=dev)
        self.fresh += n_fr

    def first_of_each(self):
        """The set a full selection of this layer yields: the first token of every label.
        Returns ascending lists (B, T) int32, zero past the counts, and the counts (B)."""
        dev = self.gen.device
        idx = torch.zeros((self.B, self.T), dtype=torch.int32, device=dev)
        cnt = torch.zeros((self.B,), dtype=torch.int32, device=dev)
        t = torch.arange(self.T, device=dev)
        for b in range(self.B):
            first = torch.full((self.fresh,), self.T, device=dev).scatter_reduce_(0, self.labels[b], t, "amin")
            reps = first[first < self.T].sort().values
            idx[b, :reps.numel()] = reps.to(torch.int32)
            cnt[b] = reps.numel()
        return idx, cnt


def _protos(T, q):
    return min(T, max(1, int(round(q * T))))


def _lists(L, B, T, dev, gamma):
    """The output buffers of L selection calls, kept from call to call: one tensor per list,
    and per call a view of each."""
    keep = {k: torch.zeros((L, B, T), dtype=torch.int32, device=dev) for k in ("rep", "add", "rem")}
    keep.update({k + "_cnt": torch.zeros((L, B), dtype=torch.int32, device=dev) for k in ("rep", "add", "rem")})
    if gamma:
        keep.update({k: torch.zeros((L, B, T), device=dev) for k in ("gamma_rep", "gamma_cross")})
    outs = []
    for l in range(L):
        o = ada.CascadeOut(1, 1, dev, want_gamma=False)
        o.rep_out, o.rep_out_cnt = keep["rep"][l], keep["rep_cnt"][l]
        o.add_idx, o.add_cnt = keep["add"][l], keep["add_cnt"][l]
        o.rem_idx, o.rem_cnt = keep["rem"][l], keep["rem_cnt"][l]
        if gamma:
            o.gamma_rep, o.gamma_cross = keep["gamma_rep"][l], keep["gamma_cross"][l]
        outs.append(o)
    return keep, outs


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    op, B, T, d, h, L = case["op"], case["B"], case["T"], case["d"], case["h"], case["L"]
    kind = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    code = ada.ADA_F32 if case["dtype"] == "f32" else ada.ADA_BF16
    P = _protos(T, case["q"])
    st = {"op": op, "flags": ada.ADA_CROSS_CAUSAL if case["causal"] else 0}

    if op == "attend":
        act = _Activations(gen, 1, T, h * d, P)
        st["rep"], st["rep_cnt"] = act.first_of_each()
        st["X"] = act.X.to(kind)
        del act
        st["QKV"] = [torch.randn((T, h, d), generator=gen, device=dev).to(kind) for _ in range(3)]
        st["out"] = torch.zeros((T, h, d), device=dev)
        st["flags"] = ada.ADA_ATTN_CAUSAL if case["causal"] else 0
        st["ctx"] = ada.ada_create(1, T, h * d, code, device=dev.index)
        return st

    n_seq = h if op == "heads" else B
    act = _Activations(gen, n_seq, T, d, P)
    st["ctx"] = ada.ada_create(n_seq, T, d, code, device=dev.index)
    if op == "full":
        st["X"] = act.X.to(kind)
        st["idx"] = torch.zeros((B, T), dtype=torch.int32, device=dev)
        st["cnt"] = torch.zeros((B,), dtype=torch.int32, device=dev)
        st["gamma"] = torch.zeros((B, T), device=dev)
    elif op == "pipe":
        st["layers"] = []
        for l in range(L):
            if l:
                act.advance()
            st["layers"].append(act.X.to(kind))
        st["keep"], st["outs"] = _lists(L, B, T, dev, gamma=False)
        st["tau"] = None
        if case["adaptive"]:
            st["tau"] = torch.empty((B,), dtype=torch.float64, device=dev)
            st["policy"] = ada.TauPolicy(0.2, 0.1, 0.25, 0.35)
            st["turnover"] = torch.zeros((L, B), device=dev)
    else:                                  # step, heads, host: the set of the layer before
        st["rep"], st["rep_cnt"] = act.first_of_each()
        act.advance()
        if op == "heads":                  # (T, h, d): the heads of a token side by side
            st["X"] = act.X.transpose(0, 1).contiguous().to(kind)
        else:
            st["X"] = act.X.to(kind)
        if op == "host":
            pinned = lambda t: t.cpu().pin_memory()  # noqa: E731
            st["X"], st["rep"], st["rep_cnt"] = pinned(st["X"]), pinned(st["rep"]), pinned(st["rep_cnt"])
            st["lists"] = [torch.zeros(s, dtype=torch.int32).pin_memory() for _ in range(3) for s in ((B, T), (B,))]
            st["gammas"] = [torch.zeros((B, T)).pin_memory() for _ in range(2)]
        else:
            st["keep"], st["outs"] = _lists(1, n_seq, T, dev, gamma=True)
    return st


# ---------------------------------------------------------------- one pass
def run(st):
    op, ctx, flags = st["op"], st["ctx"], st["flags"]
    if op == "full":
        ada.ada_select_full(ctx, st["X"], TAU, st["idx"], st["cnt"], st["gamma"])
        return st["idx"], st["cnt"], st["gamma"]
    if op == "step":
        ada.ada_cascade_step(ctx, st["X"], TAU, st["rep"], st["rep_cnt"], out=st["outs"][0], flags=flags)
        return st["keep"]
    if op == "heads":
        ada.ada_cascade_step_heads(ctx, st["X"], TAU, st["rep"], st["rep_cnt"], out=st["outs"][0], flags=flags)
        return st["keep"]
    if op == "pipe":
        layers, outs, tau = st["layers"], st["outs"], st["tau"]
        ada.ada_select_full(ctx, layers[0], TAU, outs[0].rep_out, outs[0].rep_out_cnt, want_gamma=False)
        if tau is None:
            for l in range(1, len(layers)):
                ada.ada_cascade_step(ctx, layers[l], TAU, outs[l - 1].rep_out, outs[l - 1].rep_out_cnt,
                                     out=outs[l], flags=flags)
            return st["keep"]
        tau.fill_(TAU)                     # every prompt starts from the same threshold
        for l in range(1, len(layers)):
            ada.ada_cascade_step_adaptive(ctx, layers[l], tau, st["policy"], outs[l - 1].rep_out,
                                          outs[l - 1].rep_out_cnt, out=outs[l], flags=flags,
                                          turnover=st["turnover"][l])
        return st["keep"], tau, st["turnover"]
    if op == "attend":
        near, g = ada.ada_nearest_rep(ctx, st["X"], st["rep"], st["rep_cnt"])
        ada.ada_attention_reps(ctx, *st["QKV"], st["rep"][0], st["rep_cnt"], nearest_idx=near[0], out=st["out"],
                               flags=flags)
        return near, g, st["out"]
    rep, rep_cnt, add, add_cnt, rem, rem_cnt = st["lists"]
    ada.ada_cascade_step_host(ctx, st["X"], TAU, st["rep"], st["rep_cnt"], rep, rep_cnt, add, add_cnt, rem, rem_cnt,
                              *st["gammas"], flags=flags)
    # host lists come back at full capacity with whatever the device buffers held past the counts
    for x, c in ((rep, rep_cnt), (add, add_cnt), (rem, rem_cnt)):
        for b, n in enumerate(c.tolist()):
            x[b, n:].zero_()
    return st["lists"], st["gammas"]


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    op, B, T, d, h, L = case["op"], case["B"], case["T"], case["d"], case["h"], case["L"]
    es = 4 if case["dtype"] == "f32" else 2
    r = _protos(T, case["q"])

    def full(n):                            # lower triangle of the Gram
        return d * T * (T - 1.0) * n

    def step(n, r):                         # r x r among the inherited, (T - r) x r across
        return (d * r * (r - 1.0) + 2.0 * d * (T - r) * r) * n

    x = float(T) * d * es
    if op == "full":
        return {"bytes": B * (x + T * 4 + r * 4), "flops": full(B)}
    if op == "pipe":
        fl = full(B) + sum(step(B, min(T, r + l * int(PHI * T))) for l in range(L - 1))
        return {"bytes": L * B * (x + 2 * r * 4), "flops": fl}
    if op == "attend":
        hd = h * d
        # X once for the map; Q, K, V only at the representatives; every output row once
        b = float(T) * hd * es + 3.0 * r * hd * es + float(T) * hd * 4 + 2.0 * T * 4
        att = 4.0 * r * r * hd * (0.5 if case["causal"] else 1.0)
        return {"bytes": b, "flops": 2.0 * hd * (T - r) * r + att}
    n = h if op == "heads" else B
    return {"bytes": n * (x + 2 * T * 4 + 3 * r * 4), "flops": step(n, r)}


def tolerance(case):
    # Lists, counts and the map are whole numbers: no correlation of these inputs lies near the
    # threshold and no two candidates of the map are close, so they are the same.
    if case["op"] == "pipe" and not case["adaptive"]:
        return "exact"
    if case["op"] == "attend":
        # bf16 operands, probabilities rounded to bf16 between the two contractions
        return {"rel": 1e-2, "max": 0.1}
    return {"rel": 1e-5, "max": 1e-4}       # fp32 sums of exact products
