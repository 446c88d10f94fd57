"""The work whose speed is tracked: serving and set-up calls of the library as
a user's program makes them.

A case is a dict of plain values.  ``kind`` names the entry points it takes:

* ``apply``  grouped centroid + residual applies of one layer's projections
             (the batch is grouped beforehand: one build serves every layer);
* ``step``   a serving step: residual swaps on a side stream (when ``swap``),
             the build of the batch's segments, the applies of ``layers``
             layers;
* ``base``   the projections with their base weight, y = x W + delta;
* ``fold``   a scaled centroid folded into base weights (one call for one
             weight, a plan for several);
* ``align``  the alignment regulariser over pairs of adapters and centroids.

``shapes`` lists the projections of a layer as d_in x d_out, ``+`` between
projections that read the same activations (one grouped launch) and ``|``
between groups.  ``batch`` is how tokens are laid out: ``decode`` has one
token a request, users drawn Zipf(1.1) in arrival order; ``prefill`` has runs
of one user's tokens.  ``graph`` replays the launches from a CUDA graph, as a
decode loop does; without it they are launched one by one.
"""
import math
import random

import numpy as np
import torch

from paper_2608_03579_gb300 import salt
from paper_2608_03579_gb300.workloads import GAMMA_BINS, LLAMA3B_MLP, LLAMA3B_QKV, LLAMA8B_LAYER, MISTRAL7B_QV


def _text(*groups):
    return "|".join("+".join("%dx%d" % (a, b) for (_, a, b) in g) for g in groups)


QKV_3B = _text(LLAMA3B_QKV)
MLP_3B = _text(LLAMA3B_MLP[:2], LLAMA3B_MLP[2:])
LAYER_8B = _text(LLAMA8B_LAYER[:3], LLAMA8B_LAYER[3:4], LLAMA8B_LAYER[4:6], LLAMA8B_LAYER[6:])
QV_7B = _text(MISTRAL7B_QV)


def _serving(**kw):
    c = {"layers": 1, "batch": "decode", "mixed": False, "gamma": False, "none": 0.0, "ids": "host", "swap": 0,
         "graph": False, "layout": "out_in"}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: 16 tokens of four users on one small projection, launched on its own (latency)
        _serving(name="tiny apply", kind="apply", shapes="512x512", tokens=16, domains=2, rc=8, users=4, r=2, mixed=True),
        # decoding 64 requests of a 3B model: the q/k/v launch of a layer
        _serving(name="decode qkv 3b", kind="apply", shapes=QKV_3B, tokens=64, domains=4, rc=16, users=64, r=2),
        # decoding 256 requests of an 8B model whose requests carry gamma bins: a layer's four launches in a graph
        _serving(name="decode layer 8b gamma", kind="apply", shapes=LAYER_8B, tokens=256, domains=8, rc=64, users=256,
                 r=2, gamma=True, graph=True),
        # an 8192-token prefill batch of a 3B model: a layer's gate/up and down launches
        _serving(name="prefill mlp 3b", kind="apply", shapes=MLP_3B, tokens=8192, domains=4, rc=32, users=14, r=2,
                 mixed=True, batch="prefill"),
        # a whole decode step of an 8B model (four of its layers): 64 residuals swapped in, the build, the applies
        _serving(name="decode step 8b", kind="step", shapes=LAYER_8B, layers=4, tokens=512, domains=8, rc=64, users=512,
                 r=2, swap=64, graph=True),
        # the largest batch, ids already on the GPU, gamma bins, some requests without a centroid or a residual:
        # the build and the q/v launches of two layers
        _serving(name="prefill step qv 7b", kind="step", shapes=QV_7B, layers=2, tokens=16384, domains=4, rc=32,
                 users=48, r=2, mixed=True, gamma=True, none=0.1, ids="device", batch="prefill"),
        # the projections of an 8B layer with their base weights: 24 decode requests (bound by reading the weights)
        _serving(name="base decode 8b", kind="base", shapes=LAYER_8B, tokens=24, domains=4, rc=64, users=24, r=2,
                 graph=True),
        # the same for a full decode batch
        _serving(name="base step 8b", kind="base", shapes=LAYER_8B, tokens=512, domains=8, rc=64, users=448, r=2,
                 graph=True),
        # the same for a prefill batch of a 3B model's MLP, weights stored [d_in][d_out]
        _serving(name="base prefill mlp 3b", kind="base", shapes=MLP_3B, tokens=8192, domains=4, rc=32, users=14, r=2,
                 mixed=True, batch="prefill", layout="in_out"),
        # a centroid folded into one weight of a running node
        {"name": "fold one 3b", "kind": "fold", "shapes": "3072x3072", "copies": 1, "rc": 16, "layout": "in_out",
         "plan": False},
        # a node's start: a centroid folded into every weight of two 8B layers by one plan
        {"name": "fold plan 8b", "kind": "fold", "shapes": LAYER_8B, "copies": 2, "rc": 64, "layout": "out_in",
         "plan": True},
        # monitoring every adapted weight of an 8B model against its centroid
        {"name": "align 8b", "kind": "align", "shapes": LAYER_8B, "copies": 32, "r": 16, "rc": 64},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo=64, hi=14336):
    """A projection width: half the time a common one, else any multiple of 8 of the range."""
    if rng.random() < 0.5:
        return rng.choice([w for w in (512, 768, 1024, 2048, 3072, 4096, 5120, 8192, 14336) if lo <= w <= hi])
    return max(lo, min(hi, _log_int(rng, lo, hi) // 8 * 8))


def draw(rng):
    kind = rng.choice(["apply", "apply", "step", "base", "base", "fold", "align"])
    if kind == "fold":
        plan = rng.random() < 0.6
        groups, n = [], rng.randint(2, 7) if plan else 1
        for _ in range(n):
            groups.append("%dx%d" % (_width(rng), _width(rng)))
        return {"kind": "fold", "shapes": "|".join(groups), "copies": 1, "rc": rng.randint(1, 64),
                "layout": rng.choice(["in_out", "out_in"]), "plan": plan}
    if kind == "align":
        rc = rng.choice([8, 16, 32, 64, rng.randint(1, 64)])
        return {"kind": "align", "shapes": "|".join("%dx%d" % (_width(rng), _width(rng)) for _ in range(rng.randint(1, 7))),
                "copies": _log_int(rng, 1, 32), "r": rng.choice([1, 2, 16, rng.randint(1, 64)]), "rc": rc}
    batch = rng.choice(["decode", "prefill"])
    tokens = _log_int(rng, 1, 768) if batch == "decode" else _log_int(rng, 128, 8192)
    d_in = _width(rng)
    while True:  # one to three projections of the same activations
        outs = [_width(rng) for _ in range(rng.randint(1, 3))]
        if tokens * d_in * sum(outs) <= 1.5e11 and tokens * (d_in + 2 * sum(outs)) <= 2.5e8:
            break
        d_in = max(64, d_in // 2 // 8 * 8)
    plain = rng.random() < 0.15  # standard multi-LoRA: no centroid, larger ranks
    r = rng.choice([4, 8, 16]) if plain else rng.choice([1, 2, 2])
    users = max(1, min(tokens, _log_int(rng, 1, 256)))
    if batch == "prefill":
        users = max(1, min(users, tokens // 64))
    c = _serving(kind=kind, shapes="+".join("%dx%d" % (d_in, b) for b in outs), tokens=tokens,
                 domains=0 if plain else rng.randint(1, 8), rc=0 if plain else rng.choice([4, 8, 16, 32, 64, rng.randint(1, 64)]),
                 users=users, r=r, mixed=rng.random() < 0.5, batch=batch, gamma=not plain and rng.random() < 0.3,
                 none=rng.choice([0.0, 0.0, 0.1]), ids=rng.choice(["host", "device"]),
                 graph=batch == "decode" and rng.random() < 0.5, layout=rng.choice(["in_out", "out_in"]))
    if kind == "step":
        c["layers"] = rng.randint(1, 2)
        c["swap"] = rng.choice([0, max(1, users // 8)]) if batch == "decode" else 0
    return c


# ---------------------------------------------------------------- inputs
def _groups(case):
    return [[tuple(int(v) for v in p.split("x")) for p in g.split("+")] for g in case["shapes"].split("|")]


def _projections(case):
    """(d_in, d_out) of every adapted matrix, and the groups of their indices."""
    table, groups = [], []
    for _ in range(case.get("layers", case.get("copies", 1))):
        for g in _groups(case):
            groups.append(list(range(len(table), len(table) + len(g))))
            table += g
    return table, groups


def _ids(case, seed, turn=0):
    """(domains, slots, gamma bins) of the batch of one step.  A step that
    swaps reads the slots below ``users`` and, of the two regions above them
    that it fills in turn, the one filled the step before."""
    rs = np.random.RandomState((seed * 7919 + turn * 104729 + 17) % (1 << 31))
    T, n = case["tokens"], case["users"]
    if case["batch"] == "decode":
        readable = n + case["swap"]
        p = np.arange(1, readable + 1, dtype=np.float64) ** -1.1
        u = rs.permutation(readable)[rs.choice(readable, size=T, p=p / p.sum())]
    else:
        cuts = np.sort(rs.choice(np.arange(1, T), size=n - 1, replace=False)) if n > 1 else np.array([], dtype=np.int64)
        lens = np.diff(np.concatenate([[0], cuts, [T]]))
        u = np.repeat(rs.permutation(n), lens)
    slot = np.where(u < n, u, u + (case["swap"] if turn % 2 == 0 else 0)).astype(np.int32)
    dom = (slot % case["domains"]).astype(np.int32) if case["domains"] else np.full(T, -1, np.int32)
    if case["none"]:
        dom[rs.rand(T) < case["none"]] = -1
        slot[rs.rand(T) < case["none"]] = -1
    gb = rs.randint(0, len(GAMMA_BINS), T).astype(np.int32) if case["gamma"] else None
    return dom, slot, gb


def _rank(case, u):
    return 1 + (u + 1) % case["r"] if case["mixed"] else case["r"]


def _slots(case):
    return case["users"] + 2 * case["swap"]


class _Draws:
    """Seeded bf16 normals on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def __call__(self, *shape, std=1.0):
        return (torch.randn(*shape, generator=self.gen, device="cuda") * std).to(torch.bfloat16)


def _factors(case, seed):
    """Centroids per domain and residuals per slot, and per projection the
    activations, the y that comes in and (base) the weight."""
    table, groups = _projections(case)
    g = _Draws(seed)
    T, nd, rc = case["tokens"], case["domains"], case["rc"]
    ranks = [_rank(case, u) for u in range(_slots(case))]
    f = {"A": [], "B": [], "a": [], "b": [], "x": [], "y": [], "W": []}
    for din, dout in table:
        f["A"].append(g(nd, rc, din, std=din ** -0.5))
        f["B"].append(g(nd, rc, dout, std=max(rc, 1) ** -0.5))
        f["a"].append(g(len(ranks), case["r"], din, std=din ** -0.5))
        f["b"].append(g(len(ranks), case["r"], dout, std=case["r"] ** -0.5))
    for members in groups:
        x = g(T, table[members[0]][0])
        f["x"] += [x] * len(members)
        for l in members:
            din, dout = table[l]
            f["y"].append(g(T, dout) if case["kind"] != "base" else torch.empty(T, dout, dtype=torch.bfloat16, device="cuda"))
            if case["kind"] == "base":
                f["W"].append(g(din, dout, std=din ** -0.5) if case["layout"] == "in_out" else g(dout, din, std=din ** -0.5))
    return table, groups, ranks, f


S_C, S_U = 0.8, 1.25  # the centroids' and the residuals' scales


# ---------------------------------------------------------------- the states
_streams = []


def _engine_streams():
    """The engine's compute stream and its side stream for swaps: every batch
    goes through the same two, one after another."""
    if not _streams:
        _streams.extend([torch.cuda.Stream(), torch.cuda.Stream()])
    return _streams


class _Serving:
    """A context with its centroids pinned and its residual slots filled, a
    segments object and the batch's tensors."""

    def __init__(self, case, seed):
        self.case = case
        self.ctx = self.seg = self.graph = None
        table, self.groups, ranks, f = _factors(case, seed)
        d_in, d_out = [a for a, _ in table], [b for _, b in table]
        n_slots = len(ranks)
        self.ctx = salt.salt_ctx_create(d_in, d_out, case["domains"], case["rc"], n_slots, case["r"], case["tokens"])
        for d in range(case["domains"]):
            A = torch.cat([t[d].reshape(-1) for t in f["A"]])
            B = torch.cat([t[d].reshape(-1) for t in f["B"]])
            salt.salt_centroid_pin(self.ctx, d, case["rc"], A, B, S_C)
        self.comp, self.side = _engine_streams()
        # the host's residual cache: a blob for every slot, then one more for each slot that a step refills
        sizes = [salt.salt_residual_blob_bytes(d_in, d_out, r) for r in ranks]
        at = np.concatenate([[0], np.cumsum([(s + 255) // 256 * 256 for s in sizes])])
        self.host = salt.salt_host_alloc(int(at[-1]))
        packed = {}
        for r in sorted(set(ranks)):
            packed[r] = [torch.cat([t[:, :r].reshape(n_slots, -1) for t in f[k]], dim=1).view(torch.int16).cpu().numpy()
                         for k in ("a", "b")]
        blobs = []
        for u, r in enumerate(ranks):
            blob = self.host.tensor[int(at[u]):int(at[u]) + sizes[u]]
            salt.salt_residual_blob_pack(d_in, d_out, r, S_U, packed[r][0][u], packed[r][1][u], blob.numpy(), sizes[u])
            blobs.append(blob)
        salt.salt_residual_load_batch(self.ctx, list(range(n_slots)), blobs, self.comp)
        self.seg = salt.salt_segments_create(self.ctx)
        n, k = case["users"], case["swap"]
        self.regions = [list(range(n, n + k)), list(range(n + k, n + 2 * k))]
        # a refilled slot gets the other region's residual, back and forth
        self.refill = [[blobs[s] for s in self.regions[1 - i]] for i in range(2)]
        self.turn = 0
        self.ids = [_ids(case, seed, t) for t in range(2)]
        if case["ids"] == "device":
            self.ids = [tuple(None if v is None else torch.from_numpy(v).cuda() for v in i) for i in self.ids]
        self.xs, self.ys, self.ws = f["x"], f["y"], f["W"]
        self.layout = salt.SALT_W_IN_OUT if case["layout"] == "in_out" else salt.SALT_W_OUT_IN
        torch.cuda.synchronize()
        self.build(0)
        if case["graph"]:
            y0 = [y.clone() for y in self.ys]
            self.launches()
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=self.comp):
                self.launches()
            for y, keep in zip(self.ys, y0):
                y.copy_(keep)
            self.graph = g
        torch.cuda.synchronize()

    def build(self, turn):
        dom, slot, gb = self.ids[turn]
        if gb is None:
            salt.salt_build_segments(self.ctx, self.seg, dom, slot, stream=self.comp)
        else:
            salt.salt_build_segments_gamma(self.ctx, self.seg, dom, gb, slot, GAMMA_BINS, stream=self.comp)

    def launches(self):
        if self.case["kind"] == "base":
            for l, (x, w, y) in enumerate(zip(self.xs, self.ws, self.ys)):
                salt.salt_lora_apply_with_base(self.ctx, self.seg, l, x, w, self.layout, y, self.comp)
            return
        for g in self.groups:
            xs, ys = [self.xs[l] for l in g], [self.ys[l] for l in g]
            if len(g) == 1:
                salt.salt_lora_apply(self.ctx, self.seg, g[0], xs[0], ys[0], self.comp)
            else:
                salt.salt_lora_apply_grouped(self.ctx, self.seg, g, xs, ys, self.comp)

    def run(self):
        if self.case["kind"] == "step":
            if self.case["swap"]:
                salt.salt_residual_load_batch(self.ctx, self.regions[self.turn], self.refill[self.turn], self.side)
            self.build(self.turn)
            self.turn ^= 1
        if self.graph is not None:
            with torch.cuda.stream(self.comp):
                self.graph.replay()
        else:
            self.launches()
        return self.ys

    def __del__(self):
        if self.ctx:
            torch.cuda.synchronize()
            self.graph = None
            salt.salt_segments_destroy(self.seg)
            salt.salt_ctx_destroy(self.ctx)
            self.ctx = None


class _Fold:
    """A context with one pinned centroid and base weights to fold it into."""

    GAMMA = 0.6

    def __init__(self, case, seed):
        self.ctx = self.plan = None
        table, _ = _projections(case)
        A, B, self.ws = _fold_inputs(case, seed)
        self.ctx = salt.salt_ctx_create([a for a, _ in table], [b for _, b in table], 1, case["rc"], 1, 1, 16)
        salt.salt_centroid_pin(self.ctx, 0, case["rc"], torch.cat([t.reshape(-1) for t in A]),
                               torch.cat([t.reshape(-1) for t in B]), S_C)
        self.layout = salt.SALT_W_IN_OUT if case["layout"] == "in_out" else salt.SALT_W_OUT_IN
        self.gamma = self.GAMMA
        if case["plan"]:
            self.plan = salt.salt_fold_plan_create(self.ctx, 0, list(range(len(table))), self.ws, self.layout)

    def run(self):
        if self.plan is not None:
            salt.salt_fold_plan_run(self.plan, self.gamma)
        else:
            salt.salt_centroid_fold(self.ctx, 0, 0, self.gamma, self.ws[0], self.layout)
        self.gamma = -self.gamma  # folded in, taken out, in turn
        return self.ws

    def __del__(self):
        if self.ctx:
            torch.cuda.synchronize()
            salt.salt_fold_plan_destroy(self.plan)
            salt.salt_ctx_destroy(self.ctx)
            self.ctx = None


def _fold_inputs(case, seed):
    table, _ = _projections(case)
    g, rc = _Draws(seed), case["rc"]
    A = [g(rc, a, std=a ** -0.5) for a, _ in table]
    B = [g(rc, b, std=rc ** -0.5) for _, b in table]
    W = [g(*((a, b) if case["layout"] == "in_out" else (b, a)), std=a ** -0.5) for a, b in table]
    return A, B, W


class _Align:
    """Adapters close to their centroids, as training leaves them, and the prepared pairs."""

    def __init__(self, case, seed):
        self.tensors = _align_inputs(case, seed)
        table, _ = _projections(case)
        self.pairs = salt.salt_align_pairs([dict(At=t[0], B=t[1], At_c=t[2], B_c=t[3], r=case["r"], rc=case["rc"],
                                                 d_in=a, d_out=b, s=S_U, s_c=S_C)
                                            for t, (a, b) in zip(self.tensors, table)])
        n = len(table)
        self.loss, self.cosine = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")

    def run(self):
        salt.salt_align_loss(self.pairs, 1e-8, self.loss, self.cosine)
        return {"loss": self.loss, "cosine": self.cosine}


def _align_inputs(case, seed):
    table, _ = _projections(case)
    g, r, rc = _Draws(seed), case["r"], case["rc"]
    out = []
    for a, b in table:
        Ac, Bc = g(rc, a, std=a ** -0.5), g(rc, b, std=rc ** -0.5)
        At, Bt = g(r, a, std=a ** -0.5), g(r, b, std=rc ** -0.5)
        m = min(r, rc)
        At[:m] = (At[:m] * 0.5 + Ac[:m]).to(torch.bfloat16)
        Bt[:m] = (Bt[:m] * 0.5 + Bc[:m]).to(torch.bfloat16)
        out.append((At, Bt, Ac, Bc))
    return out


def prepare(case, seed):
    if case["kind"] == "fold":
        return _Fold(case, seed)
    if case["kind"] == "align":
        return _Align(case, seed)
    return _Serving(case, seed)


def run(state):
    return state.run()


# ---------------------------------------------------------------- accounting
def work(case):
    table, groups = _projections(case)
    if case["kind"] == "fold":
        rc = case["rc"]
        return {"bytes": sum(4 * a * b + 2 * rc * (a + b) for a, b in table), "flops": sum(2 * rc * a * b for a, b in table)}
    if case["kind"] == "align":
        s = case["r"] + case["rc"]
        return {"bytes": sum(2 * s * (a + b) for a, b in table) + 8 * len(table),
                "flops": sum(2 * s * s * (a + b) for a, b in table)}
    dom, slot, gb = _ids(case, 0)
    T = case["tokens"]
    act = int(((dom >= 0) | (slot >= 0)).sum())
    base = case["kind"] == "base"
    per_row = case["rc"] * (len(np.unique(dom[dom >= 0]))) + sum(_rank(case, int(u)) for u in np.unique(slot[slot >= 0]))
    per_tok = case["rc"] * int((dom >= 0).sum()) + sum(_rank(case, int(u)) for u in slot[slot >= 0])
    n_bytes = n_flops = 0
    for members in groups:
        n_bytes += 2 * (T if base else act) * table[members[0]][0]
        for l in members:
            a, b = table[l]
            n_bytes += 2 * per_row * (a + b) + (2 * T * b + 2 * a * b if base else 4 * act * b)
            n_flops += 2 * per_tok * (a + b) + (2 * T * a * b if base else 0)
    if case["kind"] == "step":
        n_bytes += 4 * T * (2 if gb is None else 3)
        n, k = case["users"], case["swap"]
        n_bytes += sum(2 * _rank(case, u) * sum(a + b for a, b in table) for u in range(n, n + k))
    return {"bytes": n_bytes, "flops": n_flops}


def tolerance(case):
    if case["kind"] == "align":
        return {"rel": 2e-5}  # fp32 sums of products of exactly represented values
    return {"rel": 6e-3}  # bf16 results, the low-rank intermediate rounded to bf16 too


# ---------------------------------------------------------------- the same in 64 bits
def exact(case, seed):
    f64 = torch.float64
    if case["kind"] == "fold":
        A, B, W = _fold_inputs(case, seed)
        out = []
        for a, b, w in zip(A, B, W):
            d = a.to(f64).T @ b.to(f64) if case["layout"] == "in_out" else b.to(f64).T @ a.to(f64)
            out.append(w.to(f64) + _Fold.GAMMA * S_C * d)
        return out
    if case["kind"] == "align":
        loss, cosine = [], []
        for t in _align_inputs(case, seed):
            At, Bt, Ac, Bc = (v.to(f64) for v in t)

            def inner(p, q, u, v):  # <p^T q, u^T v> from the factors' Gram matrices
                return ((p @ u.T) * (q @ v.T)).sum()

            num = S_U * S_C * inner(At, Bt, Ac, Bc)
            den = S_U * S_C * torch.sqrt(inner(At, Bt, At, Bt) * inner(Ac, Bc, Ac, Bc))
            cosine.append(num / (den + 1e-8))
            loss.append(1 - cosine[-1])
        return {"loss": torch.stack(loss), "cosine": torch.stack(cosine)}
    table, _, ranks, f = _factors(case, seed)
    dom, slot, gb = _ids(case, seed, 0)
    T = case["tokens"]
    dom_t, slot_t = torch.from_numpy(dom).cuda().long(), torch.from_numpy(slot).cuda().long()
    scale = torch.full((T,), S_C, dtype=f64, device="cuda")
    if gb is not None:
        scale *= torch.tensor(np.array(GAMMA_BINS, np.float32).astype(np.float64), device="cuda")[torch.from_numpy(gb).cuda().long()]
    rank_t = torch.tensor(ranks, device="cuda")
    out = []
    for l, (din, dout) in enumerate(table):
        x = f["x"][l].to(f64)
        if case["kind"] == "base":
            y = x @ (f["W"][l].to(f64) if case["layout"] == "in_out" else f["W"][l].to(f64).T)
        else:
            y = f["y"][l].to(f64)
        for d in range(case["domains"]):
            at = (dom_t == d).nonzero()[:, 0]
            if len(at):
                y[at] += (scale[at, None] * (x[at] @ f["A"][l][d].to(f64).T)) @ f["B"][l][d].to(f64)
        for first in range(0, T, 512):
            at = torch.arange(first, min(T, first + 512), device="cuda")
            at = at[slot_t[at] >= 0]
            if len(at):
                s = slot_t[at]
                v = torch.einsum("td,trd->tr", x[at], f["a"][l][s].to(f64))
                v = v * (torch.arange(case["r"], device="cuda")[None, :] < rank_t[s][:, None])
                y[at] += S_U * torch.einsum("tr,trd->td", v, f["b"][l][s].to(f64))
        out.append(y)
    return out


if __name__ == "__main__":  # what the cases are and what they cost at least
    for c in listed() + [dict(draw(random.Random(i)), name="drawn %d" % i) for i in range(6)]:
        w = work(c)
        print("%-24s %10.2f MB %10.2f GFLOP" % (c["name"], w["bytes"] / 1e6, w["flops"] / 1e9))
