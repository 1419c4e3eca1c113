"""What is measured: the work that users of this framework have it do, through its public entry points.

A robot's control loop binds the new observation (``Expert.set_prefix``: the prefix keys and values, or
the prefix tokens, that the vision-language encoder left on the GPU), starts a chunk
(``Expert.denoise``) and reads the actions back (``Expert.finish``); a server does the same for many
robots at once. ``uad_linear`` is the projection op on its own, for callers with layers of their own.
The experts are those of the repository's configurations, benchmark and tests; weights N(0, 0.02),
prefixes and noise N(0, 1), rounded to bf16 where the expert is bf16, everything drawn from the seed.
"""
import math
import random

import numpy as np
import torch

import paper_2609_37772_gb300 as uad

# The experts, by their sizes: fp32 "tiny" and its RoPE / grouped-head variant; the pi0-like action
# expert and its small variant (joint attention over the prefix and the chunk, adaptive RMSNorm);
# the DiT head and its small variant (self- and cross-attention, adaLN); and the SmolVLA-style
# expert whose time embedding joins the action embedding.
EXPERTS = {
    "tiny": dict(kind="adarms", dtype="f32", n_layers=2, width=256, n_heads=4, n_kv_heads=4, head_dim=64,
                 mlp_dim=1024, action_dim=7, chunk_len=16, prefix_len=64, prefix_width=0, rope=False),
    "tiny_rope": dict(kind="adarms", dtype="f32", n_layers=2, width=256, n_heads=4, n_kv_heads=2, head_dim=64,
                      mlp_dim=1024, action_dim=7, chunk_len=16, prefix_len=64, prefix_width=0, rope=True),
    "pi0": dict(kind="adarms", dtype="bf16", n_layers=18, width=1024, n_heads=8, n_kv_heads=1, head_dim=256,
                mlp_dim=4096, action_dim=32, chunk_len=50, prefix_len=816, prefix_width=0, rope=True),
    "pi0_small": dict(kind="adarms", dtype="bf16", n_layers=2, width=512, n_heads=4, n_kv_heads=1, head_dim=128,
                      mlp_dim=1536, action_dim=32, chunk_len=50, prefix_len=200, prefix_width=0, rope=True),
    "dit": dict(kind="dit", dtype="bf16", n_layers=16, width=1536, n_heads=24, n_kv_heads=24, head_dim=64,
                mlp_dim=6144, action_dim=32, chunk_len=16, prefix_len=300, prefix_width=2048, rope=False),
    "dit_small": dict(kind="dit", dtype="bf16", n_layers=2, width=384, n_heads=6, n_kv_heads=6, head_dim=64,
                      mlp_dim=1536, action_dim=32, chunk_len=16, prefix_len=72, prefix_width=256, rope=False),
    "concat_small": dict(kind="concat", dtype="bf16", n_layers=2, width=512, n_heads=8, n_kv_heads=2, head_dim=64,
                         mlp_dim=1536, action_dim=32, chunk_len=50, prefix_len=120, prefix_width=0, rope=True),
}

L2_BYTES = 129e6


def _chunk(expert, robots, n_star, first, urgent, observe, **more):
    """A chunk: `robots` robots of `expert`, N* = n_star, the first `urgent` actions released after `first`
    steps ("mixed": each robot draws its own from the sweep grid); `observe`: every robot binds a new
    observation first."""
    return dict(op="chunk", expert=expert, robots=robots, n_star=n_star, first=first, urgent=urgent, observe=observe, **more)


def _linear(rows, k, n, static=False):
    return dict(op="linear", rows=rows, k=k, n=n, static=static)


def listed():
    return [
        # one DiT token block through its qkv projection: the smallest call, one weight read
        dict(name="linear-16", **_linear(16, 1536, 4608)),
        # the MLP down projection of 13 robots' chunks (odd number of rows), long K
        dict(name="linear-637", **_linear(637, 4096, 1024)),
        # the gate/up projection of a 64-robot batch: the largest single projection
        dict(name="linear-3200", **_linear(3200, 1024, 8192)),
        # a small fp32 expert for one robot: latency of a chain of short kernels
        dict(name="tiny-b1", **_chunk("tiny", 1, 10, 5, 4, True)),
        # the same expert serving a batch of simulated robots, each on its own schedule
        dict(name="tiny-b32", **_chunk("tiny", 32, 10, 5, 4, False, mixed=True)),
        # the headline control loop: one robot replans on a new observation
        dict(name="pi0-b1", **_chunk("pi0", 1, 10, 4, 10, True, middle=7)),
        # a few robots on one GPU, odd prefix and chunk lengths (another camera set and horizon)
        dict(name="pi0-b4", **_chunk("pi0", 4, 10, 4, 10, False, mixed=True, prefix_len=579, chunk_len=45)),
        # a server's batch, every robot with a new observation
        dict(name="pi0-b16", **_chunk("pi0", 16, 10, 4, 10, True, mixed=True)),
        # the largest batch: throughput serving
        dict(name="pi0-b64", **_chunk("pi0", 64, 10, 4, 10, False, mixed=True)),
        # the DiT head replans on a new observation with few steps
        dict(name="dit-b1", **_chunk("dit", 1, 4, 2, 4, True)),
        # the DiT head for four robots at many steps (uniform schedule: plain flow matching)
        dict(name="dit-b4", **_chunk("dit", 4, 16, 16, 0, False)),
        # the SmolVLA-style expert with odd lengths, rotation-vector dimensions corrected on SO(3)
        dict(name="concat-b5", **_chunk("concat_small", 5, 10, 3, 9, True, mixed=True, prefix_len=113, chunk_len=37, rot_dim=3)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """The same ranges: projections of 1 to 3200 rows over the experts' widths, chunks of every expert
    from one robot to the batches above, with other chunk and prefix lengths, step counts and release
    groups, with and without a new observation. A drawn chunk costs no more than the 64-robot one."""
    if rng.random() < 0.25:
        rows, k, n = _log_int(rng, 1, 3200), 64 * _log_int(rng, 4, 96), 128 * _log_int(rng, 3, 64)
        return _linear(rows, k, n, rows * n <= 1 << 20 and rng.random() < 0.3)
    expert = rng.choice(["tiny", "tiny_rope", "pi0", "pi0", "pi0", "pi0_small", "dit", "dit", "dit_small", "concat_small"])
    most = dict(tiny=64, tiny_rope=64, pi0=32, pi0_small=64, dit=8, dit_small=32, concat_small=32)[expert]
    base = EXPERTS[expert]
    robots = _log_int(rng, 1, most)
    n_star = rng.randint(4, 16 if expert != "pi0" else 12)
    observe = rng.random() < 0.5
    if expert == "dit" and observe:
        robots, n_star = min(robots, 2), min(n_star, 10)   # the prefix projections of a DiT are a chunk's worth each
    h = rng.randint(base["chunk_len"] // 2, base["chunk_len"])
    p = rng.randint(base["prefix_len"] // 2, base["prefix_len"])
    first = rng.randint(1, n_star)
    more = dict(mixed=True) if robots > 1 and rng.random() < 0.5 else {}
    if rng.random() < 0.25:
        more["rot_dim"] = 3
    if rng.random() < 0.15:
        more["released_frozen"] = True   # the ablation without Trajectory Reconciliation
    return _chunk(expert, robots, n_star, first, rng.randint(1, h // 2) if first < n_star else 0, observe,
                  prefix_len=p, chunk_len=h, **more)


# ---- inputs -----------------------------------------------------------------------------------------


def _arch(case):
    a = dict(EXPERTS[case["expert"]])
    for key in ("prefix_len", "chunk_len"):
        a[key] = case.get(key, a[key])
    return a


def _weight_shapes(a):
    """The tensors of the weight blob in the order that the library documents."""
    W, D, F, Pw = a["width"], a["action_dim"], a["mlp_dim"], a["prefix_width"]
    q, kv = a["n_heads"] * a["head_dim"], a["n_kv_heads"] * a["head_dim"]
    if a["kind"] == "concat":
        s = [("in_w", (D, W)), ("in_b", (W,)), ("ti_wa", (W, W)), ("ti_wt", (W, W)), ("ti_b", (W,)), ("to_w", (W, W)), ("to_b", (W,))]
    else:
        s = [("t_w1", (W, W)), ("t_b1", (W,)), ("t_w2", (W, W)), ("t_b2", (W,)), ("in_w", (D, W)), ("in_b", (W,))]
    for i in range(a["n_layers"]):
        if a["kind"] == "dit":
            layer = [("mod_w", (W, 6 * W)), ("mod_b", (6 * W,)), ("wq", (W, q)), ("wk", (W, q)), ("wv", (W, q)), ("wo", (q, W)),
                     ("wqc", (W, q)), ("wkc", (Pw, q)), ("wvc", (Pw, q)), ("woc", (q, W)),
                     ("w1", (W, F)), ("b1", (F,)), ("w2", (F, W)), ("b2", (W,))]
        else:
            attn = [("wq", (W, q)), ("wk", (W, kv)), ("wv", (W, kv)), ("wo", (q, W))]
            mlp = [("wg", (W, F)), ("wu", (W, F)), ("wd", (F, W))]
            if a["kind"] == "adarms":
                attn = [("mod1_w", (W, 3 * W)), ("mod1_b", (3 * W,))] + attn
                mlp = [("mod2_w", (W, 3 * W)), ("mod2_b", (3 * W,))] + mlp
            layer = attn + mlp
        s += [("l%d.%s" % (i, n), sh) for n, sh in layer]
    if a["kind"] != "concat":
        s += [("modf_w", (W, 2 * W)), ("modf_b", (2 * W,))]
    return s + [("out_w", (W, D)), ("out_b", (D,))]


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    return g


def _randn(shape, g, dtype):
    """N(0, 1) values of the expert's type, as the fp32 tensor that holds them."""
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    return x.bfloat16().float() if dtype == "bf16" else x


def _weights(a, g):
    n = sum(math.prod(s) for _, s in _weight_shapes(a))
    w = torch.randn(n, generator=g, device="cuda", dtype=torch.float32).mul_(0.02)
    return w.bfloat16().float() if a["dtype"] == "bf16" else w


def _prefixes(a, robots, g):
    """Per robot: keys and values [L][P][Hkv][dh], or prefix tokens [P][prefix_width]."""
    got = []
    for _ in range(robots):
        if a["kind"] == "dit":
            got.append((_randn((a["prefix_len"], a["prefix_width"]), g, a["dtype"]), None))
        else:
            shape = (a["n_layers"], a["prefix_len"], a["n_kv_heads"], a["head_dim"])
            got.append((_randn(shape, g, a["dtype"]), _randn(shape, g, a["dtype"])))
    return got


def _budgets(case, a, seed):
    """int32 [robots][H]: a first group of urgent actions, perhaps a middle one, the rest at N*."""
    B, H, N = case["robots"], a["chunk_len"], case["n_star"]
    r = random.Random(seed)
    out = np.full((B, H), N, dtype=np.int32)
    for b in range(B):
        k, u = case["first"], case["urgent"]
        if case.get("mixed"):
            k, u = min(N, r.choice((2, 3, 4, 6))), min(H - 1, r.choice((5, 10, 20)))
        if case.get("middle"):
            out[b, : H // 2] = min(N, case["middle"])
        out[b, :u] = k
    return out


def _chunk_inputs(case, seed):
    a = _arch(case)
    g = _generator(seed)
    weights = _weights(a, g)
    prefixes = _prefixes(a, case["robots"], g)
    noise = torch.randn((case["robots"], a["chunk_len"], a["action_dim"]), generator=g, device="cuda", dtype=torch.float32)
    options = dict(tr=True, gac=True)
    if case.get("released_frozen"):
        options = dict(tr=False, gac=False)
    elif case.get("rot_dim"):
        options["rot_dim"] = case["rot_dim"]
    return a, weights, prefixes, noise, _budgets(case, a, seed), options


def _linear_inputs(case, seed):
    g = _generator(seed)
    x = torch.randn((case["rows"], case["k"]), generator=g, device="cuda").bfloat16()
    w = torch.randn((case["k"], case["n"]), generator=g, device="cuda").mul_(0.02).bfloat16().float()
    bias = torch.randn(case["n"], generator=g, device="cuda").mul_(0.02)
    return x, w, bias


def prepare(case, seed):
    if case["op"] == "linear":
        x, w, bias = _linear_inputs(case, seed)
        tiled = torch.from_numpy(uad.tile_weight(w.cpu().numpy()).view(np.int16)).cuda()
        out = torch.empty((case["rows"], case["n"]), device="cuda")
        return dict(case=case, x=x, w=tiled, bias=bias, out=out)
    a, weights, prefixes, noise, budgets, options = _chunk_inputs(case, seed)
    expert = uad.Expert(a, weights, max_batch=case["robots"])
    if a["dtype"] == "bf16":
        prefixes = [(k.bfloat16(), None if v is None else v.bfloat16()) for k, v in prefixes]
    torch.cuda.synchronize()
    for b, (k, v) in enumerate(prefixes):
        expert.set_prefix(b, k, v, dtype=a["dtype"])
    expert.prepare_times(case["n_star"])   # as a program does at start-up, before its control loop
    return dict(case=case, expert=expert, dtype=a["dtype"], prefixes=prefixes, noise=noise, budgets=budgets, options=options)


def run(state):
    case = state["case"]
    stream = torch.cuda.current_stream()
    if case["op"] == "linear":
        x, out = state["x"], state["out"]
        entry = uad.uad_linear_static_scratch if case["static"] else uad.uad_linear
        rc = entry(x.data_ptr(), state["w"].data_ptr(), state["bias"].data_ptr(), out.data_ptr(),
                   case["rows"], case["n"], case["k"], stream.cuda_stream)
        if rc:
            raise RuntimeError("uad_linear: %d" % rc)
        return out
    expert = state["expert"]
    if case["observe"]:
        for b, (k, v) in enumerate(state["prefixes"]):
            expert.set_prefix(b, k, v, dtype=state["dtype"])
    expert.denoise(state["noise"], state["budgets"], stream=stream, **state["options"])
    out = expert.finish()
    # E, the estimate that the tail of `final` is corrected by, is a sum of differences of nearly equal
    # actions: its own relative error says nothing, and what it is for shows in `final`
    return {"final": out["final"], "ghost": out["ghost"]}


# ---- what a pass cannot do without, and how exact its results are ----------------------------------


def _layer_params(a):
    """Weights of one layer's projections (the time conditioning is tabulated at start-up)."""
    W, F = a["width"], a["mlp_dim"]
    q, kv = a["n_heads"] * a["head_dim"], a["n_kv_heads"] * a["head_dim"]
    if a["kind"] == "dit":
        return W * 3 * q + q * W + 2 * W * q + 2 * W * F
    return W * (q + 2 * kv) + q * W + 3 * W * F


def work(case):
    if case["op"] == "linear":
        m, k, n = case["rows"], case["k"], case["n"]
        return {"bytes": 2.0 * (m * k + k * n) + 4.0 * (n + m * n), "flops": 2.0 * m * k * n}
    a = _arch(case)
    es = 2 if a["dtype"] == "bf16" else 4
    B, H, P, D, W, L, N = (case["robots"], a["chunk_len"], a["prefix_len"], a["action_dim"], a["width"], a["n_layers"], case["n_star"])
    q, kv = a["n_heads"] * a["head_dim"], a["n_kv_heads"] * a["head_dim"]
    M = B * H
    params = L * _layer_params(a) + 2 * W * D + (2 * W * W if a["kind"] == "concat" else 0)
    keys = P + H
    flops = 2.0 * M * params + 4.0 * M * L * q * keys
    # each evaluation reads the weights and the prefix keys and values once, unless the L2 can hold them
    resident = es * (params + 2.0 * B * L * P * (q if a["kind"] == "dit" else kv))
    total = resident * (N if resident > L2_BYTES else 1) + 4.0 * M * D * 3
    flops *= N
    if case["observe"]:
        if a["kind"] == "dit":
            flops += 2.0 * B * P * a["prefix_width"] * 2 * q * L
            total += es * (B * P * a["prefix_width"] + 2.0 * L * a["prefix_width"] * q + 2.0 * B * L * P * q)
        else:
            total += 2.0 * es * 2 * B * L * P * kv
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # about four times what the path is from 64 bits
    if case["op"] == "linear":
        return {"rel": 2e-5, "max": 2e-4}     # bf16 products summed in 32 bits: 2e-7 (K = 1536) to 4.4e-6 (K = 4096)
    if EXPERTS[case["expert"]]["dtype"] == "f32":
        return {"rel": 1e-6, "max": 2e-5}     # 32 bits throughout: 1e-7
    return {"rel": 4e-3, "max": 5e-2}         # bf16 operands through every layer: 5e-4 to 1.1e-3


# ---- the same in 64 bits ------------------------------------------------------------------------------


def _sinusoid(values, width, scale):
    half = width // 2
    f = torch.exp(-math.log(10000.0) * torch.arange(half, dtype=torch.float64, device="cuda") / half)
    ang = scale * values[:, None] * f[None, :]
    return torch.cat([torch.sin(ang), torch.cos(ang)], dim=1)


def _silu(x):
    return x * torch.sigmoid(x)


def _gelu(x):
    return 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))


def _rope(x, first):
    """x [B][n][heads][dh], rotate-half at positions first + i."""
    dh, n = x.shape[-1], x.shape[1]
    inv = 10000.0 ** (-torch.arange(dh // 2, dtype=torch.float64, device="cuda") * 2 / dh)
    ang = (first + torch.arange(n, dtype=torch.float64, device="cuda"))[:, None] * inv[None, :]
    c, s = torch.cos(ang)[None, :, None, :], torch.sin(ang)[None, :, None, :]
    x1, x2 = x[..., : dh // 2], x[..., dh // 2:]
    return torch.cat([x1 * c - x2 * s, x2 * c + x1 * s], dim=-1)


def _attend(q, k, v):
    """q [B][n][Hq][dh], k and v [B][m][Hkv][dh]."""
    rep = q.shape[2] // k.shape[2]
    k, v = (t.repeat_interleave(rep, dim=2).permute(0, 2, 1, 3) for t in (k, v))
    s = q.permute(0, 2, 1, 3) @ k.transpose(-1, -2) / math.sqrt(q.shape[-1])
    return (torch.softmax(s, dim=-1) @ v).permute(0, 2, 1, 3).reshape(q.shape[0], q.shape[1], -1)


def _rms(h):
    return h / torch.sqrt((h * h).mean(-1, keepdim=True) + 1e-6)


def _ln(h):
    return (h - h.mean(-1, keepdim=True)) / torch.sqrt(h.var(-1, unbiased=False, keepdim=True) + 1e-6)


class _Exact:
    """The velocity network in 64 bits, all robots at once."""

    def __init__(self, a, blob, prefixes):
        self.a, self.w, off = a, {}, 0
        for name, shape in _weight_shapes(a):
            n = math.prod(shape)
            self.w[name] = blob[off:off + n].reshape(shape)   # converted where it is used
            off += n
        B, L = len(prefixes), a["n_layers"]
        if a["kind"] == "dit":
            t = torch.stack([k for k, _ in prefixes]).double()
            shape = (B, a["prefix_len"], a["n_heads"], a["head_dim"])
            self.k = [(t @ self.at(i, "wkc")).reshape(shape) for i in range(L)]
            self.v = [(t @ self.at(i, "wvc")).reshape(shape) for i in range(L)]
        else:
            self.k = [torch.stack([k[i] for k, _ in prefixes]).double() for i in range(L)]
            self.v = [torch.stack([v[i] for _, v in prefixes]).double() for i in range(L)]

    def get(self, name):
        return self.w[name].double()

    def at(self, layer, name):
        return self.w["l%d.%s" % (layer, name)].double()

    def velocity(self, u, tau):
        a, W = self.a, self.a["width"]
        B, H = u.shape[:2]
        h = u @ self.get("in_w") + self.get("in_b")
        values, where = torch.unique(tau, return_inverse=True)   # tau [B][H]
        e = _sinusoid(values, W, 1000.0)
        if a["kind"] == "concat":
            te = (e @ self.get("ti_wt"))[where]
            h = _silu(h @ self.get("ti_wa") + te + self.get("ti_b")) @ self.get("to_w") + self.get("to_b")
        else:
            c = _silu(_silu(e @ self.get("t_w1") + self.get("t_b1")) @ self.get("t_w2") + self.get("t_b2"))

        def mod(w, b, n):
            m = (c @ w + b)[where]
            return [m[..., i * W:(i + 1) * W] for i in range(n)]

        def heads(x, n):
            return x.reshape(B, H, n, a["head_dim"])

        if a["kind"] == "dit":
            h = h + _sinusoid(torch.arange(H, dtype=torch.float64, device="cuda"), W, 1.0)[None]
        for i in range(a["n_layers"]):
            at = lambda n: self.at(i, n)  # noqa: E731
            if a["kind"] == "dit":
                sh1, sc1, g1, sh2, sc2, g2 = mod(at("mod_w"), at("mod_b"), 6)
                y = _ln(h) * (1 + sc1) + sh1
                q, k, v = (heads(y @ at(n), a["n_heads"]) for n in ("wq", "wk", "wv"))
                h = h + g1 * (_attend(q, k, v) @ at("wo"))
                h = h + _attend(heads(_ln(h) @ at("wqc"), a["n_heads"]), self.k[i], self.v[i]) @ at("woc")
                y = _ln(h) * (1 + sc2) + sh2
                h = h + g2 * (_gelu(y @ at("w1") + at("b1")) @ at("w2") + at("b2"))
                continue
            y = _rms(h)
            g1 = g2 = 1.0
            if a["kind"] == "adarms":
                sc, sh, g1 = mod(at("mod1_w"), at("mod1_b"), 3)
                y = y * (1 + sc) + sh
            q, k, v = heads(y @ at("wq"), a["n_heads"]), heads(y @ at("wk"), a["n_kv_heads"]), heads(y @ at("wv"), a["n_kv_heads"])
            if a["rope"]:
                q, k = _rope(q, a["prefix_len"]), _rope(k, a["prefix_len"])
            o = _attend(q, torch.cat([self.k[i], k], 1), torch.cat([self.v[i], v], 1))
            h = h + g1 * (o @ at("wo"))
            y = _rms(h)
            if a["kind"] == "adarms":
                sc, sh, g2 = mod(at("mod2_w"), at("mod2_b"), 3)
                y = y * (1 + sc) + sh
            h = h + g2 * ((_gelu(y @ at("wg")) * (y @ at("wu"))) @ at("wd"))
        if a["kind"] == "concat":
            y = _rms(h)
        elif a["kind"] == "dit":
            sh, sc = mod(self.get("modf_w"), self.get("modf_b"), 2)
            y = _ln(h) * (1 + sc) + sh
        else:
            sc, sh = mod(self.get("modf_w"), self.get("modf_b"), 2)
            y = _rms(h) * (1 + sc) + sh
        return y @ self.get("out_w") + self.get("out_b")


def _rotation(w):
    """exp of a rotation vector, float64 [3] -> [3][3]."""
    K = np.array([[0.0, -w[2], w[1]], [w[2], 0.0, -w[0]], [-w[1], w[0], 0.0]])
    t = float(np.linalg.norm(w))
    if t < 1e-12:
        return np.eye(3) + K
    return np.eye(3) + math.sin(t) / t * K + (1 - math.cos(t)) / t ** 2 * (K @ K)


def _rotation_vector(R):
    """log of a rotation, through its unit quaternion: the principal vector."""
    K = np.array([
        [R[0, 0] - R[1, 1] - R[2, 2], 0, 0, 0],
        [R[0, 1] + R[1, 0], R[1, 1] - R[0, 0] - R[2, 2], 0, 0],
        [R[0, 2] + R[2, 0], R[1, 2] + R[2, 1], R[2, 2] - R[0, 0] - R[1, 1], 0],
        [R[2, 1] - R[1, 2], R[0, 2] - R[2, 0], R[1, 0] - R[0, 1], R[0, 0] + R[1, 1] + R[2, 2]]]) / 3
    _, vec = np.linalg.eigh(K, UPLO="L")
    q = vec[:, -1] * (1 if vec[3, -1] >= 0 else -1)
    s = float(np.linalg.norm(q[:3]))
    return 2 * q[:3] if s < 1e-12 else 2 * math.atan2(s, q[3]) / s * q[:3]


def exact(case, seed):
    if case["op"] == "linear":
        x, w, bias = _linear_inputs(case, seed)
        return x.double() @ w.double() + bias.double()
    a, weights, prefixes, noise, budgets, options = _chunk_inputs(case, seed)
    if work(case)["flops"] > 1e13:
        return None   # over 20 seconds in 64 bits
    net = _Exact(a, weights, prefixes)
    B, H, D = noise.shape
    N = torch.from_numpy(budgets).cuda()
    top = N.max(dim=1, keepdim=True).values.expand(B, H)
    early = N < top
    x = noise.double()
    g = x.clone()
    tr = options["tr"]
    released = torch.zeros_like(x)
    for k in range(1, int(N.max()) + 1):
        active = k <= N
        tau = torch.where(active, (k - 1) / N.double(), (k - 1) / top.double() if tr else torch.ones_like(N, dtype=torch.float64))
        u = torch.where(active[..., None], x, g if tr else released)
        v = net.velocity(u, tau)
        running = (k <= top)[..., None]   # a robot's state rests after its own last step
        x = torch.where(active[..., None], x + v / N[..., None], x)
        if tr:
            g = torch.where(early[..., None] & running, g + v / top[..., None], g)
        released = torch.where((early & (N == k))[..., None], x, released)
    x, g, released, early = (t.cpu().numpy() for t in (x, g, released, early))
    final = x.copy()
    ghost = np.where(early[..., None], g if tr else released, x)
    E = np.zeros((B, D))
    rot = options.get("rot_dim")
    for b in range(B):
        idx, tail = np.nonzero(early[b])[0], np.nonzero(~early[b])[0]
        if not options["gac"] or not len(idx) or not len(tail):
            continue
        E[b] = (g[b, idx] - released[b, idx]).sum(0)
        plain = np.ones(D, bool)
        if rot is not None:
            rd = slice(rot, rot + 3)
            plain[rd] = False
            err = np.eye(3)
            for i in idx:
                err = _rotation(g[b, i, rd]) @ _rotation(released[b, i, rd]).T @ err
            E[b, rd] = _rotation_vector(err)
            step = _rotation(E[b, rd] / len(tail))
            for i in tail:
                # of the vectors for this rotation (whole turns apart), the one nearest to the action
                w = _rotation_vector(step @ _rotation(x[b, i, rd]))
                turn = 2 * math.pi * w / max(float(np.linalg.norm(w)), 1e-12)
                final[b, i, rd] = min((w + m * turn for m in (-1, 0, 1)), key=lambda c: float(np.linalg.norm(c - x[b, i, rd])))
        final[np.ix_([b], tail, np.nonzero(plain)[0])] += E[b, plain] / len(tail)
    return {"final": final, "ghost": ghost}
