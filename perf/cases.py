"""The work that a user of the framework has it do, as cases to measure.

Every case is a call through the package's public entry points (the C ABI of
libshard by its Python binding), on the shard shapes that this repository
names -- the tiny shard and the 8B and 70B stages, fewer layers of them where
a layer says the same as the whole stage -- or, when drawn, on generic shapes
of the same ranges.  Kinds:

  step     `shard_step`, one decode or verify step of B requests
  packed   `shard_step_packed`, S rows of one packed cache row
  host     `shard_step_host`, the step on host buffers, as the speculative
           driver and the rank pipeline call it
  prefill  `shard_prefill`, prompts (or the turns of conversations)
  top1     `head_top1`, the final stage's greedy token and its probability
  logits   `head_debug_logits`, the same head's logits

A decoding request lasts `steps` steps; then the next request, whose prompt is
already cached, takes its place, so a pass is one step of a serving loop and
the cache length stays in the request's range.  Weights are Gaussian,
quantised to uint4 as the exporter does it; K, V and hidden states are N(0, 1).
"""
import types

import numpy as np
import torch

import paper_2608_19147_gb300 as pkg

DEV = "cuda" if torch.cuda.is_available() else "cpu"
EPS, THETA = 1e-5, 500000.0

TINY = dict(hidden=256, heads=4, kv_heads=2, head_dim=64, ffn=688, group=32, sigma=0.02)
B8 = dict(hidden=4096, heads=32, kv_heads=8, head_dim=128, ffn=14336, group=128, sigma=0.02)
B70 = dict(hidden=8192, heads=64, kv_heads=8, head_dim=128, ffn=28672, group=128, sigma=0.015)
HEAD8 = dict(hidden=4096, vocab=128256, group=128, sigma=0.02)


def _step(name, shape, layers, cache, rows=1, new=1, **more):
    return dict(name=name, kind="step", layers=layers, cache=cache, rows=rows, new=new, steps=256 if new == 1 else 128,
                ragged=False, beam=False, holes=False, vocab=0, **shape) | more


def listed():
    return [
        # the smallest step there is: launch and barrier latency; token ids in
        _step("tiny-decode", TINY, 2, 72, vocab=512),
        # the whole first stage of an 8B model, chat decoding of one request (a whole model call)
        _step("8b-decode", B8, 16, 72, vocab=128256),
        # the same step fed from host buffers, as every Python driver of the framework calls it
        _step("8b-decode-host", B8, 4, 200, kind="host", vocab=32000),
        # speculative verify: the current token and four drafts; rejected drafts stay masked in the cache
        _step("8b-verify", B8, 4, 512, new=5, holes=True),
        # eight requests of unequal length decoded together, a beam permutation each step
        _step("8b-microbatch", B8, 4, 2048, rows=8, ragged=True, beam=True),
        # continuous batching: sixteen rows on one packed cache row with a mask row each
        _step("8b-packed-16", B8, 4, 1024, new=16, kind="packed"),
        # decoding and verifying at 70B width with a long cache
        _step("70b-decode", B70, 2, 4096),
        _step("70b-verify", B70, 2, 4096, new=5, holes=True),
        # a prompt through the stage
        dict(B8, name="8b-prefill-512", kind="prefill", layers=4, vocab=0, tokens=512, turns=1),
        # a conversation's turns appended to its cache: a ragged token count, the cache growing to 2000 entries
        dict(B8, name="8b-turns-77", kind="prefill", layers=4, vocab=32000, tokens=77, turns=26),
        # the last stage's head: greedy token per row; and the logits of a verify block
        dict(HEAD8, name="8b-top1", kind="top1", rows=1),
        dict(HEAD8, name="8b-logits-5", kind="logits", rows=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["step"] * 4 + ["packed", "host", "prefill", "prefill", "top1", "logits"])
    group = rng.choice([32, 64, 128, 128])
    hidden = _log_int(rng, 256, 8192)
    hidden = max(256, hidden // 128 * 128) if rng.random() < 0.6 else hidden // 8 * 8
    if kind in ("top1", "logits"):
        vocab = min(_log_int(rng, 500, 128256), 525_000_000 // hidden)
        return dict(kind=kind, hidden=hidden, vocab=vocab, group=group, sigma=0.02, rows=rng.randint(1, 16))
    d, kv, G = rng.choice([64, 128, 128]), rng.choice([1, 2, 4, 8, 8]), rng.choice([1, 2, 4, 4, 8])
    c = dict(kind=kind, hidden=hidden, heads=kv * G, kv_heads=kv, head_dim=d, ffn=_log_int(rng, 512, 28672), group=group,
             sigma=1.3 / hidden ** 0.5, vocab=rng.choice([0, _log_int(rng, 500, 32000)]))
    c["layers"] = max(1, min(rng.randint(1, 8), 850_000_000 // _params(c)))
    if kind == "prefill":
        most = max(16, min(1024, int(4e11 / _params(c) / c["layers"])))
        tokens = _log_int(rng, 1, most)
        return dict(c, tokens=tokens, turns=rng.randint(1, max(1, min(16, 2048 // tokens))))
    c.update(rows=1, new=1, ragged=False, beam=False, holes=False, cache=_log_int(rng, 1, 4096))
    if kind == "packed":
        c.update(new=rng.randint(1, 16))
    elif rng.random() < 0.5:
        c.update(rows=rng.randint(2, 16), ragged=rng.random() < 0.7, beam=rng.random() < 0.5, cache=_log_int(rng, 1, 2048))
        c["new"] = rng.randint(1, 16 // c["rows"])
    else:
        c.update(new=rng.randint(1, 16), holes=rng.random() < 0.5)
    return dict(c, steps=256 if c["new"] == 1 else 128)


# --------------------------------------------------------------------------- inputs

NAMES = ("q", "k", "v", "o", "gate", "up", "down")


def _shape(c, name):
    H, dq, dkv, F = c["hidden"], c["heads"] * c["head_dim"], c["kv_heads"] * c["head_dim"], c["ffn"]
    return {"q": (dq, H), "k": (dkv, H), "v": (dkv, H), "o": (H, dq), "gate": (F, H), "up": (F, H), "down": (H, F)}[name]


def _params(c):
    return sum(r * k for r, k in (_shape(c, n) for n in NAMES))


def _gen(seed, *tags):
    g = torch.Generator(device=DEV)
    x = seed & 0x7FFFFFFF
    for t in tags:
        x = (x * 1000003 + t + 12345) & 0x7FFFFFFFFFFF
    return g.manual_seed(x)


def _normal16(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float32).half()


def _bits(t):
    """A half tensor as the binding takes host fp16: uint16 bits."""
    return t.contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def _quantise(rows, cols, group, sigma, g):
    """(codes, zeros) uint8 [rows][cols or groups] and scales fp16: min-max uint4 per row and group."""
    G = -(-cols // group)
    q = torch.empty(rows, cols, dtype=torch.uint8, device=DEV)
    s, z = torch.empty(rows, G, dtype=torch.float16, device=DEV), torch.empty(rows, G, dtype=torch.uint8, device=DEV)
    step = max(1, (1 << 25) // cols)
    for r in range(0, rows, step):
        w = torch.randn(min(step, rows - r), cols, generator=g, device=DEV) * sigma
        n = w.shape[0]
        pad = torch.zeros(n, G * group - cols, device=DEV)
        lo = torch.cat([w, pad + float("inf")], 1).view(n, G, group).amin(2)
        hi = torch.cat([w, pad - float("inf")], 1).view(n, G, group).amax(2)
        sc = ((hi - lo) / 15).half()
        sc[sc == 0] = 1
        zp = torch.round(-lo / sc.float()).clamp(0, 15)
        each = torch.repeat_interleave(torch.stack([sc.float(), zp]), group, 2)[:, :, :cols]
        q[r:r + n] = (torch.round(w / each[0]) + each[1]).clamp(0, 15).to(torch.uint8)
        s[r:r + n], z[r:r + n] = sc, zp.to(torch.uint8)
    return q, s, z


def _nibbles(t):
    if t.shape[1] % 2:
        t = torch.cat([t, t.new_zeros(t.shape[0], 1)], 1)
    return (t[:, 0::2] | (t[:, 1::2] << 4)).contiguous()


def _packed(w):
    q, s, z = w
    return types.SimpleNamespace(codes=_nibbles(q).cpu().numpy(), scales=_bits(s), zeros=_nibbles(z).cpu().numpy())


def _dense(w, group):
    """The dequantised matrix in 64 bits."""
    q, s, z = w
    each = torch.repeat_interleave(torch.stack([s.double(), z.double()]), group, 2)[:, :, :q.shape[1]]
    return (q.double() - each[1]) * each[0]


def _unique(c):
    return min(c["layers"], 2)  # two layers' values, taken in turn (each layer has its own copy on the device)


def _weight(c, seed, layer, i):
    return _quantise(*_shape(c, NAMES[i]), c["group"], c["sigma"], _gen(seed, 1, layer, i))


def _norm(n, seed, *tags):
    return (1 + 0.1 * torch.randn(n, generator=_gen(seed, 2, *tags), device=DEV)).half()


def _embedding(c, seed):
    return _normal16(_gen(seed, 3), c["vocab"], c["hidden"])


def _lens(c):
    """Cache entries of each row when its request begins."""
    if not c["ragged"]:
        return [c["cache"]] * c["rows"]
    r = np.random.RandomState(c["rows"] * 7919 + c["cache"])
    return [int(x) for x in r.randint(max(1, c["cache"] // 16), c["cache"] + 1, c["rows"])]


def _kv(c, seed, layer, row, n):
    g = _gen(seed, 4, layer, row)
    return [_normal16(g, n, c["kv_heads"], c["head_dim"]) for _ in range(2)]


def _inputs(c, seed, count, M):
    """`count` steps' inputs: token ids [count][M] or hidden states [count][M][H]."""
    g = _gen(seed, 5)
    if c.get("vocab") and c["kind"] not in ("top1", "logits"):
        return torch.randint(0, c["vocab"], (count, M), generator=g, device=DEV, dtype=torch.int32), None
    return None, _normal16(g, count, M, c["hidden"])


class _Plan:
    """The host's view of one request batch: per step the positions, masks and beam permutation that a serving loop passes."""

    def __init__(self, c, seed):
        r = np.random.RandomState(seed & 0x7FFFFFFF)
        B, n, T = c["rows"], c["new"], c["steps"]
        lens = _lens(c)
        self.cap = max(lens) + T * n
        self.pos, self.beam = [], None
        if c["kind"] == "packed":  # S slots over one row: a shared prefix, then entries dealt to the slots in turn
            P, S = lens[0], n
            share = P // 2
            owner = np.concatenate([np.full(share, -1), np.arange(self.cap - share) % S])
            owner[P:] = np.arange(self.cap - P) % S
            base = np.array([share + int((owner[:P] == s).sum()) for s in range(S)])
            self.mask = np.zeros((T, S, self.cap), np.uint8)
            for t in range(T):
                end = P + t * S + S
                self.mask[t, :, :end] = (owner[None, :end] == -1) | (owner[None, :end] == np.arange(S)[:, None])
                self.pos.append(base + t)
        else:
            valid = np.ones((B, self.cap), np.uint8)
            length = list(lens)
            if c["holes"]:
                for b in range(B):
                    valid[b, :lens[b]] = r.rand(lens[b]) < 0.85
                    valid[b, :1] = 1
            logical = [int(valid[b, :lens[b]].sum()) for b in range(B)]
            masks, beams = [], []
            for t in range(T):
                if c["beam"]:
                    perm = r.permutation(B).astype(np.int32)
                    beams.append(perm)
                    length, logical = [length[p] for p in perm], [logical[p] for p in perm]
                masks.append(valid.copy() if c["holes"] else valid)
                self.pos.append(np.concatenate([logical[b] + np.arange(n) for b in range(B)]))
                for b in range(B):
                    kept = n
                    if c["holes"] and n > 1:  # accepted drafts: leading successes of Bernoulli(0.6)
                        kept = 1 + int(np.cumprod(r.rand(n - 1) < 0.6).sum())
                        valid[b, length[b] + kept:length[b] + n] = 0
                    length[b] += n
                    logical[b] += kept
            self.mask = np.stack(masks) if c["holes"] else valid[None]
            self.beam = np.stack(beams) if c["beam"] else None
        self.pos = np.stack(self.pos).astype(np.int32)
        self.lens = lens


class _State:
    shard = head = None

    def __del__(self):
        try:
            if self.shard:
                pkg.shard_destroy(self.shard)  # with its kv states
            if self.head:
                pkg.head_destroy(self.head)
        except Exception:
            pass


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _make_shard(c, seed, max_position):
    layers = []
    for l in range(_unique(c)):
        layers.append(types.SimpleNamespace(matrices=[_packed(_weight(c, seed, l, i)) for i in range(7)],
                                            attn_norm=_bits(_norm(c["hidden"], seed, l, 0)), ffn_norm=_bits(_norm(c["hidden"], seed, l, 1))))
    cfg = pkg.shard_config(c["layers"], c["hidden"], c["heads"], c["kv_heads"], c["head_dim"], c["ffn"], c["group"], c["vocab"],
                           max_position, 0, EPS, THETA)
    emb = _bits(_embedding(c, seed)) if c["vocab"] else None
    return pkg.shard_create(cfg, [layers[l % len(layers)] for l in range(c["layers"])], emb)


def _load(s, kv):
    """A new request's captured prefix into a kv state."""
    pkg.kv_state_reset(kv, -1)
    for b, n in enumerate(s.plan.lens):
        for l in range(s.case["layers"]):
            pkg.kv_state_load(kv, b, l, *s.prefix[b][l % len(s.prefix[b])])


def prepare(case, seed):
    c, s = case, _State()
    s.case, s.t = c, 0
    if c["kind"] in ("top1", "logits"):
        w = _packed(_quantise(c["vocab"], c["hidden"], c["group"], c["sigma"], _gen(seed, 1)))
        s.head = pkg.head_create(c["hidden"], c["vocab"], c["group"], EPS, w, _bits(_norm(c["hidden"], seed)))
        _, s.hid = _inputs(c, seed, 8, c["rows"])
        s.tok = torch.empty(c["rows"], dtype=torch.int32, device=DEV)
        s.p = torch.empty(c["rows"], dtype=torch.float32, device=DEV)
        s.logits = torch.empty(c["rows"], c["vocab"] if c["kind"] == "logits" else 1, dtype=torch.float32, device=DEV)
        return s
    if c["kind"] == "prefill":
        S, total = c["tokens"], c["tokens"] * c["turns"]
        s.shard = _make_shard(c, seed, total)
        s.rows = 8  # conversations under way; the rows are handed out anew when all have ended
        s.kv = pkg.kv_state_alloc(s.shard, s.rows, total)
        s.ids, s.hid = _inputs(c, seed, s.rows * c["turns"] if c["vocab"] else 8, S)
        s.pos = torch.arange(total, dtype=torch.int32, device=DEV)
        s.mask = torch.ones(total, dtype=torch.uint8, device=DEV)
        s.out = torch.empty(S, c["hidden"], dtype=torch.float16, device=DEV)
        return s
    plan = s.plan = _Plan(c, seed)
    M, T = c["rows"] * c["new"], c["steps"]
    s.shard = _make_shard(c, seed, int(plan.pos.max()) + 1)
    s.prefix = [[[_bits(x) for x in _kv(c, seed, l, b, n)] for l in range(_unique(c))] for b, n in enumerate(plan.lens)]
    # requests waiting with their prompts cached, a few hundred MB of them at most
    per = c["layers"] * c["rows"] * plan.cap * c["kv_heads"] * c["head_dim"] * 4
    loads = c["layers"] * sum(plan.lens) * c["kv_heads"] * c["head_dim"] * 4
    s.kvs = [pkg.kv_state_alloc(s.shard, c["rows"], plan.cap) for _ in range(max(1, min(16, 600_000_000 // per, 300_000_000 // loads)))]
    for kv in s.kvs:
        _load(s, kv)
    s.n_new, s.turn = [c["new"]] * c["rows"], 0
    if c["kind"] == "host":
        ids, hid = _inputs(c, seed, T, M)
        s.ids = None if ids is None else ids.cpu().numpy()
        s.hid = None if hid is None else _bits(hid)
        s.out = np.empty((M, c["hidden"]), np.uint16)
        return s
    s.ids, s.hid = _inputs(c, seed, T if c["vocab"] else 8, M)
    s.pos, s.mask = _dev(plan.pos), _dev(plan.mask)
    s.beam = None if plan.beam is None else _dev(plan.beam)
    s.out = torch.empty(M, c["hidden"], dtype=torch.float16, device=DEV)
    return s


# --------------------------------------------------------------------------- one pass

def _at(x, t):
    """The address of step t's slice."""
    return None if x is None else x.data_ptr() + t % x.shape[0] * x.stride(0) * x.element_size()


def run(s):
    c, kind = s.case, s.case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "top1":
        pkg.head_top1(s.head, _at(s.hid, s.t), c["rows"], s.tok.data_ptr(), s.p.data_ptr(), stream)
        s.t += 1
        return s.tok, s.p
    if kind == "logits":
        pkg.head_debug_logits(s.head, _at(s.hid, s.t), c["rows"], s.logits.data_ptr(), c["vocab"], stream)
        s.t += 1
        return s.logits
    if kind == "prefill":
        row, turn = divmod(s.t % (s.rows * c["turns"]), c["turns"])
        if s.t and row == 0 and turn == 0:
            pkg.kv_state_reset(s.kv, -1)
        P, S = turn * c["tokens"], c["tokens"]
        pkg.shard_prefill(s.shard, s.kv, row, _at(s.hid, s.t), _at(s.ids, s.t), S, _at(s.pos, P), s.mask.data_ptr(), P + S,
                          s.out.data_ptr(), stream)
        s.t += 1
        return s.out
    if s.t == c["steps"]:  # the request has ended: the next one, loaded anew once all have been used
        s.t, s.turn = 0, s.turn + 1
        if s.turn >= len(s.kvs):
            _load(s, s.kvs[s.turn % len(s.kvs)])
    t, kv = s.t, s.kvs[s.turn % len(s.kvs)]
    s.t += 1
    if kind == "packed":
        pkg.shard_step_packed(s.shard, kv, _at(s.hid, t), _at(s.ids, t), c["new"], _at(s.pos, t), _at(s.mask, t), s.plan.cap,
                              s.out.data_ptr(), stream)
        return s.out
    if kind == "host":
        end = max(s.plan.lens) + (t + 1) * c["new"]
        mask = s.plan.mask[t % len(s.plan.mask)][:, :end]
        pkg.shard_step_host(s.shard, kv, None if s.hid is None else s.hid[t], None if s.ids is None else s.ids[t], s.n_new,
                            s.plan.pos[t], mask, None if s.plan.beam is None else s.plan.beam[t], s.out, stream)
        return s.out.view(np.float16)
    pkg.shard_step(s.shard, kv, _at(s.hid, t), _at(s.ids, t), s.n_new, _at(s.pos, t), _at(s.mask, t), s.plan.cap, _at(s.beam, t),
                   s.out.data_ptr(), stream)
    return s.out


# --------------------------------------------------------------------------- what it costs, and what it gives

def _packed_bytes(rows, cols, group):
    G = -(-cols // group)
    return rows * (-(-cols // 2) + 2 * G + -(-G // 2))


def work(c):
    """Each packed weight, each visible cache entry and each input read once; the outputs and the new cache entries written once."""
    H = c["hidden"]
    if c["kind"] in ("top1", "logits"):
        V, M = c["vocab"], c["rows"]
        return {"bytes": _packed_bytes(V, H, c["group"]) + 2 * H + 2 * M * H + (8 * M if c["kind"] == "top1" else 4 * M * V),
                "flops": 2 * V * H * M}
    if c["kind"] == "prefill":
        M, rows = c["tokens"], [((c["turns"] - 1) * c["tokens"] / 2, c["tokens"])]  # the mean over a conversation
    else:
        M, rows = c["rows"] * c["new"], [(n + (c["steps"] - 1) * c["new"] / 2, c["new"]) for n in _lens(c)]
    visible = 0.8 if c.get("holes") else 1.0  # the plan's masked share of the cache
    weights = c["layers"] * (sum(_packed_bytes(*_shape(c, n), c["group"]) for n in NAMES) + 4 * H)
    kv = c["layers"] * 4 * c["kv_heads"] * c["head_dim"]
    seen = sum(P * visible for P, n in rows)
    if c["kind"] == "packed":  # a slot sees the prefix and its own share of the rest
        P = _lens(c)[0]
        pairs = sum(n * (P // 2) + (p - P // 2) + n for p, n in rows)
    else:
        pairs = sum(n * P * visible + n * (n + 1) / 2 for P, n in rows)
    return {"bytes": weights + kv * (seen + M) + 4 * M * H + 4 * M + int(seen),
            "flops": 2 * c["layers"] * _params(c) * M + 4 * c["layers"] * c["heads"] * c["head_dim"] * pairs}


def tolerance(c):
    """Measured against the same arithmetic in 64 bits with the same fp16 roundings (activations between projections, new cache
    entries).  A step or prefill is 2e-4 to 4e-4 off per layer, growing with the root of the depth (largest value 2e-3), since
    another order of sums moves single fp16 roundings and each moves what follows; the head's only rounding is its normalised
    input, and its logits are 4e-6 off (largest value 4e-5), before any such move."""
    if c["kind"] in ("top1", "logits"):
        return {"rel": 4e-5, "max": 4e-4, "differ": 0.0}
    return {"rel": 8e-4 * c["layers"] ** 0.5, "max": 4e-3 * c["layers"] ** 0.5}


def _round(x, rounded):
    return x.half().double() if rounded else x


def _rms(x, w, rounded):
    return _round(x * torch.rsqrt((x * x).mean(-1, keepdim=True) + EPS) * w.double(), rounded)


def _rope(x, pos, d):
    """x [M][heads][d], pairs (i, i + d / 2)."""
    f = THETA ** (-2.0 * torch.arange(d // 2, dtype=torch.float64, device=DEV) / d)
    a = pos.double()[:, None, None] * f
    lo, hi = x[..., :d // 2], x[..., d // 2:]
    return torch.cat([lo * a.cos() - hi * a.sin(), hi * a.cos() + lo * a.sin()], -1)


def _attend(q, k, v, see):
    """q [n][heads][d] over k, v [entries][kv_heads][d]; see [n][entries]."""
    n, heads, d = q.shape
    G = heads // k.shape[1]
    out = torch.empty_like(q)
    for h in range(heads):
        sc = (q[:, h] @ k[:, h // G].T) / d ** 0.5
        out[:, h] = torch.softmax(sc.masked_fill(~see, float("-inf")), -1) @ v[:, h // G]
    return out.reshape(n, heads * d)


def exact(case, seed, rounded=False):
    """The first pass in 64 bits (rounded=True: with the path's fp16 roundings of activations and new cache entries)."""
    c = case
    if c["kind"] in ("top1", "logits"):
        x = _rms(_inputs(c, seed, 8, c["rows"])[1][0].double(), _norm(c["hidden"], seed), rounded)
        w = _quantise(c["vocab"], c["hidden"], c["group"], c["sigma"], _gen(seed, 1))
        step = max(1, (1 << 27) // c["hidden"])
        y = torch.cat([x @ _dense([t[r:r + step] for t in w], c["group"]).T for r in range(0, c["vocab"], step)], 1)
        return y if c["kind"] == "logits" else (None, torch.softmax(y, -1).amax(-1))
    d, dq, dkv = c["head_dim"], c["heads"] * c["head_dim"], c["kv_heads"] * c["head_dim"]
    if c["kind"] == "prefill":
        S = c["tokens"]
        pos, beam, new = torch.arange(S, device=DEV), [0], S
        ids, hid = _inputs(c, seed, 8 * c["turns"] if c["vocab"] else 8, S)
        past, sees = [None], [torch.ones(S, S, device=DEV).tril().bool()]
    else:
        plan, new = _Plan(c, seed), c["new"]
        M = c["rows"] * new
        ids, hid = _inputs(c, seed, c["steps"] if c["vocab"] or c["kind"] == "host" else 8, M)
        pos = _dev(plan.pos[0])
        beam = plan.beam[0].tolist() if plan.beam is not None else list(range(c["rows"]))
        sees = []
        for b, src in enumerate(beam):
            n = plan.lens[src] + new
            m = plan.mask[0] if c["kind"] == "packed" else plan.mask[0][b:b + 1]
            see = _dev(m[:, :n]).bool().expand(new, n).clone()
            if c["kind"] != "packed":
                see &= torch.arange(n, device=DEV)[None] <= plan.lens[src] + torch.arange(new, device=DEV)[:, None]
            sees.append(see)
    x = (_embedding(c, seed)[ids[0].long()] if c["vocab"] else hid[0]).double()
    for l in range(c["layers"]):
        u = l % _unique(c)
        mat = lambda i: _dense(_weight(c, seed, u, i), c["group"]).T  # noqa: E731
        a = _rms(x, _norm(c["hidden"], seed, u, 0), rounded)
        q = _rope((a @ mat(0)).view(-1, c["heads"], d), pos, d)
        k = _round(_rope((a @ mat(1)).view(-1, c["kv_heads"], d), pos, d), rounded)
        v = _round((a @ mat(2)).view(-1, c["kv_heads"], d), rounded)
        o = []
        for b, src in enumerate(beam):
            at = slice(b * new, (b + 1) * new)
            kk, vv = k[at], v[at]
            if c["kind"] != "prefill":
                pk, pv = _kv(c, seed, u, src, plan.lens[src])
                kk, vv = torch.cat([pk.double(), kk]), torch.cat([pv.double(), vv])
            o.append(_attend(q[at], kk, vv, sees[b]))
        x = x + _round(torch.cat(o), rounded) @ mat(3)
        a = _rms(x, _norm(c["hidden"], seed, u, 1), rounded)
        g = a @ mat(4)
        x = x + _round(g * torch.sigmoid(g) * (a @ mat(5)), rounded) @ mat(6)
    return x
