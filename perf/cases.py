"""What this framework is asked to do, as cases that can be timed and compared.

Every case goes through the public Python entry points (`Pool` and
`st_harvest`), as a serving program would call them:

decode    a decode of every branch of one or more fork groups (and of unforked
          sequences beside them), the prefix KV already in the pool
turn      one agent turn: fork the branches off the context, decode a few
          tokens on each, harvest the branches' thoughts, merge their rows
          into the main thread, release the branches
merge     rows (harvested thoughts or an observation) appended to a context
          and prefilled causally
batch     several agents' rows appended and prefilled in one call
prompt    a session is restored (its cached KV appended) and the rest of its
          prompt prefilled

A pass leaves its state as it found it: what a case appends, it appends to
sequences that it forks or creates in the pass and releases again.  Sizes are
those of the workloads in `workloads/configs.py` and of `bench.py` (with fewer
layers where a whole model's KV would fill the card), or generic ones.
"""
import math

import torch

import paper_2608_13667_gb300 as st

PAGE = 16
OPEN, CLOSE = 7, 8  # the thought tags' token ids
GEOMETRY = {"8/2x64": (8, 2, 64), "32/8x128": (32, 8, 128), "64/8x128": (64, 8, 128), "32/8x64": (32, 8, 64)}


def listed():
    return [
        # the smallest call: one layer of a small model, one fork group of 1 + 4
        # branches with ragged suffixes over a short prefix; latency alone counts
        {"name": "decode_tiny", "kind": "decode", "heads": "8/2x64", "layers": 1, "groups": 1, "branches": 5,
         "prefix": 512, "spread": 0.0, "suffix": 64, "singles": 0, "single_len": 0},
        # one agent's turn in one layer, called layer by layer as a model's
        # forward pass does: 8192 tokens of context, 8 tokens on each of 5
        # branches, a harvest of 4 x 2 thoughts, the merge, the releases
        {"name": "turn_one_layer", "kind": "turn", "heads": "32/8x128", "layers": 1, "prefix": 8192, "branches": 5,
         "steps": 8, "atoms": 2, "atom_len": 11},
        # the same with all layers of a 32-layer model in each call, on the
        # context length of a main call in the measured trajectories
        {"name": "turn_all_layers", "kind": "turn", "heads": "32/8x128", "layers": 32, "prefix": 23040,
         "branches": 5, "steps": 2, "atoms": 1, "atom_len": 11},
        # one layer of a server's decode step: 16 agents of 5 branches each,
        # prefixes from 4k to 32k, suffixes up to 1k
        {"name": "decode_serving", "kind": "decode", "heads": "32/8x128", "layers": 1, "groups": 16, "branches": 5,
         "prefix": 18432, "spread": 0.77, "suffix": 1024, "singles": 0, "single_len": 0},
        # fork groups and unforked sequences side by side
        {"name": "decode_mixed", "kind": "decode", "heads": "32/8x128", "layers": 4, "groups": 8, "branches": 5,
         "prefix": 16384, "spread": 0.0, "suffix": 512, "singles": 64, "single_len": 2300},
        # long trajectories: 4 agents, 131072 tokens shared by 1 + 4 branches
        {"name": "decode_long", "kind": "decode", "heads": "64/8x128", "layers": 4, "groups": 4, "branches": 5,
         "prefix": 131072, "spread": 0.0, "suffix": 2048, "singles": 0, "single_len": 0},
        # more reasoning dimensions than the usual four: 12 branches (96 query
        # rows on each shared page)
        {"name": "decode_12_branches", "kind": "decode", "heads": "64/8x128", "layers": 4, "groups": 2, "branches": 12,
         "prefix": 65536, "spread": 0.0, "suffix": 1024, "singles": 0, "single_len": 0},
        # a wide fan-out: 24 branches (192 query rows on each shared page)
        {"name": "decode_24_branches", "kind": "decode", "heads": "64/8x128", "layers": 2, "groups": 2, "branches": 24,
         "prefix": 65536, "spread": 0.0, "suffix": 512, "singles": 0, "single_len": 0},
        # one layer's merge of one turn's thoughts into a main thread
        {"name": "merge_one_layer", "kind": "merge", "heads": "32/8x128", "layers": 1, "context": 23041, "rows": 133},
        # a long observation with the thoughts after it
        {"name": "merge_observation", "kind": "merge", "heads": "32/8x128", "layers": 4, "context": 16896,
         "rows": 2048},
        # 16 agents' observations that arrive together, one layer
        {"name": "batch_serving", "kind": "batch", "heads": "32/8x128", "layers": 1, "agents": 16, "context": 18432,
         "spread": 0.77, "rows": 600, "rows_spread": 0.8},
        # a session restored from its cached KV, then the new part of its prompt
        {"name": "prompt_restored", "kind": "prompt", "heads": "64/8x128", "layers": 4, "cached": 12290,
         "rows": 1021},
    ]


def _log(rng, lo, hi):
    """A whole number, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges; none costs more than the largest listed ones."""
    kind = rng.choice(["decode", "decode", "decode", "turn", "merge", "merge", "batch", "prompt"])
    heads = rng.choice(["8/2x64", "32/8x64", "32/8x128", "32/8x128", "64/8x128", "64/8x128"])
    hq, hkv, d = GEOMETRY[heads]
    row = hkv * d * 4  # bytes of K and V of a token in a layer
    if kind == "decode":
        c = {"kind": kind, "heads": heads, "layers": rng.choice([1, 1, 2, 4, 8]), "groups": _log(rng, 1, 16),
             "branches": rng.choice([2, 3, 4, 5, 5, 5, 5, 6, 7, 8, 9, 11, 13, 16, 20, 27]),
             "prefix": _log(rng, 300, 131072), "spread": round(rng.uniform(0.0, 0.8), 2), "suffix": _log(rng, 4, 2048),
             "singles": rng.choice([0, 0, 0, _log(rng, 1, 48)]), "single_len": _log(rng, 20, 4000)}
        while _decode_tokens(c) * row * c["layers"] > 5e9:
            c["prefix"], c["single_len"] = max(300, int(c["prefix"] * 0.7)), max(20, int(c["single_len"] * 0.7))
            c["suffix"], c["groups"] = max(4, int(c["suffix"] * 0.7)), max(1, c["groups"] - 1)
        return c
    if kind == "turn":
        c = {"kind": kind, "heads": heads, "layers": rng.choice([1, 1, 4, 16]), "prefix": _log(rng, 500, 32768),
             "branches": rng.choice([3, 5, 5, 5, 9]), "steps": rng.randint(2, 8), "atoms": rng.randint(1, 5),
             "atom_len": rng.randint(3, 25)}
        while c["steps"] * c["prefix"] * row * c["layers"] > 5e9:
            c["prefix"] = int(c["prefix"] * 0.8)
        return c
    if kind == "merge":
        c = {"kind": kind, "heads": heads, "layers": rng.choice([1, 1, 2, 4, 8]), "context": _log(rng, 300, 40000),
             "rows": _log(rng, 1, 2048)}
    elif kind == "batch":
        c = {"kind": kind, "heads": heads, "layers": rng.choice([1, 1, 2]), "agents": _log(rng, 2, 16),
             "context": _log(rng, 300, 20000), "spread": round(rng.uniform(0.0, 0.8), 2), "rows": _log(rng, 8, 600),
             "rows_spread": round(rng.uniform(0.0, 0.9), 2)}
    else:
        c = {"kind": kind, "heads": heads, "layers": rng.choice([1, 2, 4, 8]),
             "cached": rng.choice([0, _log(rng, 300, 20000)]), "rows": _log(rng, 16, 4096)}
    size = "rows"
    while work(c)["flops"] > 2.4e12:
        c[size] = max(1, int(c[size] * 0.8))
    return c


# ---- shapes ------------------------------------------------------------------------


def _spread(n, mid, share, salt):
    """n lengths between mid (1 - share) and mid (1 + share), the same on every call."""
    out = []
    for i in range(n):
        x = math.modf(abs(math.sin(12.9898 * (i + 1) + 78.233 * salt) * 43758.5453))[0]
        out.append(max(1, int(round(mid * (1 + share * (2 * x - 1))))))
    return out


def _decode_shape(c):
    """Prefix length per group, suffix lengths per group and branch, lengths of the unforked sequences."""
    prefix = _spread(c["groups"], c["prefix"], c["spread"], 1)
    flat = _spread(c["groups"] * c["branches"], (c["suffix"] + 1) / 2, 1.0, 2)
    suffix = [flat[g * c["branches"]:(g + 1) * c["branches"]] for g in range(c["groups"])]
    return prefix, suffix, _spread(c["singles"], c["single_len"], 0.2, 3)


def _decode_tokens(c):
    prefix, suffix, singles = _decode_shape(c)
    return sum(prefix) + sum(map(sum, suffix)) + sum(singles)


def _batch_shape(c):
    return (_spread(c["agents"], c["context"], c["spread"], 4), _spread(c["agents"], c["rows"], c["rows_spread"], 5))


def _pages(n):
    return n // PAGE + 2


def _pool(c, tokens, longest, seqs, branches):
    """A pool for pieces of `tokens` lengths (pages each), the longest sequence's length, with some room."""
    hq, hkv, d = GEOMETRY[c["heads"]]
    return st.Pool(n_layers=c["layers"], n_q_heads=hq, n_kv_heads=hkv, head_dim=d, seed=11,
                   n_blocks=sum(_pages(n) for n in tokens) + 64, max_seqs=seqs + 4, max_pages=_pages(longest) + 64,
                   max_decode_branches=max(1, branches), max_splits=32 if c["layers"] * branches <= 400 else 16)


# ---- inputs ------------------------------------------------------------------------


class _Draw:
    """Seeded bf16 N(0, 1) values on the GPU (small ones for the smallest model, as in its workload)."""

    def __init__(self, c, seed):
        self.c = c
        self.hq, self.hkv, self.d = GEOMETRY[c["heads"]]
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(int(seed))
        self.scale = 0.125 if c["heads"] == "8/2x64" else 1.0

    def _normal(self, shape):
        out = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
        for l in range(shape[0]):
            x = torch.randn(shape[1:], generator=self.gen, device="cuda")
            out[l].copy_(x.mul_(self.scale) if self.scale != 1.0 else x)
        return out

    def kv(self, n):
        shape = (self.c["layers"], n, self.hkv, self.d)
        return self._normal(shape), self._normal(shape)

    def q(self, n):
        return self._normal((self.c["layers"], n, self.hq, self.d))


def _append(pool, seq, kv):
    k, v = kv
    pool.append_kv([seq], k.unsqueeze(1), v.unsqueeze(1))


def _streams(c, seed):
    """Token ids of each auxiliary branch: `atoms` closed thoughts of `atom_len` tokens between other tokens, and
    an unfinished one at the end."""
    g = torch.Generator()
    g.manual_seed(int(seed) + 1)
    n_aux, gap = c["branches"] - 1, 6
    rows, stride = [], c["atoms"] * (c["atom_len"] + gap) + gap
    for _ in range(n_aux):
        ids = torch.randint(100, 30000, (stride,), generator=g, dtype=torch.int32)
        for a in range(c["atoms"]):
            at = a * (c["atom_len"] + gap) + int(torch.randint(0, gap, (1,), generator=g))
            ids[at], ids[at + c["atom_len"] - 1] = OPEN, CLOSE
        ids[stride - 2] = OPEN
        rows.append(ids)
    return torch.stack(rows)


def _out(c, n):
    hq, _, d = GEOMETRY[c["heads"]]
    return (torch.empty((c["layers"], n, hq, d), dtype=torch.float32, device="cuda"),
            torch.empty((c["layers"], n, hq), dtype=torch.float32, device="cuda"))


def _inputs(c, seed):
    """Everything that a case's state is made of, drawn in a fixed order."""
    x = _Draw(c, seed)
    if c["kind"] == "decode":
        prefix, suffix, singles = _decode_shape(c)
        n = sum(map(len, suffix)) + len(singles)
        return {"q": x.q(n), "prefix": [x.kv(p) for p in prefix],
                "suffix": [[x.kv(s) for s in row] for row in suffix], "singles": [x.kv(s) for s in singles]}
    if c["kind"] == "turn":
        t = (c["branches"] - 1) * c["atoms"] * c["atom_len"]
        return {"prefix": x.kv(c["prefix"]),
                "steps": [(x.kv(c["branches"]), x.q(c["branches"])) for _ in range(c["steps"])],
                "merge": (x.kv(t), x.q(t)), "streams": _streams(c, seed)}
    if c["kind"] == "merge":
        return {"context": x.kv(c["context"]), "rows": (x.kv(c["rows"]), x.q(c["rows"]))}
    if c["kind"] == "batch":
        context, rows = _batch_shape(c)
        return {"context": [x.kv(n) for n in context], "rows": (x.kv(sum(rows)), x.q(sum(rows)))}
    return {"cached": x.kv(c["cached"]) if c["cached"] else None, "rows": (x.kv(c["rows"]), x.q(c["rows"]))}


# ---- the passes --------------------------------------------------------------------


def prepare(case, seed):
    c, i = case, _inputs(case, seed)
    if c["kind"] == "decode":
        prefix, suffix, singles = _decode_shape(c)
        n = i["q"].shape[1]
        pool = _pool(c, prefix + sum(suffix, []) + singles, max(prefix + singles) + c["suffix"], n, n)
        br = []
        for g in range(c["groups"]):
            main = pool.seq_create()
            _append(pool, main, i["prefix"][g])
            group = [main] + pool.fork(main, c["branches"] - 1)
            for seq, kv in zip(group, i["suffix"][g]):
                _append(pool, seq, kv)
            br += group
        for kv in i["singles"]:
            seq = pool.seq_create()
            _append(pool, seq, kv)
            br.append(seq)
        return {"case": c, "pool": pool, "br": br, "q": i["q"], "out": _out(c, n)}
    if c["kind"] == "turn":
        b, t = c["branches"], i["merge"][1].shape[1]
        pool = _pool(c, [c["prefix"]] + [c["steps"]] * b + [t], c["prefix"] + c["steps"] + t, b + 1, b)
        main = pool.seq_create()
        _append(pool, main, i["prefix"])
        streams = i["streams"].cuda()
        lens = torch.full((b - 1,), streams.shape[1], dtype=torch.int32, device="cuda")
        return {"case": c, "pool": pool, "main": main, "streams": streams, "lens": lens,
                "steps": [(k, v, q) + _out(c, b) for (k, v), q in i["steps"]],
                "merge": i["merge"][0] + (i["merge"][1],), "out": _out(c, t)}
    if c["kind"] == "merge":
        pool = _pool(c, [c["context"], c["rows"]], c["context"] + c["rows"], 2, 1)
        main = pool.seq_create()
        _append(pool, main, i["context"])
        return {"case": c, "pool": pool, "main": main, "rows": i["rows"][0] + (i["rows"][1],),
                "out": _out(c, c["rows"])}
    if c["kind"] == "batch":
        context, rows = _batch_shape(c)
        pool = _pool(c, context + rows, max(context) + max(rows), 2 * len(rows), len(rows))
        mains = []
        for kv in i["context"]:
            mains.append(pool.seq_create())
            _append(pool, mains[-1], kv)
        return {"case": c, "pool": pool, "mains": mains, "counts": rows, "rows": i["rows"][0] + (i["rows"][1],),
                "out": _out(c, sum(rows))}
    pool = _pool(c, [c["cached"] + c["rows"]], c["cached"] + c["rows"], 1, 1)
    cached = tuple(x.unsqueeze(1) for x in i["cached"]) if i["cached"] else None
    return {"case": c, "pool": pool, "cached": cached, "rows": i["rows"][0] + (i["rows"][1],),
            "out": _out(c, c["rows"])}


def run(state):
    pool, kind = state["pool"], state["case"]["kind"]
    if kind == "decode":
        o, lse = pool.decode_attn(state["br"], state["q"], *state["out"])
        return {"o": o, "lse": lse}
    if kind == "turn":
        # the first of the forked sequences goes on as the main thread, so that the context itself stays as it is
        br = pool.fork(state["main"], state["case"]["branches"])
        steps = [pool.decode_step(br, k, v, q, o, lse) for k, v, q, o, lse in state["steps"]]
        ids, src, atoms = st.st_harvest(state["streams"], state["lens"], OPEN, CLOSE)
        k, v, q = state["merge"]
        assert ids.shape[0] == q.shape[1]
        merged = pool.merge(br[0], q, k, v, *state["out"])
        for seq in br:
            pool.release(seq)
        return {"steps": [list(x) for x in steps], "ids": ids, "src": src, "atoms": atoms, "merged": list(merged)}
    k, v, q = state["rows"]
    if kind == "merge":
        seq, = pool.fork(state["main"], 1)
        o, lse = pool.merge(seq, q, k, v, *state["out"])
        pool.release(seq)
    elif kind == "batch":
        seqs = [pool.fork(m, 1)[0] for m in state["mains"]]
        o, lse = pool.prefill_batch(seqs, state["counts"], q, k, v, *state["out"])
        for seq in seqs:
            pool.release(seq)
    else:
        seq = pool.seq_create()
        if state["cached"]:
            pool.append_kv([seq], *state["cached"])
        o, lse = pool.merge(seq, q, k, v, *state["out"])
        pool.release(seq)
    return {"o": o, "lse": lse}


# ---- what a pass cannot do without ---------------------------------------------------


def work(case):
    c = case
    hq, hkv, d = GEOMETRY[c["heads"]]
    # bytes of a token's K and V, of a query's Q, O and LSE; operations of a (query, key) pair
    row, query, flop = hkv * d * 4, hq * (6 * d + 4), 4 * d * hq

    def causal(context, rows):
        return rows * context + rows * (rows + 1) // 2

    if c["kind"] == "decode":
        prefix, suffix, singles = _decode_shape(c)
        n = sum(map(len, suffix)) + len(singles)
        keys = sum(len(s) * p + sum(s) for p, s in zip(prefix, suffix)) + sum(singles)
        size, pairs = _decode_tokens(c) * row + n * query, keys
    elif c["kind"] == "turn":
        b, n, p = c["branches"], c["steps"], c["prefix"]
        t = (b - 1) * c["atoms"] * c["atom_len"]
        # a step reads the prefix and the branches' own rows, and reads and writes the new ones
        size = sum(p * row + b * (s + 2) * row + b * query for s in range(n)) + (p + n + 2 * t) * row + t * query
        pairs = sum(b * (p + s + 1) for s in range(n)) + causal(p + n, t)
    elif c["kind"] == "merge":
        size, pairs = (c["context"] + 2 * c["rows"]) * row + c["rows"] * query, causal(c["context"], c["rows"])
    elif c["kind"] == "batch":
        context, rows = _batch_shape(c)
        size = (sum(context) + 2 * sum(rows)) * row + sum(rows) * query
        pairs = sum(causal(n, r) for n, r in zip(context, rows))
    else:
        # the cached rows are read, written and read again by the prefill
        size, pairs = (3 * c["cached"] + 2 * c["rows"]) * row + c["rows"] * query, causal(c["cached"], c["rows"])
    return {"bytes": float(size * c["layers"]), "flops": float(flop * pairs * c["layers"])}


def tolerance(case):
    # fp32 sums whose probabilities are held to about 16 bits (two bf16 terms).
    # Measured against 64 bits: 2e-6 to 6e-6 for a decode, whose sums end at each
    # run of pages; up to 5.4e-5 for the rows of a merge, each of them one sum
    # over the whole context in the tensor cores' accumulator.  About four times
    # that, since another order of the sums moves them as much.
    return {"rel": 2.5e-5} if case["kind"] == "decode" else {"rel": 2e-4}


# ---- in 64 bits ----------------------------------------------------------------------


def _attend(q, k, v, first):
    """q [T][Hq][D] over k, v [n][Hkv][D], query t over the first `first` + t + 1 keys (all of them if None)."""
    t, hq, d = q.shape
    hkv = k.shape[1]
    g = hq // hkv
    o = torch.empty((t, hq, d), dtype=torch.float64, device=q.device)
    lse = torch.empty((t, hq), dtype=torch.float64, device=q.device)
    for h in range(hkv):
        kk, vv = k[:, h].double(), v[:, h].double()
        for t0 in range(0, t, 512):
            t1 = min(t, t0 + 512)
            qq = q[t0:t1, h * g:(h + 1) * g].double().reshape(-1, d)
            s = (qq @ kk.T) / math.sqrt(d)
            if first is not None:
                last = torch.arange(t0, t1, device=q.device).repeat_interleave(g) + first
                s.masked_fill_(torch.arange(k.shape[0], device=q.device)[None, :] > last[:, None], -math.inf)
            z = torch.logsumexp(s, 1)
            o[t0:t1, h * g:(h + 1) * g] = (torch.exp(s - z[:, None]) @ vv).reshape(t1 - t0, g, d)
            lse[t0:t1, h * g:(h + 1) * g] = z.reshape(t1 - t0, g)
    return o, lse


def _layers(c, f):
    got = [f(l) for l in range(c["layers"])]
    return torch.stack([o for o, _ in got]), torch.stack([z for _, z in got])


def _over(parts, l):
    return torch.cat([k[l] for k, _ in parts]), torch.cat([v[l] for _, v in parts])


def exact(case, seed):
    c = case
    if work(c)["flops"] > 6e12:
        return None
    i = _inputs(c, seed)
    if c["kind"] == "decode":
        seqs = [[i["prefix"][g], kv] for g in range(c["groups"]) for kv in i["suffix"][g]]
        seqs += [[kv] for kv in i["singles"]]

        def layer(l):
            got = [_attend(i["q"][l, b:b + 1], *_over(parts, l), None) for b, parts in enumerate(seqs)]
            return torch.cat([o for o, _ in got]), torch.cat([z for _, z in got])

        o, lse = _layers(c, layer)
        return {"o": o, "lse": lse}
    if c["kind"] == "turn":
        n, steps = c["branches"], []
        for s in range(c["steps"]):
            def layer(l):
                pk, pv = (x[l] for x in i["prefix"])
                got = []
                for b in range(n):
                    ks = torch.stack([i["steps"][x][0][0][l, b] for x in range(s + 1)])
                    vs = torch.stack([i["steps"][x][0][1][l, b] for x in range(s + 1)])
                    got.append(_attend(i["steps"][s][1][l, b:b + 1], torch.cat([pk, ks]), torch.cat([pv, vs]), None))
                return torch.cat([o for o, _ in got]), torch.cat([z for _, z in got])
            steps.append(list(_layers(c, layer)))

        def merged(l):
            (mk, mv), q = i["merge"]
            ks = torch.stack([x[0][0][l, 0] for x in i["steps"]])
            vs = torch.stack([x[0][1][l, 0] for x in i["steps"]])
            k, v = torch.cat([i["prefix"][0][l], ks, mk[l]]), torch.cat([i["prefix"][1][l], vs, mv[l]])
            return _attend(q[l], k, v, c["prefix"] + c["steps"])

        return {"steps": steps, "ids": None, "src": None, "atoms": None, "merged": list(_layers(c, merged))}
    kv, q = i["rows"]
    if c["kind"] == "batch":
        context, rows = _batch_shape(c)

        def layer(l):
            got, at = [], 0
            for x, n in zip(i["context"], rows):
                new = tuple(y[:, at:at + n] for y in kv)
                got.append(_attend(q[l, at:at + n], *_over([x, new], l), x[0].shape[1]))
                at += n
            return torch.cat([o for o, _ in got]), torch.cat([z for _, z in got])
    else:
        before = i["context"] if c["kind"] == "merge" else i["cached"]
        first = before[0].shape[1] if before else 0

        def layer(l):
            return _attend(q[l], *_over([before, kv] if before else [kv], l), first)

    o, lse = _layers(c, layer)
    return {"o": o, "lse": lse}
