"""The work that programs give this library, as cases to be timed: content-addressing the
KV-cache fragments that agents deliver, merging replicas and rendering the merged cache,
from a merge of a few dozen tokens to the Qwen3-4B-shaped one of 16,384 and a group of
serving requests. Every case goes through the package's public entry points.

A case names its kind (what the program does), the cache shape (layers, kv heads, head_dim)
and the fragments' lengths ("37,53"; of a serving group: "37,53;12" by request).
`messages` is the delivery schedule by fragment index: an index that returns is a re-sent
copy, in a buffer of its own, as a replica receives it.
"""
import numpy as np
import torch

import paper_2607_01308_gb300 as cm

ROPE_THETA = 1.0e6

# One context per option set for the life of the process, as a serving process keeps it.
_contexts = {}


def _context(dedup=False, overlap=False):
    key = (dedup, overlap)
    if key not in _contexts:
        ctx = cm.Context(0, ROPE_THETA)
        if dedup:
            cm.cm_context_set_dedup_by_bytes(ctx.handle, True)
        if overlap:
            cm.cm_context_set_render_warps(ctx.handle, 8)
        _contexts[key] = ctx
    return _contexts[key]


def listed():
    return [
        # The smallest merge: two short thoughts of a small model, one of them re-sent.
        # Launches and latency are all of it.
        {"name": "merge_tiny", "kind": "merge", "layers": 4, "heads": 2, "dim": 64,
         "lengths": "37,53", "messages": "0,1,0"},
        # Two agents' 512-token thoughts on the Qwen3-1.7B shape, one replica each.
        {"name": "merge_17b_2x512", "kind": "merge", "layers": 28, "heads": 8, "dim": 128,
         "lengths": "512,512", "messages": "0,1"},
        # Five thinkers of ragged lengths, eight messages of which three are re-sent copies.
        {"name": "merge_17b_arity", "kind": "merge", "layers": 28, "heads": 8, "dim": 128,
         "lengths": "421,1789,1430,1042,1417", "messages": "3,1,0,4,1,2,0,3"},
        # The repository's benchmark: four 4096-token fragments on the Qwen3-4B shape.
        {"name": "merge_4b_4x4096", "kind": "merge", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "4096,4096,4096,4096", "messages": "0,1,2,3"},
        # A replica takes one message in: an ordinary thought of odd length.
        {"name": "ingest_4b_1021", "kind": "ingest", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "1021", "messages": "0"},
        # A serving engine without free device memory addresses a short fragment.
        {"name": "address_17b_200", "kind": "address", "layers": 28, "heads": 8, "dim": 128,
         "lengths": "200", "messages": "0"},
        # BagMerge of three fragments of a small model (head_dim 64, odd lengths), in the
        # caller's order: a small render.
        {"name": "bag_d64_3x300", "kind": "bag", "layers": 16, "heads": 4, "dim": 64,
         "lengths": "300,333,271", "messages": "0,1,2"},
        # A replica that holds its fragments renders its state: the largest single render.
        {"name": "render_4b_4x4096", "kind": "render", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "4096,4096,4096,4096", "messages": "0,1,2,3"},
        # The same into a paged KV cache (16-token blocks, shuffled table), ragged lengths.
        {"name": "paged_4b_ragged", "kind": "paged", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "1531,2777,900", "messages": "0,1,2", "block": 16},
        # One more thought arrives at a state that is rendered already.
        {"name": "append_4b", "kind": "append", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "2048,1500,777,1024", "messages": "0,1,2,3"},
        # A group of eight serving requests, three fragments each, some messages re-sent.
        {"name": "serve_4b_8x3", "kind": "serve", "layers": 36, "heads": 8, "dim": 128,
         "lengths": "828,3286,1855;2871,640,3998;1243,2210,517;3522,1116,2047;"
                    "705,1932,2680;3071,595,1404;2266,3777,961;1698,1350,3103",
         "messages": "2,0,1;0,1,2;1,2,0,1;2,1,0;0,2,1;1,0,2,2;0,1,2;2,0,1", "overlap": False},
        # Gossip: every fragment arrives three times, the byte comparison is on.
        {"name": "gossip_17b_3x3", "kind": "gossip", "layers": 28, "heads": 8, "dim": 128,
         "lengths": "1024,700,512", "messages": "0,2,1,1,0,2,2,0,1"},
    ]


_SHAPES = [(28, 8, 128), (36, 8, 128), (16, 4, 64), (24, 4, 256), (12, 12, 64), (8, 2, 32)]


def draw(rng):
    kind = rng.choice(["merge", "merge", "merge", "ingest", "address", "bag", "render", "paged",
                       "append", "serve", "gossip"])
    layers, heads, dim = rng.choice(_SHAPES)

    def length(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    def schedule(n, p):
        msgs = list(range(n)) + [i for i in range(n) if rng.random() < p]
        rng.shuffle(msgs)
        return ",".join(str(m) for m in msgs)

    case = {"kind": kind, "layers": layers, "heads": heads, "dim": dim}
    if kind == "serve":
        # the shapes that are served, one or two groups' worth of requests
        layers, heads, dim = rng.choice(_SHAPES[:2])
        case.update(layers=layers, heads=heads, dim=dim, overlap=rng.random() < 0.5)
        requests, groups, messages = rng.randint(2, 8), [], []
        for _ in range(requests):
            groups.append(",".join(str(length(512, 3200)) for _ in range(3)))
            messages.append(schedule(3, 0.1))
        case.update(lengths=";".join(groups), messages=";".join(messages))
        return case
    n = {"ingest": 1, "address": 1, "append": rng.randint(2, 4)}.get(kind) or rng.randint(2, 5)
    # one scale per case, from a few tokens to the largest, the lengths ragged around it
    top = length(24, 3600 if kind != "address" else 1800)
    lengths = [max(1, int(top * rng.uniform(0.4, 1.0))) for _ in range(n)]
    case["lengths"] = ",".join(str(t) for t in lengths)
    p = {"merge": 0.3, "gossip": 1.0}.get(kind, 0.0)
    case["messages"] = schedule(n, p)
    if kind == "paged":
        case["block"] = rng.choice([16, 16, 32, 64, 8, 24])
    return case


# ---------------------------------------------------------------- inputs

def _ints(text):
    return [int(x) for x in text.split(",")]


def _fragment(case, seed, T):
    """K and V [layers, heads, T, dim]: standard normal times a per-fragment scale, bf16. (A
    key rotated to its position stays standard normal, so K is drawn as it is stored.)"""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    scale = 0.5 + torch.rand((), generator=gen, device="cuda")
    out = []
    for _ in range(2):
        x = torch.empty((case["layers"], case["heads"], T, case["dim"]), dtype=torch.bfloat16,
                        device="cuda")
        step = max(1, (1 << 26) // max(1, x[0].numel()))
        for l in range(0, case["layers"], step):
            part = x[l:l + step]
            part.copy_(torch.randn(part.shape, generator=gen, device="cuda") * scale)
        out.append(x)
    return tuple(out)


def _requests(case, seed):
    """[(distinct fragments, messages)] of each request; a re-sent message is a copy."""
    got = []
    lengths, messages = case["lengths"].split(";"), case["messages"].split(";")
    for r in range(len(lengths)):
        frags = [_fragment(case, seed * 1009 + 101 * r + i, T) for i, T in enumerate(_ints(lengths[r]))]
        seen, msgs = set(), []
        for i in _ints(messages[r]):
            msgs.append(frags[i] if i not in seen else tuple(x.clone() for x in frags[i]))
            seen.add(i)
        got.append((frags, msgs))
    return got


def _cache(case, tokens):
    shape = (case["layers"], case["heads"], tokens, case["dim"])
    return torch.zeros(shape, dtype=torch.bfloat16, device="cuda"), torch.zeros(shape, dtype=torch.bfloat16, device="cuda")


def _table(case, seed, tokens):
    """Logical block -> physical block, shuffled over a pool with some blocks to spare."""
    blocks = -(-tokens // case["block"])
    return np.random.RandomState(seed % (1 << 31)).permutation(blocks + 5)[:blocks].astype(np.int32)


def prepare(case, seed):
    kind = case["kind"]
    reqs = _requests(case, seed)
    frags, msgs = reqs[0]
    tokens = sum(K.shape[2] for K, _ in frags)
    s = {"case": case, "kind": kind, "msgs": msgs, "ctx": _context(kind == "gossip", bool(case.get("overlap")))}
    if kind in ("merge", "gossip", "bag", "render", "append"):
        s["k"], s["v"] = _cache(case, tokens)
    if kind == "merge":
        s["desc"] = [cm.fragment_from_tensors(K, V) for K, V in msgs]
    elif kind == "address":
        s["desc"] = cm.fragment_from_tensors(*msgs[0])
        s["id"] = torch.zeros(16, dtype=torch.uint8, device="cuda")
        s["key"] = torch.zeros(tokens, dtype=torch.int64, device="cuda")
    elif kind in ("render", "paged"):
        s["set"] = cm.FragmentSet(s["ctx"])
        s["set"].ingest_batch(msgs)
        if kind == "paged":
            table = _table(case, seed, tokens)
            pool = (case["layers"], len(table) + 5, case["block"], case["heads"], case["dim"])
            s["k"] = torch.zeros(pool, dtype=torch.bfloat16, device="cuda")
            s["v"] = torch.zeros(pool, dtype=torch.bfloat16, device="cuda")
            s["table"] = torch.from_numpy(table).cuda()
            s["paged"] = cm.cm_paged_cache(
                s["k"].data_ptr(), s["v"].data_ptr(), s["table"].data_ptr(), len(table), case["block"],
                s["k"].stride(1), s["k"].stride(0), s["k"].stride(3), s["k"].stride(2))
    elif kind == "append":
        # the state before the last message, rendered
        s["base"] = cm.FragmentSet(s["ctx"])
        s["base"].ingest_batch(msgs[:-1])
        s["order"] = s["base"].render(s["k"], s["v"])[1]
    elif kind == "serve":
        s["requests"] = [m for _, m in reqs]
        s["caches"] = [_cache(case, sum(K.shape[2] for K, _ in f)) for f, _ in reqs]
        if case["overlap"]:
            s["streams"] = (torch.cuda.Stream(), torch.cuda.Stream())
    return s


# ---------------------------------------------------------------- one pass

def _ids(ids):
    return np.frombuffer(b"".join(ids), dtype=np.uint8).reshape(len(ids), 16)


def _serve(s):
    """Every request's messages into a set of its own, then every set into its cache. With
    overlap, half of the requests at a time: one half renders while the next is ingested."""
    ctx, requests, caches = s["ctx"], s["requests"], s["caches"]
    sets = [cm.FragmentSet(ctx) for _ in requests]
    results = []
    if "streams" not in s:
        results += cm.ingest_many([(S, K, V) for S, msgs in zip(sets, requests) for K, V in msgs])
        lengths = cm.render_many([(S, k, v) for S, (k, v) in zip(sets, caches)])
        return sets, results, lengths
    hashing, rendering = s["streams"]
    current = torch.cuda.current_stream()
    hashing.wait_stream(current)
    rendering.wait_stream(current)
    lengths, half = [], (len(requests) + 1) // 2
    for g in range(0, len(requests), half):
        part = slice(g, g + half)
        results += cm.ingest_many([(S, K, V) for S, msgs in zip(sets[part], requests[part]) for K, V in msgs],
                                  stream=hashing)
        lengths += cm.render_many([(S, k, v) for S, (k, v) in zip(sets[part], caches[part])],
                                  stream=rendering)
    current.wait_stream(rendering)
    return sets, results, lengths


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "merge":
        # two replicas take the messages in turn; their union is rendered
        A, B = cm.FragmentSet(ctx), cm.FragmentSet(ctx)
        half = (len(s["desc"]) + 1) // 2
        where = [A.handle] * half + [B.handle] * (len(s["desc"]) - half)
        got, n, order, _ = cm.cm_ingest_render(where, s["desc"], A.handle, s["k"].data_ptr(),
                                               s["v"].data_ptr(), s["k"].shape[2])
        return {"ids": _ids([i for i, _ in got]), "absorbed": [a for _, a in got], "tokens": n,
                "order": _ids(order), "k": s["k"], "v": s["v"]}
    if kind == "ingest":
        S = cm.FragmentSet(ctx)
        fid, absorbed = S.ingest(*s["msgs"][0])
        return {"ids": _ids([fid]), "absorbed": [absorbed]}
    if kind == "address":
        cm.cm_fragment_id_static(s["desc"], s["id"].data_ptr(), s["key"].data_ptr())
        return {"id": s["id"], "key": s["key"]}
    if kind == "bag":
        n = ctx.bagmerge(s["msgs"], s["k"], s["v"])
        return {"tokens": n, "k": s["k"], "v": s["v"]}
    if kind == "render":
        n, order = s["set"].render(s["k"], s["v"])
        return {"tokens": n, "order": _ids(order), "k": s["k"], "v": s["v"]}
    if kind == "paged":
        n, order = cm.cm_render_paged(s["set"].handle, s["paged"])
        return {"tokens": n, "order": _ids(order), "k": s["k"], "v": s["v"]}
    if kind == "append":
        S = cm.FragmentSet(ctx)
        S.union(s["base"])
        fid, absorbed = S.ingest(*s["msgs"][-1])
        n, order, kept = S.render_incremental(s["k"], s["v"], s["order"])
        return {"ids": _ids([fid]), "absorbed": [absorbed], "tokens": n, "kept": kept,
                "order": _ids(order), "k": s["k"], "v": s["v"]}
    if kind == "gossip":
        S = cm.FragmentSet(ctx)
        got = S.ingest_batch(s["msgs"])
        n, order = S.render(s["k"], s["v"])
        return {"ids": _ids([i for i, _ in got]), "absorbed": [a for _, a in got], "tokens": n,
                "order": _ids(order), "k": s["k"], "v": s["v"]}
    _, got, lengths = _serve(s)
    return {"ids": _ids([i for i, _ in got]), "absorbed": [a for _, a in got], "tokens": lengths,
            "k": [k for k, _ in s["caches"]], "v": [v for _, v in s["caches"]]}


# ---------------------------------------------------------------- what a pass needs

def work(case):
    """Bytes: every message's K and V read once, every rendered token's K and V written
    once. Flops: three per element of a rotated key (the hash is integer work)."""
    row = case["layers"] * case["heads"] * case["dim"]
    token = 2 * row * 2
    lengths = [_ints(t) for t in case["lengths"].split(";")]
    messages = [_ints(t) for t in case["messages"].split(";")]
    read = sum(lens[i] for lens, msgs in zip(lengths, messages) for i in msgs)
    written = sum(sum(lens) for lens in lengths)
    if case["kind"] in ("ingest", "address"):
        return {"bytes": read * token, "flops": 2 * lengths[0][0] * case["heads"] * case["dim"]}
    return {"bytes": (read + written) * token, "flops": 3 * written * row}


def tolerance(case):
    """Ids, orders, V and the key's norms are whole values. A rotated key is the fp64
    rotation rounded once to bf16, which leaves one right answer."""
    return "exact"


# ---------------------------------------------------------------- the 64-bit answer

def _norm_key(K):
    """Q[t] of the middle layer: over heads, the sum of round(2^20 |K|) with the squares
    summed in element order."""
    x = K[K.shape[0] // 2].double()
    ss = torch.zeros(x.shape[:2], dtype=torch.float64, device=x.device)
    for j in range(x.shape[2]):
        ss += x[:, :, j] * x[:, :, j]
    return torch.round(torch.sqrt(ss) * 1048576.0).to(torch.int64).sum(dim=0)


def _ordered(frags):
    keys = [_norm_key(K) for K, _ in frags]
    tail = min(len(q) for q in keys)
    sums = [int(q[len(q) - tail:].sum()) for q in keys]
    return [frags[i] for i in sorted(range(len(frags)), key=lambda i: -sums[i])]


def _merged(case, frags):
    """The fragments one after another, each K rotated by its offset (rotate-half pairs)."""
    tokens, half = sum(K.shape[2] for K, _ in frags), case["dim"] // 2
    shape = (case["layers"], case["heads"], tokens, case["dim"])
    k = torch.empty(shape, dtype=torch.float64, device="cuda")
    v = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    at = 0
    omega = torch.tensor([ROPE_THETA ** (-2.0 * j / case["dim"]) for j in range(half)],
                         dtype=torch.float64, device="cuda")
    for K, V in frags:
        T = K.shape[2]
        v[:, :, at:at + T] = V
        cos, sin = torch.cos(at * omega), torch.sin(at * omega)
        for l in range(case["layers"]):
            x, y = K[l, :, :, :half].double(), K[l, :, :, half:].double()
            k[l, :, at:at + T, :half] = x * cos - y * sin
            k[l, :, at:at + T, half:] = y * cos + x * sin
        at += T
    return k, v


def exact(case, seed):
    kind = case["kind"]
    reqs = _requests(case, seed)
    frags = reqs[0][0]
    if kind == "ingest":
        return None   # an id and a flag: nothing to round
    if kind == "address":
        return {"id": None, "key": _norm_key(frags[0][0])}
    if kind == "serve":
        merged = [_merged(case, _ordered(f)) for f, _ in reqs]
        return {"ids": None, "absorbed": None, "tokens": [k.shape[2] for k, _ in merged],
                "k": [k for k, _ in merged], "v": [v for _, v in merged]}
    k, v = _merged(case, [m for m in reqs[0][1]] if kind == "bag" else _ordered(frags))
    got = {"tokens": k.shape[2], "k": k, "v": v}
    if kind == "paged":
        table = _table(case, seed, k.shape[2])
        for name in ("k", "v"):
            flat = got[name]
            L, H, n, d = flat.shape
            pool = torch.zeros((L, len(table) + 5, case["block"], H, d), dtype=flat.dtype, device="cuda")
            for b, phys in enumerate(table.tolist()):
                part = flat[:, :, b * case["block"]:(b + 1) * case["block"]]
                pool[:, phys, :part.shape[2]] = part.transpose(1, 2)
            got[name] = pool
    return got
