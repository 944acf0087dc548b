"""Workloads of the string sort, from the smallest calls to the largest.

Each case is one call (or one pass over a kept plan) through the public entry
points of paper_1808_00963_gb300: plain sorts, the allocation-free sort, the
host-buffer sort, sorts with DNA codes, batches, the K-way LCP merge and the
suffix array.  Inputs are generated on the GPU from a seed, with the recipes of
gen/: URL-like strings with Zipf-distributed hosts, random strings, DNA-like
texts and records under one long common prefix.
"""
import math

import torch

import paper_1808_00963_gb300 as ss

DEV = "cuda"


def listed():
    return [
        # the smallest request of the serving trace: a thousand URLs, the caller waits for the answer
        {"name": "url_1k", "op": "sort", "data": "url", "n": 1000, "max_len": 0, "lcp": True, "wait": True},
        # a latency-critical caller that may not allocate: twenty thousand short keys
        {"name": "noalloc_random_20k", "op": "noalloc", "data": "random", "n": 20011, "max_len": 0},
        # 100 000 random keys of 8 to 32 letters (an index build's usual chunk), enqueued without waiting
        {"name": "random_100k", "op": "sort", "data": "random", "n": 100000, "max_len": 0, "lcp": True, "wait": False},
        # a crawl segment of a million URLs, an odd size, the caller waits
        {"name": "url_1m", "op": "sort", "data": "url", "n": 999983, "max_len": 0, "lcp": True, "wait": True},
        # the headline sort: 20 million URLs, 1.19 GB of characters
        {"name": "url_20m", "op": "sort", "data": "url", "n": 20000000, "max_len": 0, "lcp": True, "wait": False},
        # a million records under one 200-character key path, many of them equal; only the order is wanted
        {"name": "prefix200_1m", "op": "sort", "data": "prefix", "n": 1000000, "prefix": 200, "max_len": 0,
         "lcp": False, "wait": False},
        # all suffixes of a 4 M-character DNA-like text with repeats, compared up to 500 characters
        {"name": "dna_4m", "op": "sort", "data": "dna", "n": 4000000, "max_len": 500, "lcp": True, "wait": False},
        # the same kind of suffixes through the 3-bit character codes
        {"name": "dna_codes_4m", "op": "dna", "data": "dna", "n": 4000000, "max_len": 500},
        # the full suffix and LCP arrays of such a text
        {"name": "suffix_array_4m", "op": "suffix_array", "data": "dna", "n": 4000000},
        # 16 sorted runs of a log-structured store compacted into one: 20 million URLs
        {"name": "merge16_url_20m", "op": "merge", "data": "url", "n": 20000000, "runs": 16},
        # a served mix: 512 sets of 100 to 200 000 strings of all kinds as one planned batch
        {"name": "batch_512", "op": "batch", "sets": 512, "smin": 100, "smax": 200000},
        # a caller whose strings live in pinned host memory: two million URLs in, order and LCPs out
        {"name": "host_url_2m", "op": "host", "data": "url", "n": 2000003, "max_len": 0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["sort", "sort", "sort", "sort", "noalloc", "host", "dna", "suffix_array", "merge", "batch"])
    if op == "sort":
        data = rng.choice(["url", "url", "random", "bytes", "binary", "dna", "prefix"])
        top = {"url": 20000000, "random": 10000000, "bytes": 10000000, "binary": 2000000, "dna": 4000000,
               "prefix": 1500000}[data]
        case = {"op": op, "data": data, "n": _log_uniform(rng, 300, top),
                "max_len": 500 if data == "dna" else rng.choice([0, 0, 0, 20]),
                "lcp": rng.random() < 0.8, "wait": rng.random() < 0.5}
        if data == "prefix":
            case["prefix"] = _log_uniform(rng, 12, 300)
        return case
    if op == "noalloc":
        return {"op": op, "data": rng.choice(["url", "random", "bytes"]), "n": _log_uniform(rng, 300, 65536),
                "max_len": 0}
    if op == "host":
        return {"op": op, "data": rng.choice(["url", "random"]), "n": _log_uniform(rng, 1000, 4000000), "max_len": 0}
    if op == "dna":
        return {"op": op, "data": "dna", "n": _log_uniform(rng, 1000, 4000000), "max_len": 500}
    if op == "suffix_array":
        return {"op": op, "data": "dna", "n": _log_uniform(rng, 1000, 4000000)}
    if op == "merge":
        return {"op": op, "data": rng.choice(["url", "random"]), "n": _log_uniform(rng, 5000, 12000000),
                "runs": rng.randint(2, 40)}
    return {"op": "batch", "sets": _log_uniform(rng, 8, 600), "smin": 100, "smax": _log_uniform(rng, 5000, 200000)}


# ---- inputs ------------------------------------------------------------------------------


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randint(g, lo, hi, n, dtype=torch.int64):
    """n uniform whole numbers of [lo, hi]."""
    return torch.randint(lo, hi + 1, (n,), generator=g, device=DEV, dtype=dtype)


def _pack(lens):
    """Start offsets of strings laid out back to back with one terminator each, and the bytes in all."""
    ends = torch.cumsum(lens + 1, 0)
    return ends - (lens + 1), int(ends[-1])


HOSTS, HOST_MAX = 2000, 40
TLDS = (b".com", b".org", b".net", b".de", b".edu", b".io", b".info")


def _host_table(g):
    """2000 host names: an optional "www.", 8 to 18 letters, an optional dot and 3 to 8 letters, a top-level domain."""
    def put(text, where):
        for j, ch in enumerate(text):
            table[where, length[where] + j] = ch
        length[where] += len(text)

    table = _randint(g, ord("a"), ord("z"), HOSTS * HOST_MAX, torch.uint8).view(HOSTS, HOST_MAX).cpu()
    u = torch.rand((HOSTS, 3), generator=g, device=DEV).cpu()
    label, sub = _randint(g, 8, 18, HOSTS).cpu(), _randint(g, 3, 8, HOSTS).cpu()
    tld = _randint(g, 0, len(TLDS) - 1, HOSTS).cpu()
    length = torch.zeros(HOSTS, dtype=torch.int64)
    put(b"www.", torch.nonzero(u[:, 0] < 0.5).view(-1))
    length += label
    dotted = torch.nonzero(u[:, 1] < 0.5).view(-1)
    put(b".", dotted)
    length[dotted] += sub[dotted]
    for k, text in enumerate(TLDS):
        put(text, torch.nonzero(tld == k).view(-1))
    return table.to(DEV), length.to(DEV)


def _url_set(n, seed):
    """URL-like strings: http:// or https://, a Zipf(1.1) host, 1 to 6 path segments of 3 to 12 letters and digits."""
    g = _gen(seed)
    table, hlen = _host_table(g)
    cdf = torch.cumsum(torch.arange(1, HOSTS + 1, dtype=torch.float64, device=DEV) ** -1.1, 0)
    host = torch.searchsorted(cdf / cdf[-1], torch.rand(n, generator=g, device=DEV, dtype=torch.float64))
    host.clamp_(max=HOSTS - 1)
    secure = _randint(g, 0, 1, n)
    nseg = _randint(g, 1, 6, n)
    seglen = [_randint(g, 3, 12, n) for _ in range(6)]
    lens = 7 + secure + hlen[host]
    for j in range(6):
        lens += (nseg > j) * (1 + seglen[j])
    offsets, total = _pack(lens)
    chars = _randint(g, 0, 35, total, torch.uint8)
    chars = torch.where(chars < 26, chars + ord("a"), chars + (ord("0") - 26))
    chars[offsets + lens] = 0
    for j, ch in enumerate(b"http"):
        chars[offsets + j] = ch
    chars[(offsets + 4)[secure == 1]] = ord("s")
    at = offsets + 4 + secure
    for j, ch in enumerate(b"://"):
        chars[at + j] = ch
    at = at + 3
    for j in range(HOST_MAX):
        on = torch.nonzero(hlen[host] > j).view(-1)
        if on.numel():
            chars[at[on] + j] = table[host[on], j]
    at = at + hlen[host]
    for j in range(6):
        on = nseg > j
        chars[at[on]] = ord("/")
        at = at + 1 + seglen[j]
    return chars, offsets


def _random_set(n, seed, lmin, lmax, lo, hi):
    g = _gen(seed)
    lens = _randint(g, lmin, lmax, n)
    offsets, total = _pack(lens)
    chars = _randint(g, lo, hi, total, torch.uint8)
    chars[offsets + lens] = 0
    return chars, offsets


def _prefix_set(n, seed, prefix):
    """Records under one key path: a common prefix, then 0 to 12 characters of a small alphabet."""
    g = _gen(seed)
    lens = prefix + _randint(g, 0, 12, n)
    offsets, total = _pack(lens)
    chars = _randint(g, ord("a"), ord("c"), total, torch.uint8)
    head = _randint(g, ord("a"), ord("z"), prefix, torch.uint8)
    for j in range(prefix):
        chars[offsets + j] = head[j]
    chars[offsets + lens] = 0
    return chars, offsets


def _dna_text(n, seed):
    """n characters of A, C, G, T: order-3 Markov chains, 5 % of the text overwritten by 1000-character copies."""
    g = _gen(seed)
    prob = torch.distributions.Exponential(1.0).icdf(torch.rand((64, 4), generator=g, device=DEV) * 0.999 + 5e-4)
    cum = torch.cumsum(prob / prob.sum(1, keepdim=True), 1)[:, :3].contiguous()
    steps = max(16, min(512, n // 64))
    chains = (n + steps - 1) // steps
    u = torch.rand((steps, chains, 1), generator=g, device=DEV)
    out = torch.empty((steps, chains), dtype=torch.uint8, device=DEV)
    ctx = _randint(g, 0, 63, chains)
    for s in range(steps):
        a = (u[s] > cum[ctx]).sum(1)
        out[s] = a
        ctx = ((ctx << 2) | a) & 63
    text = torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV)[out.t().reshape(-1)[:n].long()]
    block = 1000
    copies = n * 5 // 100 // block
    if copies:
        to = torch.randperm(n // block, generator=g, device=DEV)[:copies] * block
        source = _randint(g, 0, n - block, copies)
        step = torch.arange(block, device=DEV)
        text[(to[:, None] + step).view(-1)] = text[(source[:, None] + step).view(-1)]
    return torch.cat([text, torch.zeros(1, dtype=torch.uint8, device=DEV)])


def _strings(case, seed):
    data, n = case["data"], case["n"]
    if data == "url":
        return _url_set(n, seed)
    if data == "random":
        return _random_set(n, seed, 8, 32, ord("a"), ord("z"))
    if data == "bytes":  # every byte value, empty strings
        return _random_set(n, seed, 0, 40, 1, 255)
    if data == "binary":  # two letters, many equal strings
        return _random_set(n, seed, 0, 24, ord("0"), ord("1"))
    if data == "prefix":
        return _prefix_set(n, seed, case["prefix"])
    return _dna_text(n, seed), torch.arange(n, device=DEV)


def _batch_sizes(case):
    """Sizes and kinds of a batch's sets: spread evenly over the logarithm, in a mixed order, the kinds in turn."""
    k, lo, hi = case["sets"], math.log(case["smin"]), math.log(case["smax"])
    sizes = [int(round(math.exp(lo + (hi - lo) * ((j * 0.6180339887498949) % 1.0)))) for j in range(k)]
    return [(("random", "url", "dna")[j % 3], s) for j, s in enumerate(sizes)]


def _batch_sets(case, seed):
    specs = _batch_sizes(case)
    total = sum(s for _, s in specs)
    perm = torch.empty(total, dtype=torch.int32, device=DEV)
    lcp = torch.empty(total, dtype=torch.int32, device=DEV)
    sets, first = [None] * len(specs), 0
    firsts = []
    for _, size in specs:
        firsts.append(first)
        first += size
    for kind in ("random", "url", "dna"):
        mine = [j for j, (k, _) in enumerate(specs) if k == kind]
        if not mine:
            continue
        n = sum(specs[j][1] for j in mine)
        if kind == "dna":
            text = _dna_text(n + len(mine), seed + 2)
        else:
            chars, offsets = _strings({"data": kind, "n": n}, seed + (kind == "url"))
            starts = offsets.cpu()
        at = 0
        for j in mine:
            size = specs[j][1]
            out = (perm[firsts[j]:firsts[j] + size], lcp[firsts[j]:firsts[j] + size])
            if kind == "dna":  # the suffixes of a stretch of the text, which ends in a zero byte
                text[at + size] = 0
                sets[j] = (text[at:at + size + 1], torch.arange(size, device=DEV), 500) + out
                at += size + 1
            else:
                end = int(starts[at + size]) if at + size < n else chars.numel()
                begin = int(starts[at])
                sets[j] = (chars[begin:end], offsets[at:at + size] - begin, 0) + out
                at += size
    return sets, perm, lcp


def prepare(case, seed):
    op = case["op"]
    state = {"case": case}
    if op == "batch":
        sets, state["perm"], state["lcp"] = _batch_sets(case, seed)
        state["plan"] = ss.Batch(sets)
        return state
    if op == "suffix_array":
        state["text"] = _dna_text(case["n"], seed)
        return state
    state["chars"], state["offsets"] = chars, offsets = _strings(case, seed)
    n = case["n"]
    if op == "noalloc":
        state["out"] = (torch.empty(n, dtype=torch.int32, device=DEV), torch.empty(n, dtype=torch.int32, device=DEV))
    elif op == "merge":
        owner = _randint(_gen(seed + 1), 0, case["runs"] - 1, n)
        state["runs"] = []
        for k in range(case["runs"]):
            member = torch.nonzero(owner == k).view(-1)
            perm, lcp = ss.sort(chars, offsets[member])
            state["runs"].append((member.int()[perm.long()], lcp))
    elif op == "host":
        state["chars"], state["offsets"] = chars.cpu().pin_memory(), offsets.cpu().pin_memory()
        state["perm"] = torch.empty(n, dtype=torch.int32).pin_memory()
        state["lcp"] = torch.empty(n, dtype=torch.int32).pin_memory()
    return state


def run(state):
    case = state["case"]
    op = case["op"]
    if op == "sort":
        perm, lcp = ss.sort(state["chars"], state["offsets"], max_len=case["max_len"], with_lcp=case["lcp"],
                            sync=case["wait"])
        return [perm, lcp] if case["lcp"] else [perm]
    if op == "noalloc":
        return list(ss.sort_noalloc(state["chars"], state["offsets"], max_len=case["max_len"], out=state["out"]))
    if op == "dna":
        return list(ss.sort(state["chars"], state["offsets"], max_len=case["max_len"], dna=True))
    if op == "suffix_array":
        return list(ss.suffix_array(state["text"]))
    if op == "merge":
        return list(ss.merge(state["chars"], state["offsets"], state["runs"]))
    if op == "batch":
        state["plan"].run()
        return [state["perm"], state["lcp"]]
    return list(ss.sort_host(state["chars"], state["offsets"], max_len=case["max_len"], perm=state["perm"],
                             lcp=state["lcp"]))


# ---- what a pass cannot do without ---------------------------------------------------------


def _string_bytes(data, n, case):
    """Characters a sort has to look at: its distinguishing prefixes, or all characters where those are fewer."""
    digits = math.log2(max(n, 2))
    if data == "url":
        d = 19.0 + 0.6 * digits
    elif data == "random":
        d = digits / 4.7 + 1.5
    elif data == "bytes":
        d = digits / 8 + 1.5
    elif data == "binary":
        d = min(13.0, digits)
    elif data == "prefix":
        d = case["prefix"] + 7.0
    else:  # suffixes share their text
        d = 1.0
    return n * (min(d, case["max_len"]) if case.get("max_len") else d)


def work(case):
    op = case["op"]
    if op == "batch":
        specs = _batch_sizes(case)
        return {"bytes": sum(16 * s + _string_bytes(k, s, {}) for k, s in specs), "flops": 0}
    n = case["n"]
    if op == "suffix_array":
        return {"bytes": 9 * n, "flops": 0}  # the text in, both arrays out
    if op == "merge":  # offsets, runs' orders and LCPs, characters; order and LCPs out
        return {"bytes": 24 * n + _string_bytes(case["data"], n, case), "flops": 0}
    if op == "host":  # every character and offset crosses to the device
        mean = 61.0 if case["data"] == "url" else 21.0
        return {"bytes": n * (mean + 16), "flops": 0}
    out = 8 if case.get("lcp", True) else 4
    return {"bytes": (8 + out) * n + _string_bytes(case["data"], n, case), "flops": 0}
