"""The measured workloads of this library: what a program that serves LLM agents
with MemDecay eviction has it do, called through the public entry points.

A case keeps a paged KV cache at a steady occupancy, as a server under a page
budget does: `prepare` fills the cache with agent traces (region spans, turn by
turn insertion steps) and sets every sequence's budget to the pages it then
holds; one pass appends what the turn or the decode steps bring, decodes, and
evicts back to the budget, so a state can be passed over any number of times.

Fields of a case:
  entry    "step"    md_decode_step for all layers at once, then md_evict
           "host"    md_decode_step_host (pinned host buffers), md_evict, md_sync
           "layers"  md_decode_layer, one call per layer as a model's loop makes
                     them, then md_evict
           "append"  md_append_tokens of `new` tokens to every sequence (a prompt
                     or a tool's output), the decode step after it, md_evict
           "noalloc" md_attend_mass_noalloc over a cache that the caller owns
  layers, q_heads, kv_heads, page   the model's attention geometry, tokens per page
  batch, tokens, ragged   sequences, tokens of the longest, and the share by which
                     the others may be shorter
  new      tokens appended per sequence and pass ("append")
  window   decode steps per observation (md_evict)
  aligned  region-aligned page allocation
  mode, reduce, calib   score form, page reduction, calibration histogram
  inspect  the pass also reads the token state back (device to device)

Keys, values and queries are N(0, 1) in bf16, with the system span and 2% of the
tokens attended more strongly along one direction, so that some clocks refresh."""
import math
import random

import numpy as np
import torch

import paper_2607_10582_gb300 as md

D = 128
SYSTEM, SCRATCHPAD = 0, 6
BASE = (1.0, 0.8, 0.7, 0.4, 0.3, 0.5, 0.2)
HALF_LIFE = (160.0, 80.0, 60.0, 30.0, 25.0, 40.0, 15.0)
RHO, GAMMA, TAU_SCALE, ATTN_WEIGHT = 0.9, 0.1, 2.0, 1.0
HOT_DIMS, HOT_KEY, HOT_QUERY, HOT_SHARE = 16, 2.0, 0.5, 0.02

DEFAULTS = {"entry": "step", "layers": 36, "q_heads": 16, "kv_heads": 2, "page": 16, "batch": 1, "tokens": 448,
            "ragged": 0.0, "new": 0, "window": 1, "aligned": False, "mode": 0, "reduce": 0, "calib": False,
            "inspect": False}


def _case(name, **kw):
    c = dict(DEFAULTS, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one short agent episode on one layer: the smallest call, launches and latency
        _case("step 1x448 L1", layers=1, q_heads=12, tokens=448),
        # one agent's full 1,700-token episode, 1.5B geometry: an interactive single user
        _case("step 1x1700 L28", layers=28, q_heads=12, tokens=1700),
        # the same user under a model that runs its other layers between the attentions
        _case("layers 1x1700 L28", entry="layers", layers=28, q_heads=12, tokens=1700),
        # a serving batch at a 25% budget, 3B geometry: the steady state of the decode loop
        _case("step 32x430 L36", batch=32, tokens=430, ragged=0.25, inspect=True),
        # that batch with its inputs and outputs in host memory
        _case("host 32x430 L36", entry="host", batch=32, tokens=430, ragged=0.25),
        # that batch layer by layer, as a model's forward pass calls it
        _case("layers 32x430 L36", entry="layers", batch=32, tokens=430, ragged=0.25, inspect=True),
        # long contexts layer by layer
        _case("layers 16x13001 L36 p32", entry="layers", batch=16, tokens=13001, ragged=0.3, page=32, mode=2,
              inspect=True),
        # a windowed observation with region-aligned pages, page max and the histogram on
        _case("window 12x2400 L16 aligned", layers=16, q_heads=12, batch=12, tokens=2400, ragged=0.5, page=32,
              window=4, aligned=True, reduce=1, calib=True, inspect=True),
        # eight agents each get a tool's output of 317 tokens
        _case("append 8x317 L36", entry="append", batch=8, tokens=1500, ragged=0.5, new=317, mode=2, inspect=True),
        # one long prompt arrives and is cut back to its budget
        _case("append 1x8192 L36", entry="append", tokens=816, new=8192, mode=2, inspect=True),
        # attention and mass over a cache that a serving engine owns
        _case("noalloc 24x999 L16", entry="noalloc", layers=16, batch=24, tokens=999, ragged=0.6),
        # long agent histories, the largest call
        _case("step 8x131072 L36 p32", batch=8, tokens=131072, page=32, mode=2, inspect=True),
    ]


MAX_KV_BYTES = 8 * 131072 * 36 * 2 * 4 * D


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        entry = rng.choice(("step", "step", "step", "host", "layers", "layers", "append", "noalloc"))
        q_heads, kv_heads = rng.choice(((12, 2), (16, 2), (16, 2), (8, 2), (8, 1), (28, 4), (32, 8)))
        c = _case("", entry=entry, layers=rng.choice((1, 2, 4, 8, 16, 24, 28, 36)), q_heads=q_heads,
                  kv_heads=kv_heads, page=rng.choice((16, 32)), batch=_log_int(rng, 1, 64),
                  ragged=rng.choice((0.0, 0.3, 0.8)), tokens=_log_int(rng, 100, 131072))
        if entry == "append":
            c["tokens"] = _log_int(rng, 200, 8000)
            c["new"] = _log_int(rng, 20, 16000)
            c["batch"] = _log_int(rng, 1, 8)
        if entry == "noalloc":
            c["tokens"] = _log_int(rng, 100, 1024)     # the sizes its fixed scratch always takes
        if entry in ("step", "layers"):
            c["window"] = rng.choice((1, 1, 1, 2, 5))
            c["aligned"] = rng.random() < 0.2
            c["reduce"] = rng.choice((0, 0, 1))
            c["calib"] = rng.random() < 0.15
        c["mode"] = 2 if c["tokens"] + c["new"] > 2000 else rng.choice((0, 0, 1, 2))
        w = work(c)
        c["inspect"] = entry != "noalloc" and w["bytes"] > 2e8
        if c["batch"] * (c["tokens"] + c["new"]) * c["layers"] * kv_heads * 4 * D <= MAX_KV_BYTES and \
                w["bytes"] <= MAX_KV_BYTES:
            return c


# ------------------------------------------------------------------ shapes ----
def _lengths(c):
    """Tokens per sequence before the first pass (the same for every seed)."""
    r = random.Random(c["batch"] * 1000003 + c["tokens"])
    return [max(8, int(c["tokens"] * (1.0 - (c["ragged"] * r.random() if b else 0.0)))) for b in range(c["batch"])]


def work(case):
    """The cached K/V read once per decode step, the queries, outputs and new
    tokens' K/V, appended K/V read and written once, and per observation the
    token state (region, a, clock, window, observed mass, priority: 33 bytes)
    and the block table."""
    c = dict(DEFAULTS, **case)
    L, Hq, Hkv, k = c["layers"], c["q_heads"], c["kv_heads"], c["window"]
    n = sum(_lengths(c))
    kv_token = L * Hkv * 4 * D
    if c["entry"] == "noalloc":
        return {"bytes": n * kv_token + 2 * c["batch"] * L * Hq * 2 * D + 4 * n * L * Hkv + 4 * n // c["page"],
                "flops": 4 * Hq * D * L * n}
    held = n + c["batch"] * c["new"]
    attended = sum(held + c["batch"] * (s + 1) for s in range(k))
    appended = c["batch"] * (c["new"] + k)
    held += c["batch"] * k
    return {"bytes": attended * kv_token + 2 * k * c["batch"] * L * Hq * 2 * D + 2 * appended * kv_token +
            33 * held + 12 * held // c["page"], "flops": 4 * Hq * D * L * attended}


def _blocks(n, rng):
    """Region labels and insertion steps of one trace: a pinned system span, then
    turn blocks, a turn every 16 decode steps before now."""
    lo = max(4, min(64, n // 16))
    hi = max(lo, min(589, n // 5))
    spans = [(SYSTEM, max(1, min(512, n // 7)))]
    used = spans[0][1]
    while used < n:
        m = min(rng.randint(lo, hi), n - used)
        spans.append((rng.randint(1, 6), m))
        used += m
    lab = np.concatenate([np.full(m, r, np.uint8) for r, m in spans])
    ins = np.concatenate([np.full(m, -(len(spans) - i) * 16, np.int32) for i, (_, m) in enumerate(spans)])
    return lab, ins


def _trace(c, seed, b, n):
    """(labels, insertion steps, labels of the tokens that a pass appends) of sequence b.
    Region-aligned pages are counted by the labels: those are the same for every
    seed there, so that the state arrays keep their sizes."""
    rng = random.Random((0 if c["aligned"] else seed) * 7919 + b)
    lab, ins = _blocks(n, rng)
    more = np.zeros(0, np.uint8)
    while len(more) < c["new"]:
        more = np.concatenate([more, np.full(rng.randint(16, 400), rng.randint(1, 6), np.uint8)])
    return lab, ins, more[:c["new"]]


def _gen(seed, *what):
    g = torch.Generator(device="cuda")
    x = seed
    for w in what:
        x = (x * 1000003 + w + 17) % (1 << 61)
    g.manual_seed(x)
    return g


def _kv(c, seed, b, part, n, lab):
    """K and V of n tokens of sequence b: bf16 [layers][kv_heads][n][D]."""
    g = _gen(seed, 1, b, part)
    shape = (c["layers"], c["kv_heads"], n, D)
    k = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    v = torch.randn(shape, generator=g, device="cuda", dtype=torch.bfloat16)
    hot = torch.rand(n, generator=g, device="cuda") < HOT_SHARE
    hot |= torch.from_numpy(lab == SYSTEM).cuda()
    k[..., :HOT_DIMS] += HOT_KEY * hot[:, None].to(torch.bfloat16)
    return k, v


def _step_inputs(c, seed):
    """q [window][batch][layers][q_heads][D], new K and V [window][batch][layers][kv_heads][D]."""
    g = _gen(seed, 2)
    lead = (c["window"], c["batch"], c["layers"])
    q = torch.randn(lead + (c["q_heads"], D), generator=g, device="cuda", dtype=torch.bfloat16)
    q[..., :HOT_DIMS] += HOT_QUERY
    k = torch.randn(lead + (c["kv_heads"], D), generator=g, device="cuda", dtype=torch.bfloat16)
    v = torch.randn(lead + (c["kv_heads"], D), generator=g, device="cuda", dtype=torch.bfloat16)
    return q, k, v


def _pages(lab, page, aligned):
    """Page and offset in it of every token of a sequence, in order."""
    n = len(lab)
    if not aligned:
        return np.arange(n) // page, np.arange(n) % page
    start = np.concatenate([[True], lab[1:] != lab[:-1]])
    first = np.maximum.accumulate(np.where(start, np.arange(n), 0))
    off = (np.arange(n) - first) % page
    return np.cumsum(off == 0) - 1, off


# -------------------------------------------------------------------- state ----
def prepare(case, seed):
    c = dict(DEFAULTS, **case)
    lens = _lengths(c)
    traces = [_trace(c, seed, b, n) for b, n in enumerate(lens)]
    if c["entry"] == "noalloc":
        return _prepare_noalloc(c, seed, lens, traces)
    B, L, page = c["batch"], c["layers"], c["page"]
    pages = [int(_pages(t[0], page, c["aligned"])[0][-1]) + 1 for t in traces]
    extra = c["window"] // page + 3 + -(-c["new"] // page)
    cache = md.Cache(L, c["q_heads"], c["kv_heads"], page, B, max(pages) + extra, sum(pages) + B * extra,
                     rho=RHO, gamma=GAMMA, tau_scale=TAU_SCALE, attn_weight=ATTN_WEIGHT, score_mode=c["mode"],
                     page_reduce=c["reduce"], region_aligned_pages=int(c["aligned"]))
    for r in range(7):
        cache.set_region_params(r, BASE[r], HALF_LIFE[r], r == SYSTEM)
    if c["calib"]:
        cache.calib_enable(True)
    for b, (lab, ins, _) in enumerate(traces):
        k, v = _kv(c, seed, b, 0, lens[b], lab)
        cache.append_tokens(b, lab, k, v, insert_steps=ins)
        del k, v
    s = {"case": c, "cache": cache, "regions": np.full(B, SCRATCHPAD, np.uint8),
         "budget": np.array([cache.query(md.MD_QUERY_PAGES, b) for b in range(B)], np.int32)}
    q, k, v = _step_inputs(c, seed)
    if c["entry"] == "layers":     # a model hands over one layer's tensors at a time
        q, k, v = (x.transpose(1, 2).contiguous() for x in (q, k, v))
    if c["entry"] == "host":
        q, k, v = (x.cpu().pin_memory() for x in (q, k, v))
        s["out"] = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
    else:
        s["out"] = torch.empty_like(q)
    s["q"], s["k"], s["v"] = ([x[i] for i in range(c["window"])] for x in (q, k, v))
    s["o"] = [s["out"][i] for i in range(c["window"])]
    if c["entry"] == "layers":
        s["q"], s["k"], s["v"], s["o"] = ([[x[l] for l in range(L)] for x in s[n]] for n in ("q", "k", "v", "o"))
    if c["new"]:
        s["new"] = [(t[2],) + _kv(c, seed, b, 1, c["new"], t[2]) for b, t in enumerate(traces)]
    torch.cuda.synchronize()
    return s


def _prepare_noalloc(c, seed, lens, traces):
    L, Hkv, page = c["layers"], c["kv_heads"], c["page"]
    pages = [-(-n // page) for n in lens]
    P = sum(pages)
    ids = list(range(P))
    random.Random(seed).shuffle(ids)      # an engine's pages lie anywhere in its pool
    table = np.zeros((c["batch"], max(pages)), np.int32)
    pool = torch.zeros((L, P, Hkv, 2, page, D), dtype=torch.bfloat16, device="cuda")
    at = 0
    for b, n in enumerate(lens):
        table[b, :pages[b]] = ids[at:at + pages[b]]
        at += pages[b]
        row = torch.from_numpy(table[b, :pages[b]]).cuda().long()
        for x, t in enumerate(_kv(c, seed, b, 0, n, traces[b][0])):
            t = torch.nn.functional.pad(t, (0, 0, 0, pages[b] * page - n))
            pool[:, row, :, x] = t.view(L, Hkv, pages[b], page, D).transpose(1, 2)
    q = _step_inputs(c, seed)[0][0]
    return {"case": c, "pool": pool, "table": torch.from_numpy(table).cuda(), "tokens": np.array(lens, np.int32),
            "q": q, "out": torch.empty_like(q), "mass": torch.zeros((L * Hkv, P * page), device="cuda"), "P": P}


# --------------------------------------------------------------------- pass ----
def run(state):
    c = state["case"]
    B = c["batch"]
    if c["entry"] == "noalloc":
        st = md.lib().md_attend_mass_noalloc(
            state["pool"].data_ptr(), state["table"].data_ptr(), state["tokens"].ctypes.data, state["q"].data_ptr(),
            state["out"].data_ptr(), state["mass"].data_ptr(), B, c["layers"], c["q_heads"], c["kv_heads"],
            c["page"], state["table"].shape[1], state["P"], torch.cuda.current_stream().cuda_stream)
        if st != md.MD_OK:
            raise RuntimeError("md_attend_mass_noalloc: %d" % st)
        return {"out": state["out"], "mass": state["mass"]}
    cache, regions = state["cache"], state["regions"]
    if c["new"]:
        for b, (lab, k, v) in enumerate(state["new"]):
            cache.append_tokens(b, lab, k, v)
    for i in range(c["window"]):
        q, k, v, o = state["q"][i], state["k"][i], state["v"][i], state["o"][i]
        if c["entry"] == "layers":
            for l in range(c["layers"]):
                cache.decode_layer(l, B, q[l], k[l], v[l], regions, o[l])
        elif c["entry"] == "host":
            cache.decode_step_host(B, q, k, v, regions, o)
        else:
            cache.decode_step(B, q, k, v, regions, o)
    _, evicted = cache.evict(state["budget"])
    r = {"out": state["out"], "evicted": evicted, "page_score": cache.get_state(md.MD_STATE_PAGE_SCORE)}
    if c["inspect"]:
        r["a"] = cache.get_state(md.MD_STATE_A)
        r["t_ref"] = cache.get_state(md.MD_STATE_T_REF)
        r["block_table"] = cache.get_state(md.MD_STATE_BLOCK_TABLE)
    if c["entry"] == "host":
        cache.sync()               # the output is in host memory from here on
    return r


# -------------------------------------------------------------------- exact ----
def _attend(q, k, v):
    """Outputs [Hq][D] and per (KV head) token masses [Hkv][n] of one layer, in 64 bits."""
    Hkv, n, _ = k.shape
    q = q.double().view(Hkv, -1, D)
    p = torch.softmax(torch.matmul(q, k.double().transpose(1, 2)) / math.sqrt(D), dim=-1)
    return torch.matmul(p, v.double()).reshape(-1, D), p.sum(1)


def exact(case, seed):
    """One pass on a newly prepared state, in 64-bit torch: attention outputs,
    a and page scores.  The discrete outputs (counts, clocks, table) have none."""
    c = dict(DEFAULTS, **case)
    lens = _lengths(c)
    L, Hq, Hkv, B, page, win = c["layers"], c["q_heads"], c["kv_heads"], c["batch"], c["page"], c["window"]
    traces = [_trace(c, seed, b, n) for b, n in enumerate(lens)]
    q, kn, vn = _step_inputs(c, seed)
    if c["entry"] == "noalloc":
        pages = [-(-n // page) for n in lens]
        ids = list(range(sum(pages)))
        random.Random(seed).shuffle(ids)
        out = torch.empty((B, L, Hq, D), dtype=torch.float64, device="cuda")
        mass = torch.zeros((L * Hkv, sum(pages) * page), dtype=torch.float64, device="cuda")
        at = 0
        for b, n in enumerate(lens):
            k, v = _kv(c, seed, b, 0, n, traces[b][0])
            i = torch.arange(n, device="cuda")
            slot = torch.tensor(ids[at:at + pages[b]], device="cuda")[i // page] * page + i % page
            at += pages[b]
            for l in range(L):
                out[b, l], m = _attend(q[0, b, l], k[l], v[l])
                mass[l * Hkv:(l + 1) * Hkv, slot] = m
        return {"out": out, "mass": mass}
    labels = [np.concatenate([t[0], t[2], np.full(win, SCRATCHPAD, np.uint8)]) for t in traces]
    where = [_pages(lab, page, c["aligned"]) for lab in labels]
    # physical pages are popped in order: the prepared traces', the appended tokens', then each step's
    marks = [[lens[b], lens[b] + c["new"]] + [lens[b] + c["new"] + i + 1 for i in range(win)] for b in range(B)]
    phys = [np.zeros(where[b][0][-1] + 1, np.int64) for b in range(B)]
    top, have = 0, [0] * B
    for stage in range(2 + win):
        for b in range(B):
            upto = int(where[b][0][marks[b][stage] - 1]) + 1
            phys[b][have[b]:upto] = np.arange(top, top + upto - have[b])
            top += upto - have[b]
            have[b] = upto
    budget = [int(where[b][0][lens[b] - 1]) + 1 for b in range(B)]
    extra = win // page + 3 + -(-c["new"] // page)
    P_max, P_phys = max(budget) + extra, sum(budget) + B * extra
    out = torch.empty((win, B, L, Hq, D), dtype=torch.float64, device="cuda")
    a_all = torch.zeros(P_phys * page, dtype=torch.float64, device="cuda")
    score = torch.zeros((B, P_max), dtype=torch.float64, device="cuda")
    base = torch.tensor(BASE, dtype=torch.float64, device="cuda")
    half = torch.tensor(HALF_LIFE, dtype=torch.float64, device="cuda")
    for b in range(B):
        n = lens[b] + c["new"] + win
        k, v = _kv(c, seed, b, 0, lens[b], traces[b][0])
        if c["new"]:
            k2, v2 = _kv(c, seed, b, 1, c["new"], traces[b][2])
            k, v = torch.cat([k, k2], 2), torch.cat([v, v2], 2)
        mass = torch.zeros(n, dtype=torch.float64, device="cuda")
        for l in range(L):
            kl = torch.cat([k[l], kn[:, b, l].transpose(0, 1)], 1)
            vl = torch.cat([v[l], vn[:, b, l].transpose(0, 1)], 1)
            for i in range(win):
                m = n - win + i + 1
                out[i, b, l], p = _attend(q[i, b, l], kl[:, :m], vl[:, :m])
                mass[:m] += p.sum(0)
        abar = mass / (win * L * Hq)
        a = GAMMA * abar
        ins = np.concatenate([traces[b][1], np.zeros(c["new"], np.int32), np.arange(1, win + 1, dtype=np.int32)])
        age = win - torch.from_numpy(ins).cuda().double()
        age = torch.where(abar >= TAU_SCALE / n, torch.zeros_like(age), age)
        lab = torch.from_numpy(labels[b]).cuda().long()
        d = torch.exp2(-age / half[lab])
        w = ATTN_WEIGHT * a
        s = {0: base[lab] * d + w, 1: (base[lab] + w) * d, 2: base[lab] * d + w * n}[c["mode"]]
        s = torch.where(lab == SYSTEM, torch.full_like(s, math.inf), s)
        pg = torch.from_numpy(where[b][0]).cuda()
        P = int(pg[-1]) + 1
        if c["reduce"]:
            S = torch.full((P,), -math.inf, dtype=torch.float64, device="cuda").scatter_reduce(0, pg, s, "amax")
        else:
            S = torch.zeros(P, dtype=torch.float64, device="cuda").index_add(0, pg, s) / torch.bincount(pg, minlength=P)
        S[P - 1] = math.inf
        score[b, :P] = S
        a_all[torch.from_numpy(phys[b][where[b][0]] * page + where[b][1]).cuda()] = a
    if c["entry"] == "layers":
        out = out.transpose(1, 2).contiguous()
    r = {"out": out, "evicted": None, "page_score": score}
    if c["inspect"]:
        r.update({"a": a_all, "t_ref": None, "block_table": None})
    return r


def tolerance(case):
    """Set by the bf16 attention output: its rounding and the probabilities'
    rounding to bf16 before the PV product come to 2.1e-3 of the 64-bit result.
    The state arrays are 32-bit (1e-7) and lie far inside it; a page swapped
    against another at an equal score moves whole entries of the table."""
    return {"rel": 8e-3, "max": 0.1, "differ": 0.01}
