"""The decode path's use, as cases that can be timed: what a serving program has this library do, through its public entry points.

A case is one of these kinds of pass:

  decode   `steps` calls of gp_decode_step over all requests of a pool (the program's inner loop)
  host     the same through gp_decode_step_host_async / _wait from page-locked host buffers, the host one step behind
  layers   `steps` decode steps layer by layer with the query / key normalisation fused in, as a model's forward pass calls them
  admit    requests admitted with their prompts (the prefill's keys and values go into pages), decoded once, released
  prefix   groups of requests that share a prompt: admitted by reference, decoded past their first compaction (copy-on-write), released
  dense    gp_attention_noalloc over plain keys and values

Requests of the decoding kinds have ragged lengths, so that about one in `page` of them reaches its capacity boundary at
each step, and a pool with a few pages to spare, so that after some steps every boundary compresses: the steady state of a
server under memory pressure.  Inputs are those of the repository's workloads: per (layer, KV head) a unit direction u, heavy
keys 4u + 0.1 N(0, I) with a probability of the request's own, other keys and all values N(0, I), queries 2u + N(0, I).
"""
import math

import torch

from paper_2609_03494_b200 import binding as B

DEV = "cuda:0"
RING_BYTES = 3.0e9          # decode-step inputs kept per state: the ring is as long as this allows, 1024 steps at most


def _case(kind, name=None, **kw):
    c = dict(kind=kind, layers=1, hq=32, hkv=8, d=128, page=16, k_loc=4, rope=0.0, requests=64, lo=128, hi=1280, steps=16, group=1)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The tiny configuration: a handful of short requests, one small layer.  Launches and latency are everything.
        _case("decode", "tiny", hq=8, hkv=2, d=64, requests=4, lo=64, hi=240),
        # One Qwen3-8B-shaped layer, 64 requests on budgets of 8 to 88 pages: the repository's headline workload.
        _case("decode", "layer_8b", lo=128, hi=1400),
        # The same layer fed from and read back to host memory each step, the host one step behind the GPU.
        _case("host", "layer_8b_host", lo=128, hi=1400),
        # The whole 36-layer stack with a small batch: interactive serving.
        _case("decode", "stack_8b_small_batch", layers=36, requests=16, lo=400, hi=1000),
        # The whole 36-layer stack with many residents: throughput serving.
        _case("decode", "stack_8b_large_batch", layers=36, requests=256, lo=128, hi=1152),
        # The 64-layer Qwen3-32B shape (groups of eight query heads), rotary embedding on, a medium batch.
        _case("decode", "stack_32b", layers=64, hq=64, requests=32, lo=200, hi=1800, rope=1e6),
        # A few very long generations on groups of eight: outputs up to 32 k tokens, candidate sets of thousands of pages.
        _case("decode", "long_context", layers=4, hq=64, requests=4, lo=9000, hi=32000, rope=1e6),
        # The paper's own page geometry: pages of 256 tokens, a protected window of 16, a local quota of 64.
        _case("decode", "page_256", layers=8, page=256, k_loc=64, requests=24, lo=700, hi=5000, rope=1e6, steps=32),
        # A model's forward pass: every layer on its own, normalisation and rotation fused in.
        _case("layers", "model_forward", layers=36, requests=16, lo=400, hi=1000, rope=1e6, steps=4),
        # New requests arriving: their prompts go into pages of all 36 layers.
        _case("admit", "admission", layers=36, requests=8, lo=100, hi=1024, steps=1),
        # Prefix caching: 16 groups of 16 on a 2048-token prompt, copied on write at their first compaction.
        _case("prefix", "prefix_sharing", requests=256, group=16, lo=2048, hi=2048, steps=24),
        # Attention alone for callers that may not allocate: plain keys and values, ragged lengths.
        _case("dense", "dense_attention", requests=64, lo=60, hi=4000, steps=1),
    ]


def draw(rng):
    """One more case of the ranges above: sizes over their logarithm, odd ones among them; costs less than the largest listed one."""
    kind = rng.choice(["decode", "decode", "decode", "host", "layers", "admit", "prefix", "dense"])
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))
    hkv = rng.choice([2, 4, 8])
    hq = hkv * rng.choice([1, 2, 4, 4, 8])
    d = rng.choice([64, 128, 128])
    rope = rng.choice([0.0, 1e6])
    if kind == "dense":
        return _case(kind, hq=hq, hkv=hkv, d=d, requests=max(1, min(log(1, 96), 2048 // hq)), lo=log(1, 100), hi=log(200, 9000), steps=1)
    if kind == "prefix":
        per = rng.choice([2, 5, 8, 16])
        return _case(kind, hq=hq, hkv=hkv, d=d, rope=rope, layers=log(1, 4), requests=per * log(1, 12), group=per, lo=(p := 16 * log(8, 128)), hi=p, steps=20)
    layers = log(1, 48)
    if kind == "admit":
        hi = log(200, 3000)
        return _case(kind, hq=hq, hkv=hkv, d=d, rope=rope, layers=layers, requests=log(1, 12), lo=max(33, hi // 8), hi=hi, steps=1)
    page = rng.choice([16, 16, 16, 64, 256]) if kind == "decode" else 16
    hi = max(log(100, 12000), 3 * page + 40)
    lo = max(2 * page + 8, int(hi * rng.uniform(0.08, 0.7)))
    per_request = layers * hkv * d * 4 * (lo + hi) / 2
    most = 300e6 if kind == "host" else 4e9
    while per_request > most and layers > 1:
        layers = (layers + 1) // 2
        per_request = layers * hkv * d * 4 * (lo + hi) / 2
    requests = max(1, min(log(1, 200), int(most / per_request)))
    steps = {"layers": 2, "host": 8}.get(kind, 16)
    return _case(kind, hq=hq, hkv=hkv, d=d, rope=rope, layers=layers, page=page, k_loc=page // 4, requests=requests, lo=lo, hi=hi, steps=steps)


# ---- inputs ---------------------------------------------------------------------------------------------------------
def _lengths(case, gen):
    """Prompt lengths over [lo, hi], one from each of `requests` equal parts (so that the total hardly depends on the seed), in random order."""
    n, lo, hi = case["requests"], case["lo"], case["hi"]
    u = (torch.arange(n, dtype=torch.float64) + torch.rand(n, generator=gen, dtype=torch.float64)) / n
    x = (lo + u * (hi - lo)).round().to(torch.int64)
    return x[torch.randperm(n, generator=gen)].tolist()


def _unit(case, g):
    u = torch.randn((case["layers"], case["hkv"], case["d"]), generator=g, device=DEV)
    return (u / u.norm(dim=-1, keepdim=True)).to(torch.bfloat16)


def _keys(shape, u, heavy, g):
    """Keys of `shape` [..., hkv, d]; rows where `heavy` (broadcastable) are heavy hitters along u."""
    k = torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)
    return torch.where(heavy, torch.add(4.0 * u, k, alpha=0.1), k)


def _values(shape, g):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.bfloat16)


def _prompt(case, n, u, frac, g):
    shape = (case["layers"], n, case["hkv"], case["d"])
    heavy = (torch.rand(n, generator=g, device=DEV) < frac)[None, :, None, None]
    return _keys(shape, u[:, None], heavy, g), _values(shape, g)


def _step_inputs(case, n_req, ring, u, fracs, g):
    """`ring` decode steps' queries, keys and values: lists of [L][n_req][heads][d] bf16 tensors."""
    L, hq, hkv, d = case["layers"], case["hq"], case["hkv"], case["d"]
    uq = (2.0 * u).repeat_interleave(hq // hkv, dim=1)[:, None]
    qs, ks, vs = [], [], []
    part = max(1, min(ring, int(1.5e8 // (L * n_req * hq * d)) or 1))
    for at in range(0, ring, part):
        m = min(part, ring - at)
        heavy = (torch.rand((m, 1, n_req, 1, 1), generator=g, device=DEV) < fracs[None, None, :, None, None])
        qs += list(torch.randn((m, L, n_req, hq, d), generator=g, device=DEV, dtype=torch.bfloat16).add_(uq))
        ks += list(_keys((m, L, n_req, hkv, d), u[:, None], heavy, g))
        vs += list(_values((m, L, n_req, hkv, d), g))
    return qs, ks, vs


def _config(case, n_pages, cap, batch_tokens, boundary_tokens=0, host=False):
    return B.make_config(case["layers"], case["hq"], case["hkv"], case["d"], n_pages=n_pages, max_pages_per_req=cap,
                         max_requests=max(4, case["requests"]), k_loc=case["k_loc"], rope_theta=case["rope"], page_size=case["page"],
                         max_batch_tokens=batch_tokens, max_boundary_tokens=boundary_tokens, host_staging=host)


def _prompts(case, u, lens, fracs, g):
    """(keys, values, tokens) of every prompt that a pass or its preparation hands over, in order: one per group that shares."""
    at = range(0, case["requests"], case["group"]) if case["kind"] == "prefix" else range(case["requests"])
    for i, f in zip(at, fracs):
        yield _prompt(case, lens[i], u, f, g) + (lens[i],)


def _start(case, seed):
    """The generator, head directions, prompt lengths and shares of heavy hitters that a state's inputs begin with."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    cpu = torch.Generator()
    cpu.manual_seed(seed)
    u = _unit(case, g)
    lens = _lengths(case, cpu)
    fracs = torch.exp(torch.rand(case["requests"], generator=cpu, dtype=torch.float64) * math.log(40.0) + math.log(0.005)).tolist()
    return g, u, lens, fracs


def _dense_inputs(case, u, g):
    shape = (case["requests"], case["hkv"], case["hi"], case["d"])
    heavy = torch.rand((case["requests"], 1, case["hi"], 1), generator=g, device=DEV) < 0.05
    k, v = _keys(shape, u[0][None, :, None], heavy, g), _values(shape, g)
    q = torch.randn((case["requests"], case["hq"], case["d"]), generator=g, device=DEV, dtype=torch.bfloat16)
    q += (2.0 * u[0]).repeat_interleave(case["hq"] // case["hkv"], dim=0)[None]
    return q, k, v


def _ring(case):
    """Decode steps of inputs that a state keeps."""
    kind, steps = case["kind"], case["steps"]
    if kind in ("admit", "prefix"):
        return steps
    row = case["requests"] * case["layers"] * (case["hq"] + 2 * case["hkv"]) * case["d"] * 2
    return max(2, min(64 if kind == "layers" else 1024, int((2.0e8 if kind == "host" else RING_BYTES) / row)) // steps) * steps


def _norm_weights(case, g):
    return [1.0 + 0.1 * torch.randn(case["d"], generator=g, device=DEV) for _ in range(2)]


def _pages(case, lens):
    """Pages of the pool, and the most a request may have.  Decoding kinds: a few pages to spare, the first grants take
    them and from then on a boundary compresses."""
    kind, n_req, page = case["kind"], case["requests"], case["page"]
    pages = [n // page + 1 for n in lens]
    if kind == "admit":
        return sum(pages) + 2 * n_req, case["hi"] // page + 2
    if kind == "prefix":
        p0 = pages[0]
        return n_req // case["group"] * (p0 - 1) + n_req * (p0 + 2), p0 + 3
    return sum(pages) + max(2, sum(pages) // 50), case["hi"] // page + 5


def prepare(case, seed):
    kind, n_req, L, steps, page = case["kind"], case["requests"], case["layers"], case["steps"], case["page"]
    g, u, lens, fracs = _start(case, seed)
    if kind == "dense":
        q, k, v = _dense_inputs(case, u, g)
        return dict(case=case, q=q, k=k, v=v, lens=torch.tensor(lens, dtype=torch.int32, device=DEV),
                    out=torch.empty((n_req, case["hq"], case["d"]), dtype=torch.float32, device=DEV))

    n_pages, cap = _pages(case, lens)
    batch, bound = {"admit": (0, 0), "prefix": (n_req * cap * page, 0)}.get(kind, (n_pages * page, max(cap, n_pages // 4) * page))
    pool = B.Pool(_config(case, n_pages, cap, batch, bound, host=kind == "host"))
    st = dict(case=case, pool=pool, at=0)
    act = torch.zeros((steps, n_req), dtype=torch.int32, device=DEV)
    out = torch.zeros((steps, L, n_req, case["hq"], case["d"]), dtype=torch.float32, device=DEV)
    if kind in ("admit", "prefix"):
        st["prompts"] = list(_prompts(case, u, lens, fracs, g))       # what arrives later
    else:
        for k, v, n in _prompts(case, u, lens, fracs, g):
            status, _ = pool.request_add(-1, 0, k, v, n, 0)
            assert status == B.GP_OK, status
    qs, ks, vs = _step_inputs(case, n_req, _ring(case), u, torch.tensor(fracs, device=DEV), g)
    ids = torch.arange(n_req, dtype=torch.int32, device=DEV)
    if kind == "host":
        qs, ks, vs = (list(torch.stack(x).cpu().pin_memory()) for x in (qs, ks, vs))
        ids, act, out = ids.cpu().pin_memory(), act.cpu().pin_memory(), out.cpu().pin_memory()
    if kind == "layers":
        st["wq"], st["wk"] = _norm_weights(case, g)
        qs, ks, vs = ([list(x) for x in xs] for xs in (qs, ks, vs))          # a model hands over one layer's tensors at a time
    st.update(ids=ids, q=qs, k=ks, v=vs, out=out, act=act)
    return st


# ---- one pass -------------------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind, steps = case["kind"], case["steps"]
    if kind == "dense":
        B.gp_attention_noalloc(s["q"].data_ptr(), s["k"].data_ptr(), s["v"].data_ptr(), s["lens"].data_ptr(), case["requests"], case["hq"],
                               case["hkv"], case["d"], case["hi"], s["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return s["out"]
    pool, ids, out, act = s["pool"], s["ids"], s["out"], s["act"]
    at = s["at"]
    q, k, v = s["q"], s["k"], s["v"]
    if kind == "admit":
        rids = []
        for pk, pv, n in s["prompts"]:
            status, rid = pool.request_add(-1, 0, pk, pv, n, 0)
            assert status == B.GP_OK, status
            rids.append(rid)
        pool.decode_step(ids, q[0], k[0], v[0], out[0], act[0])
        for rid in rids:
            pool.release(rid)
        return out, act
    if kind == "prefix":
        rids = []
        for pk, pv, n in s["prompts"]:
            status, donor = pool.request_add(-1, 0, pk, pv, n, 0)
            assert status == B.GP_OK, status
            rids.append(donor)
            for _ in range(case["group"] - 1):
                status, rid = pool.request_add(donor, n // case["page"], None, None, 0, 0)
                assert status == B.GP_OK, status
                rids.append(rid)
        for j in range(steps):
            pool.decode_step(ids, q[j], k[j], v[j], out[j], act[j])
        for rid in rids:
            pool.release(rid)
        return out, act
    if kind == "host":
        for j in range(steps):
            pool.decode_step_host_async(ids, q[at + j], k[at + j], v[at + j], out[j], act[j])
            if j:
                pool.host_wait()
        pool.host_wait()
    elif kind == "layers":
        h, n, stream = pool.handle, case["requests"], pool.stream()
        ip, wq, wk = ids.data_ptr(), s["wq"].data_ptr(), s["wk"].data_ptr()
        for j in range(steps):
            qj, kj, vj, oj, ap = q[at + j], k[at + j], v[at + j], out[j], act[j].data_ptr()
            B.gp_step_begin(h, ip, n, ap, stream)
            for layer in range(case["layers"]):
                B.gp_attn_layer_qknorm(h, layer, ip, n, qj[layer].data_ptr(), kj[layer].data_ptr(), vj[layer].data_ptr(), wq, wk, 1e-6,
                                       oj[layer].data_ptr(), stream)
            B.gp_step_end(h, ip, n, ap, stream)
    else:
        for j in range(steps):
            pool.decode_step(ids, q[at + j], k[at + j], v[at + j], out[j], act[j])
    s["at"] = (at + steps) % len(q)
    return out, act


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def work(case):
    L, hq, hkv, d, n_req, steps = (case[x] for x in ("layers", "hq", "hkv", "d", "requests", "steps"))
    token = 4 * hkv * d                                        # K and V of one token and layer, bf16
    tokens = n_req * (case["lo"] + case["hi"]) / 2
    io = n_req * (2 * hq * d + token + 4 * hq * d)             # query and new key / value in, fp32 output out
    if case["kind"] == "dense":
        return {"bytes": tokens * token + n_req * 6 * hq * d, "flops": 4 * tokens * hq * d}
    # per step and layer: every retained key and value, the new row written, inputs and outputs, both fp64 summaries read and written
    step = L * (tokens * token + n_req * token + io + n_req * 2 * hq * d * 8 * 2)
    total, flops = steps * step, steps * L * 4 * tokens * hq * d
    if case["kind"] == "admit":
        total += 2 * L * tokens * token                        # prompts read once, pages written once
    if case["kind"] == "prefix":
        # the prompts in; and each request's own copy of its pages at its first compaction
        total += 2 * L * token * (tokens / case["group"] + tokens)
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Measured against the same attention in fp64: 1.7e-6 to 3.2e-6 for the decode step (fp32 sums of bf16 products, the
    # softmax weights carried as bf16 with their bf16 residual, largest difference 2.1e-5), 1.8e-7 for the dense entry point
    # (fp32 weights, largest difference 1.7e-6); four times that.  Actions are whole numbers and stay the same.
    if case["kind"] == "dense":
        return {"rel": 8e-7, "max": 7e-6}
    return {"rel": 1.3e-5, "max": 9e-5, "differ": 0.0}


# ---- the same in 64 bits --------------------------------------------------------------------------------------------
def _rotate(x, pos, theta):
    """Rotary embedding of the last dimension at a position (rotate-half pairing); theta 0: none."""
    if theta == 0.0:
        return x
    half = x.shape[-1] // 2
    ang = float(pos) * theta ** (-torch.arange(half, dtype=torch.float64, device=x.device) / half)
    c, s = ang.cos(), ang.sin()
    return torch.cat([x[..., :half] * c - x[..., half:] * s, x[..., half:] * c + x[..., :half] * s], dim=-1)


def _view(q, k):
    """Attention of a group's heads over candidate keys, each head its own softmax, averaged: [L][hkv][G][d], [L][hkv][n][d] -> [L][hkv][n]."""
    return torch.softmax(q @ k.transpose(-1, -2) / math.sqrt(q.shape[-1]), dim=-1).mean(dim=-2)


def _working_set(a, p=0.99):
    """Smallest number of weights whose sum reaches p, summed over layers and heads."""
    c = torch.cumsum(torch.sort(a, dim=-1, descending=True)[0], dim=-1)
    return int(torch.clamp((c < p).sum(dim=-1) + 1, max=a.shape[-1]).sum())


def _kept(s, page, k_loc):
    """Slots that stay when `page` of the candidates go: the k' best of every page, and the best of the rest; ascending."""
    n = s.shape[-1]
    blocks = -(-n // page)
    quota = min(k_loc, (n - page) // blocks)
    padded = torch.nn.functional.pad(s, (0, blocks * page - n), value=-1.0).unflatten(-1, (blocks, page))
    rank = torch.sort(torch.sort(padded, dim=-1, descending=True, stable=True)[1], dim=-1)[1].flatten(-2)[..., :n]
    order = torch.sort(torch.where(rank < quota, math.inf, s), dim=-1, descending=True, stable=True)[1]
    return torch.sort(order[..., :n - page], dim=-1)[0]


class _Request:
    """One request's retained keys and values (bf16, as the caller gave them) and its two query summaries in 64 bits."""

    def __init__(self, case, k, v, n, page):
        room = n + case["steps"] + page
        self.k, self.v = (torch.zeros((case["layers"], case["hkv"], room, case["d"]), dtype=torch.bfloat16, device=DEV) for _ in range(2))
        self.k[:, :, :n], self.v[:, :, :n] = k.transpose(1, 2), v.transpose(1, 2)
        self.n, self.pos, self.pages, self.short, self.long = n, n, n // page + 1, None, None


def exact(case, seed):
    """The outputs of a state's first pass in 64 bits.  None when that takes too long."""
    n_req, hq, hkv, d, steps, page, theta = (case[x] for x in ("requests", "hq", "hkv", "d", "steps", "page", "rope"))
    L, G, kind = case["layers"], hq // hkv, case["kind"]
    g, u, lens, fracs = _start(case, seed)
    if kind == "dense":
        q, k, v = _dense_inputs(case, u, g)
        out = torch.empty((n_req, hq, d), dtype=torch.float64, device=DEV)
        for i, n in enumerate(lens):
            z = q[i].double().view(hkv, G, d) @ k[i, :, :n].double().transpose(-1, -2) / math.sqrt(d)
            out[i] = (torch.softmax(z, dim=-1) @ v[i, :, :n].double()).view(hq, d)
        return out
    if steps * sum(lens) * L * hkv * d > 4e11 or steps * n_req * L * hq * d > 1.5e9:
        return None
    prompts = list(_prompts(case, u, lens, fracs, g))
    reqs = [_Request(case, *prompts[i // case["group"]], page) for i in range(n_req)]
    del prompts
    qs, ks, vs = _step_inputs(case, n_req, _ring(case), u, torch.tensor(fracs, device=DEV), g)
    weights = _norm_weights(case, g) if kind == "layers" else None
    n_pages, cap = _pages(case, lens)
    # (a prefix pool has pages for every copy and grant of the pass)
    free = 1 << 30 if kind == "prefix" else n_pages - sum(r.pages for r in reqs)
    out = torch.empty((steps, L, n_req, hq, d), dtype=torch.float64, device=DEV)
    for j in range(steps):
        for i, r in enumerate(reqs):
            q, k = qs[j][:, i].double(), ks[j][:, i].double()
            if weights:
                # normalised per head, rounded as a model rounds them, the key rotated before that
                q, k = (x / torch.sqrt((x * x).mean(dim=-1, keepdim=True) + 1e-6) * w.double() for x, w in zip((q, k), weights))
                q, k = q.float().bfloat16().double(), _rotate(k, r.pos, theta).float().bfloat16().double()
            r.k[:, :, r.n], r.v[:, :, r.n] = k.bfloat16(), vs[j][:, i]
            t, r.n, r.pos = r.pos, r.n + 1, r.pos + 1
            kk = r.k[:, :, :r.n].double()
            z = _rotate(q, t, theta).view(L, hkv, G, d) @ kk.transpose(-1, -2) / math.sqrt(d)
            out[j, :, i] = (torch.softmax(z, dim=-1) @ r.v[:, :, :r.n].double()).view(L, hq, d)
            r.short = q if r.short is None else 0.9 * r.short + (1.0 - 0.9) * q
            r.long = q if r.long is None else 0.999 * r.long + (1.0 - 0.999) * q
            if r.n < r.pages * page:
                continue
            # the capacity boundary: working sets under both summaries, then one more page, or one page of tokens evicted
            rms = lambda x: torch.sqrt((x * x).mean(dim=-1, keepdim=True))
            qs_, ql_ = (_rotate(rms(q) / rms(x) * x, t, theta).view(L, hkv, G, d) for x in (r.short, r.long))
            demand = kk[:, :, :r.n - page]
            r.wants = _working_set(_view(qs_, demand)) > _working_set(_view(ql_, demand))
            r.score = torch.maximum(_view(qs_, kk[:, :, :r.n - 16]), _view(ql_, kk[:, :, :r.n - 16]))
        for r in reqs:                                                      # ascending request id
            if r.n < r.pages * page:
                continue
            if r.wants and r.pages < cap and free > 0:
                r.pages, free = r.pages + 1, free - 1
                continue
            keep = torch.cat([_kept(r.score, page, case["k_loc"]), torch.arange(r.n - 16, r.n, device=DEV).expand(L, hkv, 16)], dim=-1)
            r.n -= page
            for x in (r.k, r.v):
                x[:, :, :r.n] = torch.gather(x, 2, keep[..., None].expand(-1, -1, -1, d))
    return out, None
