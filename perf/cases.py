"""Performance cases of the FLARE attention step, through the C ABI's Python binding.

Each case is one call (or the few calls of one pass) that a serving engine or a
training loop makes per layer.  Layer shapes:

  large   GDN 16 q/k and 32 value heads, d = 128; softmax 16 query / 2 kv heads,
          head dim 256; ShortConv over 8192 channels
  small   GDN 16 / 16 heads, d = 128; softmax 16 query / 4 kv heads, head dim 128
  tiny    GDN 2 / 2 heads, d = 64; softmax 2 query / 1 kv head, head dim 64

Inputs have the serving value distributions: q, k ~ N(0,1) L2-normalised per
head, v ~ N(0,1), log-gate -softplus(N(0,1)), beta = sigmoid(N(0,1)); softmax
q, k, v ~ N(0,1); committed states are the delta rule over random tokens; pages
lie at a random permutation of a shared pool.  Lengths (prefixes, accepted
lengths, held drafts) are spread evenly over their range and handed to the
requests in a random order, so that a case costs the same for every seed.
"""
import math

import torch

from paper_2606_01774_gb300 import flare

LAYERS = {
    "large": dict(hk=16, hv=32, d=128, hq=16, hkv=2, hd=256, channels=8192),
    "small": dict(hk=16, hv=16, d=128, hq=16, hkv=4, hd=128, channels=6144),
    "tiny": dict(hk=2, hv=2, d=64, hq=2, hkv=1, hd=64, channels=384),
}
# Tokens behind a committed state: the gates halve a state every token or so, so
# that older tokens no longer show in 32 bits.
STATE_TOKENS = 64
CHUNK = 64

MASKS = {"bidir": flare.FLARE_MASK_BLOCK_BIDIR, "causal": flare.FLARE_MASK_BLOCK_CAUSAL,
         "rows": flare.FLARE_MASK_ROW_TYPE_PER_REQUEST}


def listed():
    return [
        # One request in single precision, the numerical-parity setting: a denoise
        # pass of both layers and the commit of 5 accepted tokens.  Launch latency.
        dict(name="step_tiny_f32", kind="step", layer="tiny", dtype="f32", requests=1, block=8,
             lo=32, hi=32, page=16, accept_lo=5, accept_hi=5),
        # One interactive user: a denoise pass of both layers over a 4096-token
        # prefix, then the full-block commit.
        dict(name="step_single_request", kind="step", layer="large", dtype="bf16", requests=1,
             block=32, lo=4096, hi=4096, page=64, accept_lo=32, accept_hi=32),
        # Linear layer, denoise pass, of a 64-request serving batch.
        dict(name="linear_serving", kind="linear", layer="large", dtype="bf16", requests=64,
             block=32),
        # Linear layer, denoise pass, of a 128-request batch with blocks of 64.
        dict(name="linear_block64", kind="linear", layer="large", dtype="bf16", requests=128,
             block=64),
        # Softmax layer, denoise pass, of the serving batch over a ragged paged prefix.
        dict(name="softmax_serving", kind="softmax", layer="large", dtype="bf16", requests=64,
             block=32, lo=512, hi=8192, page=64, mask="bidir"),
        # The same over long prefixes with blocks of 64: the largest call.
        dict(name="softmax_block64", kind="softmax", layer="large", dtype="bf16", requests=128,
             block=64, lo=1024, hi=16384, page=64, mask="bidir"),
        # The small model's softmax layer: 256 requests, short blocks and prefixes.
        dict(name="softmax_small_model", kind="softmax", layer="small", dtype="bf16",
             requests=256, block=16, lo=256, hi=2048, page=64, mask="bidir"),
        # Commit of the recurrent state at ragged accepted lengths.
        dict(name="commit_block64", kind="commit", layer="large", dtype="bf16", requests=128,
             block=64, accept_lo=1, accept_hi=64),
        # State-update pass of the serving batch: commit with the token-causal
        # outputs that the next layer reads, and the block's keys and values
        # appended to the paged cache.
        dict(name="state_update_serving", kind="state_update", layer="large", dtype="bf16",
             requests=64, block=32, lo=512, hi=8192, page=64, accept_lo=32, accept_hi=32),
        # Verify round of the linear layer with a horizon of 16 (block 2 * 16 - 1):
        # verify pass with cached states, then the commit at the accepted offset.
        dict(name="verify_serving", kind="verify", layer="large", dtype="bf16", requests=64,
             horizon=16),
        # ShortConv in front of the serving batch's linear layer, with its commit.
        dict(name="shortconv_serving", kind="shortconv", layer="large", dtype="bf16",
             requests=64, block=32, commit=True),
        # Training forward of a linear layer, noisy stream: 4096 clean and 4096
        # noisy tokens in diffusion blocks of 4.
        dict(name="two_stream_train", kind="two_stream", layer="small", dtype="bf16", requests=1,
             block=4, length=4096),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "linear", "linear", "softmax", "softmax", "softmax", "commit",
                       "state_update", "verify", "shortconv", "two_stream"])
    layer = rng.choice(["large", "large", "small"])
    dtype = "bf16"
    if kind in ("step", "linear", "softmax", "commit") and rng.random() < 0.15:
        dtype, layer = "f32", "tiny"
    most = {"large": 128, "small": 256, "tiny": 16}[layer]
    c = dict(kind=kind, layer=layer, dtype=dtype)
    if kind == "two_stream":
        c.update(layer="small", requests=rng.choice([1, 1, 2, 3]), block=rng.choice([1, 2, 4, 8, 16]),
                 length=CHUNK * _log_int(rng, 1, 64))
        return c
    c["requests"] = _log_int(rng, 1, 4 if kind == "step" else most // 2 if kind == "verify" else most)
    if kind == "verify":
        c["horizon"] = rng.randint(2, 20)
        return c
    c["block"] = rng.choice([rng.randint(1, 64), 8, 16, 32, 64])
    if kind == "shortconv":
        c["commit"] = rng.random() < 0.5
    if kind in ("step", "commit", "state_update"):
        hi = rng.randint(1, c["block"])
        c.update(accept_lo=rng.randint(0, hi), accept_hi=hi)
    if kind in ("step", "softmax", "state_update"):
        top = {"large": 16384, "small": 4096, "tiny": 512}[layer]
        hi = _log_int(rng, 64, top)
        c.update(lo=rng.randint(0, hi // 2), hi=hi, page=rng.choice([16, 64, 64, 64]))
    if kind == "softmax":
        c["mask"] = rng.choice(["bidir", "bidir", "causal", "rows"])
    return c


# ---------------------------------------------------------------- inputs (plain torch)


def _spread(lo, hi, n, order):
    """n whole numbers spread evenly over [lo, hi], in the order given."""
    v = [lo + int((hi - lo + 1) * (2 * i + 1) / (2 * n)) for i in range(n)]
    return torch.tensor(v, dtype=torch.int32, device="cuda")[order]


def _lengths(lo, hi, n):
    return [lo + int((hi - lo + 1) * (2 * i + 1) / (2 * n)) for i in range(n)]


def _drafts(case):
    """Held drafts of each request, before they are put in order, and the drafts accepted."""
    held = _lengths(0, case["horizon"] - 1, case["requests"])
    return held, [(k + 1) * (i % 3) // 3 for i, k in enumerate(held)]


def _block(case):
    return 2 * case["horizon"] - 1 if case["kind"] == "verify" else case["block"]


def _type(case):
    return torch.bfloat16 if case["dtype"] == "bf16" else torch.float32


class _Draws:
    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda")
        self.gen.manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.gen, device="cuda")

    def order(self, n):
        return torch.randperm(n, generator=self.gen, device="cuda")


def _gdn(x, case, tokens):
    """q, k, v, log-gate and beta of `tokens` tokens of each request."""
    s, r, t = LAYERS[case["layer"]], case["requests"], _type(case)
    unit = lambda: torch.nn.functional.normalize(x.normal(r, tokens, s["hk"], s["d"]), dim=-1).to(t)  # noqa: E731
    return dict(q=unit(), k=unit(), v=x.normal(r, tokens, s["hv"], s["d"]).to(t),
                g=-torch.nn.functional.softplus(x.normal(r, tokens, s["hv"])),
                beta=torch.sigmoid(x.normal(r, tokens, s["hv"])))


def _delta_rule(state, b, tokens):
    """Yields the state after each of `tokens` tokens ([R, Hv, dk, dv], in the state's type)."""
    rep = state.shape[1] // b["k"].shape[2]
    for t in range(tokens):
        k = b["k"][:, t].to(state.dtype).repeat_interleave(rep, 1)
        v, g, beta = (b[n][:, t].to(state.dtype) for n in ("v", "g", "beta"))
        state = state * torch.exp(g)[..., None, None]
        u = v - torch.matmul(k[..., None, :], state)[..., 0, :]
        state = state + k[..., :, None] * (beta[..., None] * u)[..., None, :]
        yield state


def _readout(state, q, scale):
    """scale * S^T q: state [R, Hv, dk, dv], q [R, B, Hk, dk] -> [R, B, Hv, dv]."""
    rep = state.shape[1] // q.shape[2]
    q = q.to(state.dtype).repeat_interleave(rep, 2).transpose(1, 2)
    return scale * torch.matmul(q, state).transpose(1, 2)


def _inputs(case, seed):
    x = _Draws(seed)
    s, r, kind, t = LAYERS[case["layer"]], case["requests"], case["kind"], _type(case)
    i = {}
    if kind == "two_stream":
        n = case["length"]
        i["clean"], i["noisy"] = _gdn(x, case, n), _gdn(x, case, n)
        # the clean chunkwise pass's states at the chunk starts: each chunk is run
        # from zero (older tokens have decayed by its end), all of them at once
        c = n // CHUNK
        fold = {m: v.reshape(r * c, CHUNK, *v.shape[2:]) for m, v in i["clean"].items()}
        state = torch.zeros(r * c, s["hv"], s["d"], s["d"], device="cuda")
        for state in _delta_rule(state, fold, CHUNK):
            pass
        starts = torch.zeros(r, c, s["hv"], s["d"], s["d"], device="cuda")
        starts[:, 1:] = state.reshape(r, c, s["hv"], s["d"], s["d"])[:, :-1]
        i["chunk_states"] = starts.transpose(1, 2).contiguous()
        return i
    b, slots = _block(case), r + max(2, r // 16)
    i["slot"] = x.order(slots)[:r].to(torch.int32)
    if kind == "shortconv":
        ch = s["channels"]
        i["x"] = x.normal(r, b, ch).to(t)
        i["conv_state"] = x.normal(slots, 3, ch).to(t)
        i["weight"], i["bias"] = x.normal(ch, 4) / 2, 0.1 * x.normal(ch)
        i["accept"] = _spread(0, b, r, x.order(r)) if case["commit"] else None
        return i
    if kind in ("step", "linear", "commit", "state_update", "verify"):
        pool = torch.zeros(slots, s["hv"], s["d"], s["d"], device="cuda")
        state = torch.zeros(r, s["hv"], s["d"], s["d"], device="cuda")
        past = _gdn(x, case, STATE_TOKENS)
        for state in _delta_rule(state, past, STATE_TOKENS):
            pass
        pool[i["slot"].long()] = state
        i["pool"] = pool
        i["block"] = _gdn(x, case, b)
        if kind == "step":
            i["final"] = _gdn(x, case, b)
    if kind in ("step", "commit", "state_update"):
        i["accept"] = _spread(case["accept_lo"], case["accept_hi"], r, x.order(r))
    if kind == "verify":
        held, taken = (torch.tensor(v, dtype=torch.int32, device="cuda") for v in _drafts(case))
        order = x.order(r)
        i["held"], i["taken"] = held[order], taken[order]
    if kind in ("step", "softmax", "state_update"):
        page, room = case["page"], b if kind == "state_update" else 0
        i["prefix"] = _spread(case["lo"], case["hi"], r, x.order(r))
        need = [-(-(n + room) // page) for n in i["prefix"].tolist()]
        pages = sum(need) + max(4, sum(need) // 20)
        ids, table = x.order(pages).to(torch.int32), torch.full((r, max(max(need), 1)), -1, dtype=torch.int32)
        at, host = 0, ids.cpu()
        for n, row in zip(need, table):
            row[:n] = host[at:at + n]
            at += n
        i["table"] = table.cuda()
        i["k_pool"], i["v_pool"] = (torch.randn(pages, s["hkv"], page, s["hd"], generator=x.gen, device="cuda", dtype=t)
                                    for _ in range(2))
        i["k_blk"], i["v_blk"] = (x.normal(r, b, s["hkv"], s["hd"]).to(t) for _ in range(2))
        if kind != "state_update":
            i["sq"] = x.normal(r, b, s["hq"], s["hd"]).to(t)
    if kind == "softmax" and case["mask"] == "rows":
        # an anchor and its held drafts read causally, the rows after them the whole block
        held = _spread(0, b - 1, r, x.order(r))
        i["rows"] = (torch.arange(b, device="cuda", dtype=torch.int32)[None] > held[:, None]).to(torch.uint8)
    return i


# ---------------------------------------------------------------- the calls


def prepare(case, seed):
    i = _inputs(case, seed)
    s, r, kind = LAYERS[case["layer"]], case["requests"], case["kind"]
    code = flare.FLARE_DT_BF16 if case["dtype"] == "bf16" else flare.FLARE_DT_F32
    st = dict(i, kind=kind, status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if kind == "two_stream":
        st["desc"] = flare.two_stream_desc(r, case["length"], CHUNK, case["block"], s["hk"], s["hv"],
                                           s["d"], s["d"], code, s["d"] ** -0.5)
        st["out"] = torch.zeros_like(i["noisy"]["v"])
        return st
    b = _block(case)
    if kind == "shortconv":
        st["desc"] = flare.conv_desc(r, b, s["channels"], 4, i["conv_state"].shape[0], code)
        st["out"] = torch.zeros_like(i["x"])
        return st
    if "pool" in i:
        st["lin"] = flare.linear_desc(r, b, s["hk"], s["hv"], s["d"], s["d"], i["pool"].shape[0], code,
                                      s["d"] ** -0.5)
        st["lin_out"] = torch.zeros_like(i["block"]["v"])
    if kind == "verify":
        st["most"] = case["horizon"] - 1
        st["states"] = torch.zeros(r, st["most"], s["hv"], s["d"], s["d"], device="cuda")
    if "table" in i:
        st["smx"] = flare.softmax_desc(r, b, s["hq"], s["hkv"], s["hd"], case["page"], i["k_pool"].shape[0],
                                       i["table"].shape[1], code, s["hd"] ** -0.5,
                                       MASKS[case.get("mask", "bidir")], i.get("rows"))
    if "sq" in i:
        st["smx_out"] = torch.zeros_like(i["sq"])
        st["lse"] = torch.zeros(i["sq"].shape[:3], device="cuda")
        st["ws_bytes"] = flare.flare_softmax_workspace_size(st["smx"])
        st["ws"] = torch.empty(max(st["ws_bytes"], 1), dtype=torch.uint8, device="cuda")
    return st


def _linear(st):
    b = st["block"]
    flare.check(flare.flare_block_linear_attn(st["lin"], b["q"], b["k"], b["v"], b["g"], b["beta"], st["pool"],
                                              st["slot"], st["lin_out"], st["status"]), "linear")


def _softmax(st):
    flare.check(flare.flare_block_softmax_attn(st["smx"], st["sq"], st["k_blk"], st["v_blk"], st["k_pool"],
                                               st["v_pool"], st["table"], st["prefix"], st["smx_out"], st["lse"],
                                               st["ws"], st["ws_bytes"], st["status"]), "softmax")


def _commit(st, b, causal_out=None):
    flare.check(flare.flare_commit_state(st["lin"], b["q"], b["k"], b["v"], b["g"], b["beta"], st["pool"],
                                         st["slot"], st["accept"], causal_out, st["status"]), "commit")


def run(st):
    kind = st["kind"]
    if kind == "linear":
        _linear(st)
        return st["lin_out"]
    if kind == "softmax":
        _softmax(st)
        return st["smx_out"], st["lse"]
    if kind == "step":
        _linear(st)
        _softmax(st)
        _commit(st, st["final"])
        return st["lin_out"], st["smx_out"], st["lse"], st["pool"]
    if kind == "commit":
        _commit(st, st["block"])
        return st["pool"]
    if kind == "state_update":
        _commit(st, st["block"], st["lin_out"])
        flare.check(flare.flare_append_kv(st["smx"], st["k_blk"], st["v_blk"], st["k_pool"], st["v_pool"],
                                          st["table"], st["prefix"], st["accept"], st["status"]), "append")
        return st["lin_out"], st["pool"], st["k_pool"], st["v_pool"]
    if kind == "verify":
        b = st["block"]
        flare.check(flare.flare_verify_linear_attn(st["lin"], st["most"], b["q"], b["k"], b["v"], b["g"], b["beta"],
                                                   st["pool"], st["slot"], st["held"], st["lin_out"], st["states"],
                                                   st["status"]), "verify")
        flare.check(flare.flare_verify_commit(st["lin"], st["most"], [st["states"]], [st["pool"]], st["slot"],
                                              st["taken"], st["held"], st["status"]), "verify commit")
        return st["lin_out"], st["states"], st["pool"]
    if kind == "shortconv":
        flare.check(flare.flare_short_conv(st["desc"], st["x"], st["conv_state"], st["slot"], st["weight"],
                                           st["bias"], st["accept"], st["out"], st["status"]), "shortconv")
        return st["out"], st["conv_state"]
    c, n = st["clean"], st["noisy"]
    flare.check(flare.flare_two_stream_fwd(st["desc"], st["chunk_states"], c["k"], c["v"], c["g"], c["beta"], n["q"],
                                           n["k"], n["v"], n["g"], n["beta"], st["out"], st["status"]), "two stream")
    return st["out"]


# ---------------------------------------------------------------- work and accuracy


def work(case):
    s, r, kind = LAYERS[case["layer"]], case["requests"], case["kind"]
    e = 2 if case["dtype"] == "bf16" else 4
    hk, hv, d = s["hk"], s["hv"], s["d"]
    token = e * (hk * d + hv * d) + 8 * hv  # k, v and the gates
    state = hv * d * d * 4
    if kind == "two_stream":
        n = r * case["length"]
        return dict(bytes=n // CHUNK * state + n * (2 * token + e * (hk + hv) * d),
                    flops=n * hv * (8 * d * d + 4 * case["block"] * d))
    b = _block(case)
    if kind == "shortconv":
        ch = s["channels"]
        return dict(bytes=r * ch * e * (2 * b + 3 + (3 if case["commit"] else 0)) + ch * 20, flops=r * b * ch * 12)
    got = dict(bytes=0, flops=0)

    def add(nbytes, flops):
        got["bytes"] += nbytes
        got["flops"] += flops

    def linear():
        add(r * (state + b * (token + e * (hk + hv) * d)),
            r * hv * (4 * b * d * d + 4 * b * b * d + 2 * b * b * d))

    def commit(outputs):
        for n in _lengths(case["accept_lo"], case["accept_hi"], r):
            rows = b if outputs else n
            add((2 * state if n else state if outputs else 0) + rows * token +
                (b * e * (hk + hv) * d if outputs else 0),
                hv * rows * d * d * (6 if outputs else 4))

    def softmax():
        for n in _lengths(case["lo"], case["hi"], r):
            add(e * s["hd"] * (2 * s["hkv"] * (n + b) + 2 * b * s["hq"]) + 4 * b * s["hq"],
                4 * b * s["hq"] * s["hd"] * (n + b))

    if kind in ("step", "linear"):
        linear()
    if kind in ("step", "softmax"):
        softmax()
    if kind in ("step", "commit", "state_update"):
        commit(kind == "state_update")
    if kind == "state_update":
        for n in _lengths(case["accept_lo"], case["accept_hi"], r):
            add(4 * n * s["hkv"] * s["hd"] * e, 0)
    if kind == "verify":
        for k, a in zip(*_drafts(case)):
            add(state * (2 + k + (2 if a < k else 0)) + b * (token + e * (hk + hv) * d), hv * b * 6 * d * d)
    return got


def tolerance(case):
    # Measured against exact(): single precision up to 3e-7, states committed from
    # bf16 inputs 2.6e-6, bf16 outputs 1.7e-3 (one rounding) to 2.9e-3 (blocks of 64).
    if case["dtype"] == "f32":
        return {"rel": 1e-5, "max": 1e-4}
    if case["kind"] == "commit":
        return {"rel": 1.2e-5, "max": 5e-4}
    return {"rel": 1e-2, "max": 5e-2}


# ---------------------------------------------------------------- 64-bit values


def _exact_softmax(case, i):
    s, b, r = LAYERS[case["layer"]], _block(case), case["requests"]
    g, scale, f8 = s["hq"] // s["hkv"], s["hd"] ** -0.5, torch.float64
    out = torch.empty(r, b, s["hq"], s["hd"], dtype=f8, device="cuda")
    lse = torch.empty(r, b, s["hq"], dtype=f8, device="cuda")
    at = torch.arange(b, device="cuda")
    for n, p in enumerate(i["prefix"].tolist()):
        pages = i["table"][n, :-(-p // case["page"])].long()
        k, v = (torch.cat([i[m + "_pool"][pages].transpose(1, 2).reshape(-1, s["hkv"], s["hd"])[:p],
                           i[m + "_blk"][n]]).to(f8).transpose(0, 1) for m in ("k", "v"))  # [Hkv, P + B, D]
        q = i["sq"][n].to(f8).reshape(b, s["hkv"], g, s["hd"]).permute(1, 0, 2, 3).reshape(s["hkv"], b * g, s["hd"])
        z = scale * torch.matmul(q, k.transpose(1, 2))
        causal = torch.zeros(b, dtype=torch.bool, device="cuda")
        if case.get("mask") == "causal":
            causal[:] = True
        elif case.get("mask") == "rows":
            causal = i["rows"][n] == 0
        hide = causal[:, None] & (at[None] > at[:, None])  # block row, block key
        z[..., p:].masked_fill_(hide.repeat_interleave(g, 0)[None], -math.inf)
        l = torch.logsumexp(z, -1)
        o = torch.matmul(torch.exp_(z.sub_(l[..., None])), v)
        out[n] = o.reshape(s["hkv"], b, g, s["hd"]).permute(1, 0, 2, 3).reshape(b, s["hq"], s["hd"])
        lse[n] = l.reshape(s["hkv"], b, g).permute(1, 0, 2).reshape(b, s["hq"])
    return out, lse


def _exact_commit(case, i, b, causal):
    """The pool after the commit, and the token-causal outputs if asked for."""
    s, slot, f8 = LAYERS[case["layer"]], i["slot"].long(), torch.float64
    pool = i["pool"].to(f8)
    start = pool[slot]
    kept, outs = start.clone(), []
    for t, state in enumerate(_delta_rule(start, b, _block(case))):
        kept = torch.where((i["accept"] == t + 1)[:, None, None, None], state, kept)
        if causal:
            outs.append(_readout(state, b["q"][:, t:t + 1], s["d"] ** -0.5))
    pool[slot] = kept
    return pool, torch.cat(outs, 1) if causal else None


def _exact_linear(case, i):
    state = i["pool"][i["slot"].long()].to(torch.float64)
    for state in _delta_rule(state, i["block"], _block(case)):
        pass
    return _readout(state, i["block"]["q"], LAYERS[case["layer"]]["d"] ** -0.5)


def _exact_verify(case, i):
    s, slot, b, f8 = LAYERS[case["layer"]], i["slot"].long(), i["block"], torch.float64
    pool, r, n, most = i["pool"].to(f8), case["requests"], _block(case), case["horizon"] - 1
    states = torch.zeros(r, most, s["hv"], s["d"], s["d"], dtype=f8, device="cuda")
    start = pool[slot]
    kept, rows = start.clone(), []
    for t, state in enumerate(_delta_rule(start, b, n)):
        if t < most:
            states[:, t] = torch.where((i["held"] > t)[:, None, None, None], state, states[:, t])
        kept = torch.where((torch.where(i["taken"] < i["held"], i["taken"], i["held"]) == t)[:, None, None, None],
                           state, kept)
        rows.append(_readout(state, b["q"][:, t:t + 1], s["d"] ** -0.5))
    causal, whole = torch.cat(rows, 1), _readout(state, b["q"], s["d"] ** -0.5)
    out = torch.where((torch.arange(n, device="cuda")[None] <= i["held"][:, None])[..., None, None], causal, whole)
    pool[slot] = kept
    return out, states, pool


def _exact_shortconv(case, i):
    f8, b, slot = torch.float64, case["block"], i["slot"].long()
    line = torch.cat([i["conv_state"][slot], i["x"]], 1).to(f8)  # [R, 3 + B, C]
    w = i["weight"].to(f8)
    u = i["bias"].to(f8) + sum(w[:, lag] * line[:, 3 - lag:3 - lag + b] for lag in range(4))
    after = i["conv_state"].to(f8)
    if i["accept"] is not None:
        rows = i["accept"].long()[:, None] + torch.arange(3, device="cuda")
        after[slot] = torch.gather(line, 1, rows[..., None].expand(-1, -1, line.shape[2]))
    return u * torch.sigmoid(u), after


def _exact_two_stream(case, i):
    s, r, n, b, f8 = LAYERS[case["layer"]], case["requests"], case["length"], case["block"], torch.float64
    c = n // CHUNK
    fold = lambda v, m: v.reshape(r * c, m, CHUNK // m, *v.shape[2:])  # noqa: E731
    clean = {m: v.reshape(r * c, CHUNK, *v.shape[2:]) for m, v in i["clean"].items()}
    noisy = {m: fold(v, CHUNK // b) for m, v in i["noisy"].items()}  # [R * chunks, blocks, B, ...]
    state = i["chunk_states"].to(f8).transpose(1, 2).reshape(r * c, s["hv"], s["d"], s["d"])
    out = torch.empty(r * c, CHUNK // b, b, s["hv"], s["d"], dtype=f8, device="cuda")
    steps = _delta_rule(state, clean, CHUNK)
    for m in range(CHUNK // b):
        part = {x: v[:, m] for x, v in noisy.items()}
        for end in _delta_rule(state, part, b):
            pass
        out[:, m] = _readout(end, part["q"], s["d"] ** -0.5)
        for _ in range(b):
            state = next(steps)
    return out.reshape(r, n, s["hv"], s["d"])


def exact(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    if kind == "linear":
        return _exact_linear(case, i)
    if kind == "softmax":
        return _exact_softmax(case, i)
    if kind == "step":
        out, (smx, lse) = _exact_linear(case, i), _exact_softmax(case, i)
        return out, smx, lse, _exact_commit(case, i, i["final"], False)[0]
    if kind == "commit":
        return _exact_commit(case, i, i["block"], False)[0]
    if kind == "state_update":
        pool, out = _exact_commit(case, i, i["block"], True)
        for n, (p, m) in enumerate(zip(i["prefix"].tolist(), i["accept"].tolist())):
            at = p + torch.arange(m, device="cuda")
            page, row = i["table"][n].long()[at // case["page"]], at % case["page"]
            i["k_pool"][page, :, row] = i["k_blk"][n, :m]
            i["v_pool"][page, :, row] = i["v_blk"][n, :m]
        return out, pool, i["k_pool"].to(torch.float64), i["v_pool"].to(torch.float64)
    if kind == "verify":
        return _exact_verify(case, i)
    if kind == "shortconv":
        return _exact_shortconv(case, i)
    return _exact_two_stream(case, i)
