"""The performance cases of the chunk-causal attention library.

A case is a call, or a short run of calls, that a program makes through the
public binding (paper_2609_36757_gb300.fastvr) on data that is on the GPU:

  stream      a whole (short) video: reset, then per chunk one KV append and
              one attention call, with log-sum-exp
  chunk       the chunk that arrives late in a long stream: one append and one
              attention call over the cache that earlier chunks filled
  static      the allocation-free attention call on caches that the caller
              owns, over one or two visible key ranges of a ring
  oneshot     the training form's forward over a whole clip
  train_step  the training form's forward and backward over a whole clip
  one_step    the restoration update z_hat = z_lq - sigma * v

Sizes are the library's own workloads (480p, 720p, 1080p latent frames, the
64 x 64 latent tiles, the 1024 x 1024 training clip) or generic ones.  Inputs
are N(0, 1) in bf16, with the per-token U[0.5, 2] factors of the peaked
workload where the case says so.
"""
import math

import torch

from paper_2609_36757_gb300 import fastvr as FV

SIGMA = 0.75


# ------------------------------------------------------------------ cases
def _case(kind, name=None, **kw):
    c = {"kind": kind, "batch": 1, "heads": 12, "dim": 128, "tokens": 1024,
         "frames": 2, "window": -1, "chunks": 1, "last": 0, "peaked": False}
    if kind == "one_step":
        c = {"kind": kind, "n": 1 << 20, "dtype": "bf16"}
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest stream: three chunks of 2 x 64 tokens.  Nothing but
        # latency: six small launches and the host's share of each.
        _case("stream", "tiny-stream", heads=2, dim=64, tokens=64, chunks=3),
        # A 480p video from its first chunk to its eighth, every chunk over
        # all earlier ones: ragged tiles, short and middling key ranges.
        _case("stream", "480p-stream", tokens=30 * 53, chunks=8),
        # The eighth chunk of a 720p video with peaked softmax rows.
        _case("chunk", "720p-peaked-chunk", tokens=45 * 80, chunks=8,
              peaked=True),
        # The fifteenth chunk of a 1080p video, the largest: 244 800 keys.
        _case("chunk", "1080p-chunk", tokens=68 * 120, chunks=15),
        # The end of a long windowed 1080p video: the ring has wrapped many
        # times and the last chunk holds one frame of three.
        _case("chunk", "1080p-windowed-end", heads=24, tokens=68 * 120,
              frames=3, window=4, chunks=40, last=1),
        # Steady state of tiled restoration: six overlapping tiles of
        # 32 x 32 tokens batched, Eq. 1 itself (chunks of 3, one predecessor).
        _case("chunk", "tiles-32-chunk", batch=6, heads=24, tokens=32 * 32,
              frames=3, window=1, chunks=9),
        # A serving engine with caches of its own: a 480p chunk over a ring
        # of three chunks that has wrapped (two key ranges).
        _case("static", "static-480p-ring", tokens=30 * 53, window=2,
              chunks=5, last=1),
        # A narrow-head model (d = 64) on odd frames, three videos at once.
        _case("chunk", "d64-chunk", batch=3, heads=16, dim=64, tokens=1155,
              frames=3, window=2, chunks=7),
        # Validation on the 1024 x 1024 training clip: 12 latent frames of
        # 32 x 32 tokens at once, forward only.
        _case("oneshot", "clip-forward", heads=24, tokens=32 * 32, frames=3,
              window=1, chunks=4),
        # A training step's attention on that clip: forward and backward.
        _case("train_step", "clip-train-step", heads=24, tokens=32 * 32,
              frames=3, window=1, chunks=4),
        # Training on small crops with narrow heads: two clips of 11 latent
        # frames (the last chunk is short) of 16 x 16 tokens.
        _case("train_step", "crop-train-step", batch=2, heads=12, dim=64,
              tokens=16 * 16, frames=3, window=1, chunks=4, last=2),
        # The update of a 1080p video's latent: 30 frames x 48 channels.
        _case("one_step", "one-step-1080p", n=48 * 30 * 68 * 120),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["stream", "chunk", "chunk", "static", "oneshot",
                       "train_step", "train_step", "one_step"])
    if kind == "one_step":
        return _case(kind, n=_log_int(rng, 1000, 200_000_000),
                     dtype=rng.choice(["bf16", "fp32"]))
    while True:
        c = _case(kind, batch=rng.choice([1, 1, 1, 2, 3, 6]),
                  heads=rng.choice([1, 2, 3, 5, 8, 12, 12, 16, 24, 24]),
                  dim=rng.choice([64, 128, 128]),
                  tokens=_log_int(rng, 60, 8160 if kind in ("chunk", "static")
                                  else 2500),
                  frames=rng.randint(1, 4),
                  window=rng.choice([-1, -1, 0, 1, 1, 2, 4]),
                  chunks=rng.randint(2, 8) if kind != "chunk"
                  else rng.randint(2, 15),
                  peaked=rng.random() < 0.25)
        if rng.random() < 0.4:
            c["last"] = rng.randint(1, c["frames"])
        w = work(c)
        if 1e7 <= w["flops"] <= 1.5e13 and w["bytes"] <= 3e9:
            return c


# ------------------------------------------------------------------ sizes
def _frames_in(c, i):
    return c["last"] if i == c["chunks"] - 1 and c["last"] else c["frames"]


def _length(c, i):
    return _frames_in(c, i) * c["tokens"]


def _first_visible(c, i):
    return 0 if c["window"] < 0 else max(0, i - c["window"])


def _visible(c, i):
    return sum(_length(c, j) for j in range(_first_visible(c, i), i + 1))


def _config(c):
    return FV.make_config(c["batch"], c["heads"], c["dim"], c["tokens"],
                          c["frames"], c["window"],
                          c["chunks"] if c["window"] < 0 else 0)


def work(c):
    """Bytes: every input read once and every output written once (an append
    reads and writes K and V; attention reads Q and the visible K and V and
    writes O and the log-sum-exp).  Flops: 4 d per visible (query, key) pair
    and head forward, 10 d backward."""
    if c["kind"] == "one_step":
        e = 2 if c["dtype"] == "bf16" else 4
        return {"bytes": c["n"] * (2 * e + 2), "flops": 2 * c["n"]}
    bh, d = c["batch"] * c["heads"], c["dim"]
    row = 2 * bh * d  # bytes of one token's row, all heads
    last = c["chunks"] - 1
    if c["kind"] in ("oneshot", "train_step"):
        L = sum(_length(c, i) for i in range(c["chunks"]))
        pairs = sum(_length(c, i) * _visible(c, i) for i in range(c["chunks"]))
        nbytes, flops = 4 * L * row + 4 * bh * L, 4.0 * bh * d * pairs
        if c["kind"] == "train_step":  # q k v o do lse in, dq dk dv out
            nbytes += 8 * L * row + 4 * bh * L
            flops += 10.0 * bh * d * pairs
        return {"bytes": nbytes, "flops": flops}
    nbytes = flops = 0.0
    for i in range(c["chunks"]) if c["kind"] == "stream" else [last]:
        lq, lk = _length(c, i), _visible(c, i)
        nbytes += 2 * lq * row + 2 * lk * row + 4 * bh * lq
        if c["kind"] != "static":
            nbytes += 4 * lq * row
        flops += 4.0 * bh * d * lq * lk
    return {"bytes": nbytes, "flops": flops}


# ----------------------------------------------------------------- inputs
def _randn(c, seed, what, i):
    """Chunk i's rows of q, k, v or do: bf16 [B, f_i N, H, d]."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 4 * i + "qkvg".index(what))
    shape = (c["batch"], _length(c, i), c["heads"], c["dim"])
    x = torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)
    if c["peaked"] and what in "qk":
        x *= (0.5 + 1.5 * torch.rand(shape[:2], generator=g, device="cuda")
              )[:, :, None, None]
    return x.to(torch.bfloat16)


def _sequence(c, seed, what):
    return torch.cat([_randn(c, seed, what, i) for i in range(c["chunks"])], 1)


def _latents(c, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + 17)
    z = torch.randn(c["n"], generator=g, device="cuda", dtype=torch.float32)
    v = torch.randn(c["n"], generator=g, device="cuda", dtype=torch.float32)
    if c["dtype"] == "bf16":
        z = z.to(torch.bfloat16)
    return z, v.to(torch.bfloat16)


def prepare(c, seed):
    kind, last = c["kind"], c["chunks"] - 1 if "chunks" in c else 0
    s = {"case": c}
    if kind == "one_step":
        s["z"], s["v"] = _latents(c, seed)
        return s
    s["cfg"] = _config(c)
    if kind in ("oneshot", "train_step"):
        for what in "qkv" + ("g" if kind == "train_step" else ""):
            s[what] = _sequence(c, seed, what)
        return s
    if kind == "static":
        # the caller's ring: W + 1 slots (all chunks without a window),
        # chunk i in slot i mod S, head-major
        slots = c["chunks"] if c["window"] < 0 else c["window"] + 1
        span = c["frames"] * c["tokens"]
        s["q"] = _randn(c, seed, "q", last)
        for what in "kv":
            cache = torch.zeros((c["batch"], c["heads"], slots * span, c["dim"]),
                                dtype=torch.bfloat16, device="cuda")
            for i in range(_first_visible(c, last), last + 1):
                at = i % slots * span
                cache[:, :, at:at + _length(c, i)] = \
                    _randn(c, seed, what, i).transpose(1, 2)
            s[what] = cache
        segs = []
        for at, n in sorted((i % slots * span, _length(c, i))
                            for i in range(_first_visible(c, last), last + 1)):
            if segs and sum(segs[-1]) == at:
                segs[-1] = (segs[-1][0], segs[-1][1] + n)
            else:
                segs.append((at, n))
        s["segments"], s["cache_tokens"] = segs, slots * span
        s["out"] = torch.empty_like(s["q"])
        s["lse"] = torch.empty((c["batch"], c["heads"], s["q"].shape[1]),
                               dtype=torch.float32, device="cuda")
        return s
    s["att"] = FV.StreamingAttention(s["cfg"])
    if kind == "stream":
        s["chunks"] = [tuple(_randn(c, seed, w, i) for w in "qkv")
                       for i in range(c["chunks"])]
        return s
    # chunk: the visible earlier chunks are in the cache
    first = _first_visible(c, last)
    s["att"].set_state(first, c["frames"] if first else 0)
    for i in range(first, last):
        s["att"].append(_randn(c, seed, "k", i), _randn(c, seed, "v", i))
    s["chunks"] = [tuple(_randn(c, seed, w, last) for w in "qkv")]
    return s


def _cache_views(s, last_only):
    """The appended K and V as the cache holds them (bit patterns), token
    range of the last chunk or the whole of what the stream filled."""
    c, att = s["case"], s["att"]
    span = c["frames"] * c["tokens"]
    slots = c["chunks"] if c["window"] < 0 else c["window"] + 1
    shape = (c["batch"], c["heads"], slots * span, c["dim"])
    n = math.prod(shape)
    region = (2 * n + 255) // 256 * 256
    k, v = (att.cache[at:at + 2 * n].view(torch.int16).view(shape)
            for at in (0, region))
    last = c["chunks"] - 1
    if last_only:
        at = last % slots * span
        return [x[:, :, at:at + _length(c, last)] for x in (k, v)]
    parts = []
    for slot in range(min(slots, c["chunks"])):
        i = max(j for j in range(c["chunks"]) if j % slots == slot)
        parts.append((slot * span, _length(c, i)))
    return [x[:, :, at:at + n] for x in (k, v) for at, n in parts]


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "one_step":
        return FV.one_step_update(s["z"], s["v"], SIGMA)
    if kind == "oneshot":
        return FV.blockcausal_attention(s["cfg"], s["q"], s["k"], s["v"],
                                        want_lse=True)
    if kind == "train_step":
        o, lse = FV.blockcausal_attention(s["cfg"], s["q"], s["k"], s["v"],
                                          want_lse=True)
        return (o, lse) + FV.blockcausal_attention_bwd(
            s["cfg"], s["q"], s["k"], s["v"], o, s["g"], lse)
    if kind == "static":
        FV.fastvr_chunk_attn_fwd_static(
            s["cfg"], s["q"].data_ptr(), s["q"].shape[1] // c["tokens"],
            s["k"].data_ptr(), s["v"].data_ptr(), s["cache_tokens"],
            s["segments"], s["out"].data_ptr(), s["lse"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        return s["out"], s["lse"]
    att, outs = s["att"], []
    if kind == "stream":
        att.reset()
    else:  # back to the state before the late chunk
        last = c["chunks"] - 1
        att.set_state(last, c["frames"] if last else 0)
    for q, k, v in s["chunks"]:
        att.append(k, v)
        outs.extend(att.forward(q, want_lse=True))
    return outs + _cache_views(s, kind == "chunk")


# -------------------------------------------------- tolerance and 64 bits
def tolerance(c):
    """Attention: bf16 inputs, P (and dS) rounded to bf16 before the second
    product, outputs rounded to bf16 (2^-9 relative each).  Against 64 bits
    the outputs and the gradients are about 3e-3 off; two correct
    implementations differ by at most that, and four times as much is 1e-2.
    The cache holds copies of bits.  The update is one fp32 FMA, rounded
    once: the same bits in any implementation."""
    if c["kind"] == "one_step":
        return "exact"
    return {"rel": 1e-2, "max": 0.3}


_EXACT_FLOPS = 8e12  # about 10 s of 64-bit products on the GPU


def _attend(q, k, v, scale):
    """64-bit softmax attention of [H, Lq, d] over [H, Lk, d], by rows."""
    outs, lses = [], []
    step = max(1, int(2.5e8 // (q.shape[0] * k.shape[1])))
    for r in range(0, q.shape[1], step):
        sc = torch.einsum("hqd,hkd->hqk", q[:, r:r + step], k) * scale
        l = torch.logsumexp(sc, -1)
        outs.append(torch.exp(sc - l[..., None]) @ v)
        lses.append(l)
    return torch.cat(outs, 1), torch.cat(lses, 1)


def _attend_bwd(q, k, v, g, scale):
    """64-bit dq, dk, dv of the same, by rows."""
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v)
    step = max(1, int(2e8 // (q.shape[0] * k.shape[1])))
    for r in range(0, q.shape[1], step):
        qr, gr = q[:, r:r + step], g[:, r:r + step]
        p = torch.softmax(torch.einsum("hqd,hkd->hqk", qr, k) * scale, -1)
        dp = torch.einsum("hqd,hkd->hqk", gr, v)
        ds = p * (dp - (p * dp).sum(-1, keepdim=True))
        dq[:, r:r + step] = ds @ k * scale
        dk += ds.transpose(1, 2) @ qr * scale
        dv += p.transpose(1, 2) @ gr
    return dq, dk, dv


def _wide(x):
    return x.double().transpose(1, 2)  # [B, H, L, d]


def exact(c, seed):
    if c["kind"] == "one_step":
        z, v = _latents(c, seed)
        return z.double() - SIGMA * v.double()
    if work(c)["flops"] > _EXACT_FLOPS:
        return None
    scale = c["dim"] ** -0.5
    last = c["chunks"] - 1

    def attend_chunk(i):
        lo = _first_visible(c, i)
        q = _wide(_randn(c, seed, "q", i))
        k, v = (_wide(torch.cat([_randn(c, seed, w, j)
                                 for j in range(lo, i + 1)], 1)) for w in "kv")
        o, l = zip(*(_attend(q[b], k[b], v[b], scale)
                     for b in range(c["batch"])))
        return torch.stack(o).transpose(1, 2), torch.stack(l)

    if c["kind"] in ("chunk", "static"):
        o, l = attend_chunk(last)
        return (o, l) if c["kind"] == "static" else [o, l, None, None]
    if c["kind"] == "stream":
        outs = [x for i in range(c["chunks"]) for x in attend_chunk(i)]
        slots = c["chunks"] if c["window"] < 0 else c["window"] + 1
        return outs + [None] * (2 * min(slots, c["chunks"]))
    parts = [attend_chunk(i) for i in range(c["chunks"])]
    o, l = torch.cat([p[0] for p in parts], 1), torch.cat([p[1] for p in parts], 2)
    if c["kind"] == "oneshot":
        return o, l
    q, k, v, g = (_wide(_sequence(c, seed, w)) for w in "qkvg")
    dq, dk, dv = torch.zeros_like(q), torch.zeros_like(k), torch.zeros_like(v)
    at = [0]
    for i in range(c["chunks"]):
        at.append(at[-1] + _length(c, i))
    for b in range(c["batch"]):
        for i in range(c["chunks"]):
            rows = slice(at[i], at[i + 1])
            keys = slice(at[_first_visible(c, i)], at[i + 1])
            x, y, z = _attend_bwd(q[b, :, rows], k[b, :, keys], v[b, :, keys],
                                  g[b, :, rows], scale)
            dq[b, :, rows] += x
            dk[b, :, keys] += y
            dv[b, :, keys] += z
    return (o, l) + tuple(x.transpose(1, 2) for x in (dq, dk, dv))
