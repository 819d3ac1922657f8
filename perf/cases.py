"""Performance cases of the archive: what a user's program has the library do,
through the Python binding, with the inputs that program has in hand.

Kinds of pass:
  write     a K/V cache's archived positions quantised into token records
            (rvq_encode of keys and of values): the archive's tensor-core half
  append    one decode step: the position leaving the exact window is quantised
            and appended to every stream
  restore   a whole archive decoded and rebuilt into K/V caches (decode_kv)
  records   random token records rebuilt from the archive (read_kv)
  codec     symbol streams encoded, decoded and read at random positions
            (one length per stream set, or a ragged batch)
  lossy     an archive's older spans truncated, decoded and read at random
  weighted  index streams arithmetic-coded and decoded back

Shapes are those of the repository's own configurations (GPT-2-shaped: 12
layers x 12 heads x 64; Llama-3-8B-shaped: 8 KV heads x 128; 4 sink + 32 recent
positions stay outside the archive), with fewer layers where the layer count
only repeats the same work.  Inputs are Gaussian with outlier key channels (and
log-normal channel scales for 128-dimensional heads), codebooks are drawn from
the same per-channel distribution, shrinking by 0.85 per stage.
"""
import math

import numpy as np
import torch

import paper_2607_07144_gb300 as fkv

SINKS, RECENT = 4, 32
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
K_ID, V_ID = 0, 1


# ------------------------------------------------------------------ cases --
def _kv(name, kind, layers, batch, heads, dim, positions, dtype, stages_k, stages_v, codewords=256, pooled=False,
        **more):
    return dict(name=name, kind=kind, layers=layers, batch=batch, heads=heads, dim=dim, positions=positions,
                dtype=dtype, stages_k=stages_k, stages_v=stages_v, codewords=codewords, pooled=pooled, **more)


def listed():
    return [
        # one layer of one sequence leaves the window: the smallest archive write (latency)
        _kv("write_gpt2_layer_f32", "write", 1, 1, 12, 64, 988, "f32", 2, 1),
        # a GPT-2-shaped batch archived whole, the paper's hybrid bit allocation
        _kv("write_gpt2_cache_f16", "write", 12, 8, 12, 64, 988, "f16", 4, 2),
        # the same cache with one 1024-codeword codebook per layer (uint16 symbols)
        _kv("write_gpt2_pooled1024", "write", 12, 8, 12, 64, 988, "f16", 2, 2, 1024, True),
        # long Llama-shaped prefill archived: the largest write
        _kv("write_llama_bf16", "write", 8, 4, 8, 128, 16348, "bf16", 4, 2),
        # a decode step of 64 Llama-shaped sequences, all 32 layers
        _kv("append_llama_step", "append", 32, 64, 8, 128, 1, "bf16", 4, 2, prefill=61),
        # a Llama-shaped archive brought back for attention over the whole past
        _kv("restore_llama_bf16", "restore", 8, 4, 8, 128, 16348, "bf16", 4, 2),
        # a few retrieved positions of a GPT-2-shaped batch (latency)
        _kv("records_few_gpt2", "records", 12, 8, 12, 64, 988, "f16", 4, 2, requests=96),
        # every sequence of a decode step retrieves its share of past positions
        _kv("records_many_llama", "records", 8, 64, 8, 128, 2048, "bf16", 4, 2, requests=131072),
        # the archive's index streams through the symbol codec, with position reads
        dict(name="codec_archive_256", kind="codec", alphabet=256, streams=128, symbols=48 * 8183, dist="uniform",
             ragged=False, reads=65536),
        # a serving batch of unequal sequences over a small, skewed alphabet
        dict(name="codec_ragged_16", kind="codec", alphabet=16, streams=64, symbols=(1 << 24) + 5, dist="zipf",
             ragged=True, reads=8191),
        # older spans kept at 24 bits per coordinate, the recent ones exact
        dict(name="lossy_24bit", kind="lossy", alphabet=256, streams=96, symbols=71136, bits=24, keep=512,
             reads=4096),
        # index streams stored as one arithmetic code each (adaptive model)
        dict(name="weighted_adaptive", kind="weighted", alphabet=256, streams=96, symbols=17784, dist="zipf",
             adaptive=True),
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], uniform over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["write", "write", "append", "restore", "records", "codec", "codec", "lossy", "weighted"])
    if kind == "codec":
        n = rng.choice([3, 4, 16, 64, 256, 300, 512, 1024])
        total = _spread(rng, 1 << 12, 50_000_000)
        streams = _spread(rng, 1, min(128, total // 64))
        ragged = rng.random() < 0.5
        return dict(kind=kind, alphabet=n, streams=streams, symbols=total if ragged else max(1, total // streams),
                    dist=rng.choice(["uniform", "zipf"]), ragged=ragged, reads=_spread(rng, 16, 65536))
    if kind == "lossy":
        n = rng.choice([16, 256, 1024])
        return dict(kind=kind, alphabet=n, streams=_spread(rng, 1, 96), symbols=_spread(rng, 500, 71136),
                    bits=rng.choice([12, 16, 24, 32, 42]), keep=rng.choice([0, 32, 512]),
                    reads=_spread(rng, 16, 4096))
    if kind == "weighted":
        return dict(kind=kind, alphabet=rng.choice([16, 256, 1024]), streams=_spread(rng, 1, 96),
                    symbols=_spread(rng, 256, 17784), dist=rng.choice(["uniform", "zipf"]),
                    adaptive=rng.random() < 0.75)
    dim = rng.choice([64, 128])
    heads = rng.choice([8, 12, 16] if dim == 64 else [4, 8])
    codewords, pooled = 256, rng.random() < 0.15
    if dim == 64 and rng.random() < 0.3:
        codewords, pooled = 1024, rng.random() < 0.8
    sk = rng.randint(1, 2 if codewords == 1024 else 4)
    sv = rng.randint(1, 2)
    dtype = rng.choice(["f16", "bf16", "bf16", "f32"])
    layers = _spread(rng, 1, 12 if dim == 64 else 8)
    batch = _spread(rng, 1, 8)
    case = _kv(None, kind, layers, batch, heads, dim, 1, dtype, sk, sv, codewords, pooled)
    del case["name"]
    if kind == "append":
        case.update(batch=_spread(rng, 1, 64), prefill=rng.randint(1, 64))
        return case
    most = max(64, 3_000_000 // (layers * batch * heads) * 64 // dim)
    case["positions"] = _spread(rng, 33, min(16348, most))
    if kind == "records":
        case["requests"] = _spread(rng, 1, 131072)
    return case


# ----------------------------------------------------------------- inputs --
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 64 + stream)
    return g


def _scales(case, seed, kv):
    """Per-(layer, head, channel) standard deviation, float32 [layers, heads, dim]."""
    shape = (case["layers"], case["heads"], case["dim"])
    g = _gen(seed, 1 + kv)
    sig = torch.ones(shape, device="cuda")
    wide = case["dim"] == 128
    if wide:
        sig *= torch.exp(0.5 * torch.randn(shape, device="cuda", generator=g))
    if kv == K_ID:
        n = 3 if wide else 4
        ch = torch.rand(shape, device="cuda", generator=g).topk(n, dim=2).indices
        mul = torch.ones(shape, device="cuda").scatter_(2, ch, 10.0 if wide else 8.0)
        sig *= mul
    return sig


def _codebook(case, seed, kv, sig):
    """float32 [layers, heads (1 when pooled), stages, codewords, dim] on the GPU."""
    S, K = case["stages_k" if kv == K_ID else "stages_v"], case["codewords"]
    L, H, D = sig.shape
    cb = torch.randn((L, 1 if case["pooled"] else H, S, K, D), device="cuda", generator=_gen(seed, 3 + kv))
    shrink = (0.85 ** torch.arange(S, device="cuda", dtype=torch.float32)).view(1, 1, S, 1, 1)
    if case["pooled"]:      # codeword j stands for head j mod heads
        own = sig[:, torch.arange(K, device="cuda") % H].view(L, 1, 1, K, D)
    else:
        own = sig.view(L, H, 1, 1, D)
    return cb * own * shrink


def _cache(case, seed, kv, sig, positions):
    """[layers, batch, heads, positions + window, dim] in the case's dtype."""
    L, H, D = sig.shape
    T = positions + SINKS + RECENT
    x = torch.empty((L, case["batch"], H, T, D), dtype=DTYPES[case["dtype"]], device="cuda")
    g = _gen(seed, 5 + kv)
    for layer in range(L):
        for b in range(case["batch"]):
            x[layer, b] = torch.randn((H, T, D), device="cuda", generator=g) * sig[layer].view(H, 1, D)
    return x


def _codebooks(case, seed):
    return [_codebook(case, seed, kv, _scales(case, seed, kv)) for kv in (K_ID, V_ID)]


def _context(case, books):
    host = [b.cpu().numpy() for b in books]
    return fkv.Context(case["codewords"], codebooks=host, pooled=case["pooled"],
                       n_heads=case["heads"] if case["pooled"] else None)


def _record_len(case):
    return case["heads"] * (case["stages_k"] + case["stages_v"])


def _indices(case, seed, records, stream=8):
    """Random token records int64 [batch * layers, records * R] (RVQ indices are near uniform)."""
    return torch.randint(0, case["codewords"], (case["batch"] * case["layers"], records * _record_len(case)),
                         device="cuda", generator=_gen(seed, stream))


def _sym_dtype(alphabet):
    return torch.uint8 if alphabet <= 256 else torch.int16


def _symbols(case, seed, shape):
    n, g = case["alphabet"], _gen(seed, 9)
    if case.get("dist", "uniform") == "uniform":
        return torch.randint(0, n, shape, device="cuda", generator=g).to(_sym_dtype(n))
    w = torch.arange(1, n + 1, device="cuda", dtype=torch.float64) ** -1.1
    cdf = (w.cumsum(0) / w.sum()).float()
    u = torch.rand(shape, device="cuda", generator=g)
    return torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1).to(_sym_dtype(n))


def _lengths(case):
    """Stream lengths of a ragged batch: spread over a factor of about 50, adding up to the case's symbols."""
    rng = np.random.default_rng([case["streams"], case["symbols"], case["alphabet"]])
    w = np.exp(rng.uniform(0.0, 4.0, case["streams"]))
    n = np.maximum(1, (w / w.sum() * case["symbols"]).astype(np.int64))
    n[np.argmax(n)] += case["symbols"] - n.sum()
    return n


def _requests(case, seed, streams, lengths, count):
    """int64 [count, 2] = (stream, position), uniform."""
    g = _gen(seed, 10)
    s = torch.randint(0, streams, (count,), device="cuda", generator=g)
    u = torch.rand(count, device="cuda", generator=g, dtype=torch.float64)
    ln = torch.as_tensor(lengths, device="cuda").expand(streams)[s] if np.ndim(lengths) == 0 else \
        torch.as_tensor(lengths, device="cuda")[s]
    return torch.stack([s, (u * ln).to(torch.int64)], dim=1).contiguous()


class _Points:
    """The point buffer of a stream set, which lives as long as a tensor over it does."""

    def __init__(self, streams):
        n, _, stride, ptr = streams.info()
        self.owner = streams
        self.__cuda_array_interface__ = {"shape": (n, stride, 2), "typestr": "<f8", "data": (ptr, False),
                                         "version": 3, "strides": None}


# -------------------------------------------------------------- preparing --
def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("codec", "lossy", "weighted"):
        ctx = st["ctx"] = fkv.Context(case["alphabet"])
        ns, n = case["streams"], case["symbols"]
        if case.get("ragged"):
            lengths = _lengths(case)
            st["sym"] = _symbols(case, seed, (int(lengths.sum()),))
            st["so"], st["po"] = ctx.ragged_offsets(lengths)
            st["pts"] = torch.empty((int(((lengths + ctx.L - 1) // ctx.L).sum()), 2), dtype=torch.float64,
                                    device="cuda")
        else:
            lengths = n
            st["sym"] = _symbols(case, seed, (ns, n))
            st["pts"] = torch.empty((ns, ctx.n_spans(n), 2), dtype=torch.float64, device="cuda")
        st["back"] = torch.empty_like(st["sym"])
        if "reads" in case:
            st["req"] = _requests(case, seed, ns, lengths, case["reads"])
            st["out"] = torch.empty(case["reads"], dtype=ctx.sym_dtype, device="cuda")
        if kind == "lossy":
            ctx.span_encode(st["sym"], st["pts"])
        return st

    books = _codebooks(case, seed)
    ctx = st["ctx"] = _context(case, books)
    L, B, H, D, P = (case[k] for k in ("layers", "batch", "heads", "dim", "positions"))
    R, ns = _record_len(case), case["layers"] * case["batch"]
    if kind in ("write", "append"):
        st["x"] = [_cache(case, seed, kv, _scales(case, seed, kv), P) for kv in (K_ID, V_ID)]
        st["sym"] = torch.empty((ns, P * R), dtype=ctx.sym_dtype, device="cuda")
    if kind == "append":
        # room for 512 further steps, after which the sequences are replaced
        past = _indices(case, seed, case["prefill"]).to(ctx.sym_dtype)
        st["room"] = (case["prefill"] + 512) * R
        st["streams"] = fkv.Streams(ctx, ns, st["room"])
        st["streams"].append(past)
        st["length"] = case["prefill"] * R
        st["view"] = torch.as_tensor(_Points(st["streams"]), device="cuda")
    if kind in ("restore", "records"):
        sym = _indices(case, seed, P).to(ctx.sym_dtype)
        st["pts"] = ctx.span_encode(sym)
    if kind == "restore":
        shape = (L, B, H, P + SINKS + RECENT, D)
        st["y"] = [torch.zeros(shape, dtype=DTYPES[case["dtype"]], device="cuda") for _ in (K_ID, V_ID)]
    if kind == "records":
        st["req"] = _requests(case, seed, ns, P, case["requests"])
        st["out"] = torch.empty((case["requests"], 2, H, D), dtype=DTYPES[case["dtype"]], device="cuda")
    return st


# ---------------------------------------------------------------- running --
def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind == "write":
        for kv in (K_ID, V_ID):
            ctx.rvq_encode(kv, st["x"][kv], SINKS, SINKS + case["positions"], st["sym"])
        return {"sym": st["sym"]}
    if kind == "append":
        s = st["streams"]
        if st["length"] + st["sym"].shape[1] > st["room"]:
            s.reset()
            st["length"] = 0
        for kv in (K_ID, V_ID):
            ctx.rvq_encode(kv, st["x"][kv], SINKS, SINKS + 1, st["sym"])
        s.append(st["sym"])
        st["length"] += st["sym"].shape[1]
        return {"sym": st["sym"], "pts": st["view"][:, :ctx.n_spans(st["length"])]}
    if kind == "restore":
        ctx.decode_kv(st["pts"], case["positions"], st["y"][K_ID], st["y"][V_ID], t0=SINKS)
        return {"k": st["y"][K_ID], "v": st["y"][V_ID]}
    if kind == "records":
        return {"kv": ctx.read_kv(st["pts"], case["positions"], st["req"], st["out"])}
    if kind == "codec":
        if case["ragged"]:
            pts = ctx.span_encode_ragged(st["sym"], st["so"], st["po"], st["pts"])
            back = ctx.span_decode_ragged(pts, st["po"], st["so"], st["back"])
            got = ctx.read_ragged(pts, st["po"], st["so"], st["req"], st["out"])
        else:
            n = case["symbols"]
            pts = ctx.span_encode(st["sym"], st["pts"])
            back = ctx.span_decode(pts, n, st["back"])
            got = ctx.read(pts, n, st["req"], st["out"])
        return {"pts": pts, "back": back, "read": got}
    if kind == "lossy":
        n, bits, keep = case["symbols"], case["bits"], case["keep"]
        codes, tail = ctx.truncate(st["pts"], n, bits, keep)
        back = ctx.lossy_decode(codes, tail, n, bits, keep, st["back"])
        got = ctx.lossy_read(codes, tail, n, bits, keep, st["req"], st["out"])
        T, words, ts = ctx.lossy_geometry(n, bits, keep)     # a buffer is never empty: drop its unused element
        return {"codes": codes[:, :words], "tail": tail[:, :ts], "back": back, "read": got}
    words, nbits = ctx.ac_encode(st["sym"], case["adaptive"])
    back = ctx.ac_decode(words, nbits, case["symbols"], case["adaptive"], st["back"])
    return {"words": words, "nbits": nbits, "back": back}


# ------------------------------------------------------- what a pass needs --
def _ratio(n):
    """The packing ratio of the regular n-gon and the span length it allows."""
    r = 1.0 / (2.0 * (1.0 + sum(_vertex(n, k)[0] for k in range(1, n // 4 + 1))))
    return r, int(math.floor(44.0 / math.log2(1.0 / r)))


def _vertex(n, c):
    if (4 * c) % n == 0:
        return [(1.0, 0.0), (0.0, 1.0), (-1.0, 0.0), (0.0, -1.0)][4 * c // n]
    t = 2.0 * math.pi * c / n
    return math.cos(t), math.sin(t)


def work(case):
    kind = case["kind"]
    if kind in ("codec", "lossy", "weighted"):
        n, width = case["alphabet"], 1 if case["alphabet"] <= 256 else 2
        span = _ratio(n)[1]
        if case.get("ragged"):
            lengths = _lengths(case)
            total, spans = int(lengths.sum()), int(((lengths + span - 1) // span).sum())
        else:
            spans = case["streams"] * ((case["symbols"] + span - 1) // span)
            total = case["streams"] * case["symbols"]
        if kind == "codec":     # symbols in, points out, points in, symbols out; six binary64 operations a symbol
            return {"bytes": 2 * (total * width + 16 * spans) + case["reads"] * (32 + width), "flops": 6 * total}
        if kind == "lossy":     # points in; codes out and in; symbols out
            per = (case["symbols"] + span - 1) // span
            kept = min(per, case["keep"])
            codes = case["streams"] * (2 * (per - kept) * case["bits"] // 8)
            tail = case["streams"] * kept * 16
            return {"bytes": 16 * spans + 2 * (codes + tail) + total * width + case["reads"] * (32 + width),
                    "flops": 6 * total}
        code = int(total * math.log2(n)) // 8
        return {"bytes": 2 * total * width + 2 * code, "flops": 0}
    L, B, H, D, P = (case[k] for k in ("layers", "batch", "heads", "dim", "positions"))
    K, S = case["codewords"], case["stages_k"] + case["stages_v"]
    width, esz = 1 if K <= 256 else 2, 4 if case["dtype"] == "f32" else 2
    books = L * (1 if case["pooled"] else H) * S * K * D * 4
    vectors = L * B * H * P
    span = _ratio(K)[1]
    points = (P * _record_len(case) + span - 1) // span * 16 * L * B
    if kind == "write":
        return {"bytes": 2 * vectors * D * esz + books + vectors * S * width, "flops": 2 * vectors * S * K * D}
    if kind == "append":
        return {"bytes": 2 * vectors * D * esz + books + 2 * vectors * S * width + points,
                "flops": 2 * vectors * S * K * D}
    if kind == "restore":
        return {"bytes": points + books + 2 * vectors * D * esz, "flops": vectors * S * D}
    q = case["requests"]
    rec = (_record_len(case) + span - 1) // span * 16
    return {"bytes": q * (16 + rec + 2 * H * D * esz) + min(books, q * H * S * D * 4), "flops": q * H * S * D}


# Whole numbers of the codec are exact by its definition.  An RVQ index may
# differ where two codewords are as near as float32 accumulation can tell (and
# then the later stages of that vector): against 64-bit scores about 1e-6 of
# them do.  A rebuilt value is a float32 sum of at most four codewords rounded
# to the cache's type: another order of the sum moves about 1e-5 of the values
# to the neighbouring 16-bit number.
def tolerance(case):
    kind = case["kind"]
    if kind == "write":
        n = case["layers"] * case["batch"] * _record_len(case) * case["positions"]
        return {"differ": min(0.01, 2e-5 + 8.0 / n)}
    if kind == "append":
        n = case["layers"] * case["batch"] * _record_len(case)
        return {"differ": min(0.01, 2e-5 + 8.0 / n), "rel": 1e-2, "max": 0.99}
    if kind in ("restore", "records"):
        return {"rel": 1e-6, "max": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-4, "max": 1e-2}
    return "exact"


# -------------------------------------------------------- 64-bit results --
def _encode64(sym, n, r, span):
    """Points float64 [streams, spans, 2] of symbols [streams, n]: each span
    walks p <- V(c) + r (p - V(c)) from the origin."""
    V = torch.tensor([_vertex(n, c) for c in range(n)], dtype=torch.float64, device="cuda")
    ns, ln = sym.shape
    spans = (ln + span - 1) // span
    p = torch.zeros((ns, spans, 2), dtype=torch.float64, device="cuda")
    for j in range(span):
        m = (ln - j + span - 1) // span           # spans that have a symbol j
        if m > 0:
            v = V[sym[:, j::span][:, :m].long()]
            p[:, :m] = v + r * (p[:, :m] - v)
    return p


def _assign64(case, seed):
    """RVQ indices in token-record order, int64 [streams, positions * R]."""
    books = _codebooks(case, seed)
    L, B, H, D, P = (case[k] for k in ("layers", "batch", "heads", "dim", "positions"))
    out = torch.empty((B, L, P, _record_len(case)), dtype=torch.int64, device="cuda")
    for kv in (K_ID, V_ID):
        x = _cache(case, seed, kv, _scales(case, seed, kv), P)
        S = books[kv].shape[2]
        first = 0 if kv == K_ID else H * case["stages_k"]
        for layer in range(L):
            for h in range(H):
                res = x[layer, :, h, SINKS:SINKS + P].reshape(B * P, D).double()
                for s in range(S):
                    c = books[kv][layer, 0 if case["pooled"] else h, s].double()
                    i = torch.cat([((c * c).sum(1) - 2.0 * (part @ c.T)).argmin(1) for part in res.split(1 << 18)])
                    out[:, layer, :, first + h * S + s] = i.view(B, P)
                    res -= c[i]
    return out.view(B * L, P * _record_len(case))


def _chosen(case, rows, kv):
    """The K or V indices of token records rows [n, R], as [n, heads, stages]."""
    H = case["heads"]
    first, S = (0, case["stages_k"]) if kv == K_ID else (H * case["stages_k"], case["stages_v"])
    return rows[:, first:first + H * S].view(-1, H, S)


def _sum64(book, layer, at, pooled):
    """Sum of the chosen codewords: layer [rows], at [rows, heads, stages] -> float64 [rows, heads, dim]."""
    cb = book.double()
    h = torch.zeros(at.shape[1], dtype=torch.int64, device="cuda") if pooled else \
        torch.arange(at.shape[1], device="cuda")
    total = 0.0
    for s in range(at.shape[2]):
        total = total + cb[layer[:, None], h[None, :], s, at[:, :, s]]
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "write":
        return {"sym": _assign64(case, seed)}
    if kind == "append":
        # the new records' points move with a near tie's choice: no 64-bit value of their own
        return {"sym": _assign64(case, seed), "pts": None}
    if kind == "codec":
        r, span = _ratio(case["alphabet"])
        if not case["ragged"]:
            sym = _symbols(case, seed, (case["streams"], case["symbols"]))
            req = _requests(case, seed, case["streams"], case["symbols"], case["reads"])
            return {"pts": _encode64(sym.long(), case["alphabet"], r, span), "back": sym,
                    "read": sym[req[:, 0], req[:, 1]]}
        lengths = _lengths(case)
        sym = _symbols(case, seed, (int(lengths.sum()),))
        req = _requests(case, seed, case["streams"], lengths, case["reads"])
        at = np.concatenate([[0], np.cumsum(lengths)])
        pts = [_encode64(sym[a:b][None].long(), case["alphabet"], r, span)[0] for a, b in zip(at[:-1], at[1:])]
        start = torch.as_tensor(at, device="cuda")[req[:, 0]]
        return {"pts": torch.cat(pts), "back": sym, "read": sym[start + req[:, 1]]}
    if kind in ("lossy", "weighted"):
        return None          # whole numbers only (and points copied as they are)
    books = _codebooks(case, seed)
    L, B, H, D, P = (case[k] for k in ("layers", "batch", "heads", "dim", "positions"))
    R = _record_len(case)
    idx = _indices(case, seed, P).view(B * L, P, R)
    if kind == "records":
        req = _requests(case, seed, B * L, P, case["requests"])
        out = torch.empty((case["requests"], 2, H, D), dtype=torch.float64, device="cuda")
        for q in range(0, case["requests"], 8192):
            r = req[q:q + 8192]
            rows = idx[r[:, 0], r[:, 1]]
            for kv in (K_ID, V_ID):
                out[q:q + 8192, kv] = _sum64(books[kv], r[:, 0] % L, _chosen(case, rows, kv), case["pooled"])
        return {"kv": out}
    got = {}
    for kv, name in ((K_ID, "k"), (V_ID, "v")):
        y = torch.zeros((L, B, H, P + SINKS + RECENT, D), dtype=torch.float64, device="cuda")
        for b in range(B):
            for layer in range(L):
                at = _chosen(case, idx[b * L + layer], kv)
                y[layer, b, :, SINKS:SINKS + P] = _sum64(
                    books[kv], torch.full((P,), layer, device="cuda"), at, case["pooled"]).transpose(0, 1)
        got[name] = y
    return got
