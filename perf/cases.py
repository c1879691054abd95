"""The calls that a user of the compressed KV cache makes, as cases that can be timed and compared.

A case is a stack of identical global-attention layers and one way of driving it:

  stream   xkv_stream_step: one more frame through all layers of a stream whose caches are full
           (every pass appends, scores, evicts, packs and attends)
  host     xkv_stream_step_host: the same with the frame's tensors and outputs in pinned host memory
  calls    the four entry points of a layer one after the other (kv_append, kv_score_evict,
           kv_quant_pack, attn_packed_causal), for programs that interleave them with other work
  clip     xkv_reset, then the first frames of a new stream, so growing caches and no eviction at first
  chunks   xkv_reset, then an offline sequence that arrives several frames at a time
           (xkv_prefill_chunk on every layer)

tokens = tokens of a frame (patches + 5 special), budget = cached tokens per layer after eviction,
bits = storage of K and V (4, 8, or 16 = pruning only), keys = "regroup" (key groups re-quantised
when their members change) or "once" (quantised on arrival), tail = the frame attends to its own
K, V unquantised, layout = "head" ([H][n][64] tensors) or "token" ([n][H*64], as a projection
writes them).
"""
import torch

import paper_2601_01204_b200.xkv as xkv

HEAD_DIM = 64
OUTLIER_CHANNELS, OUTLIER_GAIN = 4, 15.0    # key channels with large magnitudes, per head, fixed per layer
DEVICE_FRAMES = 16                          # distinct frames a steady stream cycles through
HOST_FRAMES = 4                             # the same for frames in pinned host memory


def _case(entry, layers, tokens, budget, **more):
    c = dict(entry=entry, layers=layers, heads=16, tokens=tokens, budget=budget, bits=4, keys="regroup",
             tail=False, layout="head", frames=1, chunk=1)
    c.update(more)
    return c


def listed():
    return [
        # one layer, 224 x 224 frames: the smallest step of a live stream; latency and launches count
        _case("stream", 1, 261, 1024, name="tiny_step"),
        # the first eight frames of such a stream, from an empty cache
        _case("clip", 1, 261, 1024, frames=8, name="tiny_clip"),
        # one layer of a 518 x 518 stream through the separate entry points, tensors as a projection writes them
        _case("calls", 1, 1374, 8192, layout="token", name="layer_calls"),
        # the whole 24-layer stack on 518 x 518 frames: the headline workload
        _case("stream", 24, 1374, 16384, name="stack"),
        # the same with the other key mode
        _case("stream", 24, 1374, 16384, keys="once", name="stack_keys_once"),
        # the same when the frame attends to its own keys and values as they arrived
        _case("stream", 24, 1374, 16384, tail=True, name="stack_tail"),
        # the same with frames that come from and results that go to host memory
        _case("host", 24, 1374, 16384, name="stack_host"),
        # a tight memory budget
        _case("stream", 24, 1374, 4096, name="stack_small_budget"),
        # 518 x 378 frames, as in long video
        _case("stream", 24, 1004, 16384, name="long_stream"),
        # the same frames, 8-bit codes
        _case("stream", 24, 1004, 8192, bits=8, keys="once", name="stack_8bit"),
        # the largest budget, pruning without quantisation
        _case("stream", 24, 1374, 32768, bits=16, name="stack_prune_only"),
        # an offline sequence, four frames at a time
        _case("chunks", 24, 1004, 6144, frames=8, chunk=4, name="offline_chunks"),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, evenly over its logarithm."""
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def draw(rng):
    entry = rng.choice(["stream"] * 6 + ["calls"] * 2 + ["clip", "chunks", "host"])
    tokens = _spread(rng, 128, 1374)
    # at most forty frames fill a cache
    budget = _spread(rng, max(512, 2 * tokens), min(32768, 40 * tokens))
    bits, keys = rng.choice([(4, "regroup")] * 4 + [(4, "once")] * 2 + [(8, "once"), (16, "regroup"), (16, "regroup")])
    c = _case(entry, _spread(rng, 1, 24), tokens, budget, heads=rng.choice([8, 12, 16, 16]), bits=bits, keys=keys)
    if entry in ("stream", "calls", "clip"):
        c["layout"] = rng.choice(["head", "head", "token"])
    if entry == "stream" and bits != 8:
        c["tail"] = rng.random() < 0.2
    if entry == "clip":
        c["frames"] = rng.randint(3, 12)
    if entry == "chunks":
        c["chunk"] = rng.randint(2, 6)
        c["frames"] = c["chunk"] * rng.randint(1, 3)
    # no more work than the largest listed cases
    most = work(_case("stream", 24, 1374, 32768))["flops"]
    if entry in ("clip", "chunks"):
        most /= 3
    while c["layers"] > 1 and work(c)["flops"] > most:
        c["layers"] -= 1
    return c


def _lengths(case):
    """(query tokens, cached tokens they see, cached tokens before the arrival) of every attention of one pass, one layer."""
    n, L = case["tokens"], case["budget"]
    if case["entry"] in ("stream", "host", "calls"):
        return [(n, L, L)]
    got, T, first = [], 0, 0
    for _ in range(case["frames"] // case["chunk"]):
        arrival = n * case["chunk"]
        before = T
        first = first or arrival
        T = before + arrival
        if before and T > L:
            T = first + max(0, L - first - arrival) + arrival
        older = T - arrival
        got += [(n, older + (f + 1) * n, before if f == 0 else 0) for f in range(case["chunk"])]
    return got


def work(case):
    """Each frame tensor read and each output written once, the packed cache read once, what has
    to change in it written once: the arriving tokens, and all keys where they are re-quantised."""
    H, n = case["heads"], case["tokens"]
    row = {4: 32, 8: 64, 16: 128}[case["bits"]]
    v_row = row + (0 if case["bits"] == 16 else 8)
    k_row = row + (0 if case["bits"] == 16 else 8)       # (scale, zero) per channel and 64 tokens: 8 bytes a token
    rewritten = case["bits"] == 4 and case["keys"] == "regroup"
    nbytes = flops = 0
    for nq, seen, before in _lengths(case):
        frame = H * nq * HEAD_DIM * 2
        nbytes += 4 * frame + H * before * (k_row + v_row) + H * nq * (k_row + v_row)
        if rewritten:
            nbytes += H * before * k_row
        flops += 4 * H * nq * seen * HEAD_DIM
    return {"bytes": case["layers"] * nbytes, "flops": case["layers"] * flops}


def tolerance(case):
    # 16-bit operands, 32-bit accumulation, bf16 results; "max" is over the root mean square of outputs
    # whose largest values are several times that
    return {"rel": 5e-3, "max": 5e-2}


def _frames(case, count, tokens, gen):
    """`count` frames: (q, k, v), each a list over layers of [H][tokens][64] views."""
    L, H, d = case["layers"], case["heads"], HEAD_DIM
    outliers = torch.rand(L, H, d, device="cuda", generator=gen).argsort(dim=-1) < OUTLIER_CHANNELS
    gain = torch.where(outliers, OUTLIER_GAIN, 1.0).to(torch.bfloat16)
    got = []
    for _ in range(count):
        tensors = []
        for which in range(3):
            shape = (L, tokens, H, d) if case["layout"] == "token" else (L, H, tokens, d)
            x = torch.randn(shape, device="cuda", dtype=torch.bfloat16, generator=gen)
            if which == 1:
                x *= gain[:, None] if case["layout"] == "token" else gain[:, :, None]
            tensors.append(x)
        got.append(tuple(_per_layer(case, x) for x in tensors))
    return got


def _per_layer(case, x):
    return [t.transpose(0, 1) if case["layout"] == "token" else t for t in x]


def _outputs(case, tokens):
    L, H, d = case["layers"], case["heads"], HEAD_DIM
    shape = (L, tokens, H, d) if case["layout"] == "token" else (L, H, tokens, d)
    out = torch.zeros(shape, device="cuda", dtype=torch.bfloat16)
    return out, _per_layer(case, out)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n, arrival = case["tokens"], case["tokens"] * case["chunk"]
    p = xkv.Params(n_heads=case["heads"], head_dim=HEAD_DIM, budget=case["budget"], max_frame_tokens=arrival,
                   kv_bits=case["bits"], key_mode=xkv.KEYS_ONCE if case["keys"] == "once" else xkv.KEYS_REGROUP)
    s = {"case": case, "caches": [xkv.Cache(p) for _ in range(case["layers"])], "at": 0}
    if case["tail"]:
        for c in s["caches"]:
            c.xkv_set_unquantised_tail(True)
    if case["entry"] in ("clip", "chunks"):
        arrivals = case["frames"] // case["chunk"]
        s["pool"] = _frames(case, arrivals, arrival, gen)
        s["out"] = [_outputs(case, arrival) for _ in range(arrivals)]
        return s
    s["pool"] = _frames(case, DEVICE_FRAMES, n, gen)
    s["out"] = _outputs(case, n)
    for _ in range(case["budget"] // n + 2):             # until every cache is full and evicts
        q, k, v = s["pool"][s["at"] % DEVICE_FRAMES]
        s["at"] += 1
        xkv.xkv_stream_step(s["caches"], q, k, v, s["out"][1])
    if case["entry"] == "host":
        s["pool"] = [tuple([t.cpu().pin_memory() for t in ts] for ts in f) for f in s["pool"][:HOST_FRAMES]]
        out = torch.zeros(s["out"][0].shape, dtype=torch.bfloat16).pin_memory()
        s["out"] = (out, list(out))
        s["staging"] = torch.empty(xkv.xkv_stream_step_host_bytes(p, n), dtype=torch.uint8, device="cuda")
    return s


def run(s):
    case, caches = s["case"], s["caches"]
    if case["entry"] == "clip":
        for c in caches:
            c.xkv_reset()
        for (q, k, v), (_, outs) in zip(s["pool"], s["out"]):
            xkv.xkv_stream_step(caches, q, k, v, outs)
        return [out for out, _ in s["out"]]
    if case["entry"] == "chunks":
        sizes = [case["tokens"]] * case["chunk"]
        for c in caches:
            c.xkv_reset()
        for (q, k, v), (_, outs) in zip(s["pool"], s["out"]):
            for l, c in enumerate(caches):
                c.xkv_prefill_chunk(q[l], k[l], v[l], sizes, outs[l])
        return [out for out, _ in s["out"]]
    q, k, v = s["pool"][s["at"] % len(s["pool"])]
    s["at"] += 1
    out, outs = s["out"]
    if case["entry"] == "stream":
        xkv.xkv_stream_step(caches, q, k, v, outs)
    elif case["entry"] == "host":
        xkv.xkv_stream_step_host(caches, q, k, v, outs, s["staging"])
    else:
        for l, c in enumerate(caches):
            c.kv_append(k[l], v[l])
            c.kv_score_evict(q[l])
            c.kv_quant_pack()
            c.attn_packed_causal(q[l], outs[l])
    return out
