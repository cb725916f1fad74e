"""The work that is timed: what programs that decode with a LogQuant cache have the library do.

Kinds of work (every case says which one it is):
  decode    one decode step's attention over all layers of a filled cache: decode_attn per layer
  generate  a whole batch of requests on a new cache: the prompt of every layer (in one piece or in chunks), then
            `steps` decode steps of append_decode_attn per layer, overflow steps included
  host      the same with the decode steps' keys, values, queries and results in pinned host memory
            (decode_step_host, one synchronisation per step)
  prefill   a new cache, the prompt of every layer, the first decode step's attention
  image     decode_attn_image_static over canonical images that the caller keeps in its own device memory

Keys are N(0,1) with three channels per KV head scaled by ten (outlier channels) and, with `spikes`, a common
direction added at log-spaced distances behind the last position; values and queries are N(0,1).
"""
import math

import torch

from paper_2503_19950_b200 import LogQuantCache
from paper_2503_19950_b200.binding import LQ_FLAG_OVERLAP_DECODE, decode_attn_image_static

D = 128
N_OUTLIERS = 3


def _case(kind, L, B, Hq, Hkv, ctx, W=128, G=32, bits=2, overlap=False, bf16_out=False, padded=False, spikes=False,
          steps=0, chunk=0, name=None):
    c = dict(kind=kind, L=L, B=B, Hq=Hq, Hkv=Hkv, ctx=ctx, W=W, G=G, bits=bits, overlap=overlap, bf16_out=bf16_out,
             padded=padded, spikes=spikes, steps=steps, chunk=chunk)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one small layer on its own: nothing but launch latency and host work
        _case("decode", 1, 1, 8, 2, 1024, name="tiny-1k"),
        # one user's conversation on a Llama-3-8B-shaped stack, default flags: the latency of every launch counts
        _case("decode", 32, 1, 32, 8, 8192, name="b1-8k"),
        # the same stack serving a batch, default flags: every launch waits for the one before it
        _case("decode", 16, 8, 32, 8, 8192, name="b8-8k"),
        # a large batch of middling contexts; consecutive layers may overlap, results in bf16
        _case("decode", 8, 64, 32, 8, 4096, overlap=True, bf16_out=True, name="b64-4k"),
        # long documents with seven query heads per KV head and group 64
        _case("decode", 8, 4, 28, 4, 32768, W=256, G=64, overlap=True, spikes=True, name="gqa7-32k"),
        # one very long context without grouped queries
        _case("decode", 4, 1, 32, 32, 131072, W=256, overlap=True, name="mha-128k"),
        # the more precise setting: 4-bit codes
        _case("decode", 16, 8, 32, 8, 8192, bits=4, overlap=True, name="b8-8k-int4"),
        # prompts of different lengths, left-padded to an odd common length
        _case("decode", 16, 8, 32, 8, 7925, padded=True, name="b8-ragged"),
        # prompt ingestion in one piece
        _case("prefill", 8, 8, 32, 8, 8192, name="prefill-8k"),
        # a batch of requests from prompt to answer, prompt in odd chunks, in the paper's own setting
        # (reserved length 128: W = 42, group 64)
        _case("generate", 16, 8, 32, 8, 4000, W=42, G=64, overlap=True, steps=64, chunk=1777, name="generate-b8"),
        # the whole stack with the decode steps' data in host memory
        _case("host", 32, 8, 32, 8, 8192, overlap=True, steps=32, name="host-b8-8k"),
        # a server with a fixed memory arena that keeps canonical images itself
        _case("image", 4, 4, 32, 8, 4096, name="image-4k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["decode", "generate", "host", "prefill", "image"], [55, 17, 8, 15, 5])[0]
    Hq, Hkv = rng.choice([(8, 2), (32, 8), (32, 8), (28, 4), (64, 8), (16, 8), (24, 8), (32, 32), (40, 8)])
    W, G = rng.choice([(128, 32), (128, 32), (256, 32), (256, 64), (128, 64), (42, 64), (85, 64)])
    B = _log_int(rng, 1, 64)
    # tokens of all (sequence, KV head) pairs of one layer: at most those of the largest listed cases
    most = {"decode": 32 * 131072, "image": 32 * 4096}.get(kind, 64 * 8192) // (B * Hkv)
    ctx = min(_log_int(rng, 300, 131072), max(most, 300))
    # layers: at most the bytes of a listed case of the kind
    per_layer = B * Hkv * ctx
    budget = {"decode": 8 * 64 * 8 * 4096, "image": 4 * 32 * 4096, "prefill": 8 * 64 * 8192}.get(kind, 16 * 64 * 8192)
    L = max(1, min(rng.randint(1, 32), budget // per_layer))
    return _case(kind, L, B, Hq, Hkv, ctx, W, G, bits=rng.choice([2, 2, 2, 4]), overlap=rng.random() < 0.5,
                 bf16_out=kind not in ("host", "image") and rng.random() < 0.3,
                 padded=kind == "decode" and B > 1 and rng.random() < 0.25, spikes=rng.random() < 0.2,
                 steps=rng.randint(8, 48) if kind in ("generate", "host") else 0,
                 chunk=rng.choice([0, 0, rng.randint(300, 4096)]) if kind in ("generate", "prefill") else 0)


def _keys_values(c, n, gen):
    shape = (c["B"], c["Hkv"], n, D)
    k = torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    v = torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    gain = torch.ones(c["Hkv"], D, device="cuda", dtype=torch.bfloat16)
    gain.scatter_(1, torch.rand(c["Hkv"], D, generator=gen, device="cuda").topk(N_OUTLIERS, dim=1).indices, 10.0)
    k *= gain[None, :, None, :]
    if c["spikes"]:
        u = torch.nn.functional.normalize(torch.randn(c["Hkv"], D, generator=gen, device="cuda"), dim=1)
        at = torch.tensor([n - 1 - (1 << i) for i in range(n.bit_length()) if n - 1 - (1 << i) >= 0], device="cuda",
                          dtype=torch.long)
        k[:, :, at] += (16.0 * u).to(torch.bfloat16)[None, :, None, :]
    return k, v


def _queries(c, shape, gen):
    return torch.randn(*shape, c["B"], c["Hq"], D, generator=gen, device="cuda", dtype=torch.bfloat16)


def _new_cache(c):
    return LogQuantCache(c["L"], c["B"], c["Hq"], c["Hkv"], c["W"], c["G"], max_tokens=c["ctx"] + c["steps"] + 8,
                         bits=c["bits"], flags=LQ_FLAG_OVERLAP_DECODE if c["overlap"] else 0, allocator="torch")


def _chunks(c):
    step = c["chunk"] or c["ctx"]
    return [(t, min(step, c["ctx"] - t)) for t in range(0, c["ctx"], step)]


def prepare(case, seed):
    c, L = case, case["L"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out_type = torch.bfloat16 if c["bf16_out"] else torch.float32
    if c["kind"] in ("decode", "image"):
        cache = _new_cache(c)
        for layer in range(L):
            cache.append(layer, *_keys_values(c, c["ctx"], gen))
        if c["padded"]:
            # the first sequence fills the batch's length, the others are down to an eighth of it
            cache.set_padding([c["ctx"] * 7 * b // (8 * c["B"]) for b in range(c["B"])])
        q = _queries(c, (L,), gen)
        out = torch.empty(L, c["B"], c["Hq"], D, device="cuda", dtype=out_type)
        if c["kind"] == "decode":
            return dict(c=c, cache=cache, q=q, out=out)
        images = []
        for layer in range(L):
            img = cache.export(layer)
            images.append({n: torch.from_numpy(a.view("int16") if a.dtype == "uint16" else a).cuda()
                           for n, a in img.items() if n not in ("kept_ids", "quant_ids")})
        cache.close()
        return dict(c=c, images=images, q=q, out=out)
    # one tensor per chunk and layer, as a model's prefill leaves them
    prompt = []
    for layer in range(L):
        k, v = _keys_values(c, c["ctx"], gen)
        prompt.append([(k[:, :, t:t + n].contiguous(), v[:, :, t:t + n].contiguous()) for t, n in _chunks(c)])
    state = dict(c=c, prompt=prompt)
    steps = max(c["steps"], 1)
    state["q"] = _queries(c, (steps, L), gen)
    state["out"] = torch.empty(steps, L, c["B"], c["Hq"], D, device="cuda", dtype=out_type)
    if c["steps"]:
        new = [_keys_values(c, c["steps"] * L, gen)[i].view(c["B"], c["Hkv"], c["steps"], L, 1, D)
               .permute(2, 3, 0, 1, 4, 5).contiguous() for i in (0, 1)]
        state["k"], state["v"] = new
    if c["kind"] == "host":
        for n in ("q", "k", "v", "out"):
            state[n] = torch.empty(state[n].shape, dtype=state[n].dtype, pin_memory=True).copy_(state[n])
    return state


def run(state):
    c = state["c"]
    q, out = state["q"], state["out"]
    if c["kind"] == "decode":
        for layer in range(c["L"]):
            state["cache"].decode_attn(layer, q[layer], out[layer])
        return out
    if c["kind"] == "image":
        for layer in range(c["L"]):
            status = decode_attn_image_static(state["images"][layer], c["Hq"], c["G"], q[layer], out[layer], bits=c["bits"])
            if status:
                raise RuntimeError("decode_attn_image_static: status %d" % status)
        return out
    cache = _new_cache(c)
    for layer in range(c["L"]):
        for k, v in state["prompt"][layer]:
            cache.append(layer, k, v)
    if c["kind"] == "prefill":
        for layer in range(c["L"]):
            cache.decode_attn(layer, q[0, layer], out[0, layer])
    else:
        k, v = state["k"], state["v"]
        for step in range(c["steps"]):
            for layer in range(c["L"]):
                if c["kind"] == "generate":
                    cache.append_decode_attn(layer, k[step, layer], v[step, layer], q[step, layer], out[step, layer])
                else:
                    cache.decode_step_host(layer, k[step, layer], v[step, layer], q[step, layer], out[step, layer],
                                           sync=layer == c["L"] - 1)
    cache.close()
    return out


def _lengths(c, n):
    """(tokens at full precision, quantised tokens) of a sequence after n tokens."""
    W, G = c["W"], c["G"]
    gone = 0 if n <= 3 * W else W * ((n - 3 * W + W - 1) // W)
    return n - gone // G * G, gone // G * G


def _stored_bytes(c, n, first=0):
    """Bytes of one sequence's stores in one KV head, its first `first` tokens left out."""
    fp, quant = _lengths(c, n)
    per_token = 2 * (D * c["bits"] // 8) + 2 * (2 * D * 2 // c["G"])
    return (quant * per_token + fp * 4 * D) * (n - first) / n


def _step(c, n):
    """Bytes and operations of one decode step of one layer after n tokens."""
    pads = [c["ctx"] * 7 * b // (8 * c["B"]) if c["padded"] else 0 for b in range(c["B"])]
    stores = sum(c["Hkv"] * _stored_bytes(c, n, p) for p in pads)
    tokens = sum(n - p for p in pads)
    return stores + c["B"] * c["Hq"] * D * (2 + (2 if c["bf16_out"] else 4)), 4 * c["Hq"] * D * tokens


def work(case):
    c = case
    nbytes, flops = 0, 0
    if c["kind"] in ("generate", "host", "prefill"):
        # the prompt read once and the stores written once
        nbytes += c["B"] * c["Hkv"] * (c["ctx"] * 4 * D + _stored_bytes(c, c["ctx"]))
    for n in range(c["ctx"] + 1, c["ctx"] + c["steps"] + 1) if c["steps"] else [c["ctx"]]:
        b, f = _step(c, n)
        nbytes, flops = nbytes + b + (c["B"] * c["Hkv"] * 8 * D if c["steps"] else 0), flops + f
    return {"bytes": nbytes * c["L"], "flops": flops * c["L"]}


def tolerance(case):
    """Four times the largest distance from exact() that was seen over the sizes of this file (2-norm of the difference
    over 2-norm of the result)."""
    c = case
    if c["kind"] == "image":
        rel = 1e-5  # 32-bit sums throughout: 1.5e-6 seen
    elif c["Hq"] // c["Hkv"] <= 4:
        # probabilities in two bf16 parts, 32-bit sums: 4e-5 seen up to 80000 tokens; with longer sums, whose result is
        # the smaller the longer they are, 2e-4 at 98000 and 1.5e-3 at 131072
        rel = 1.6e-4 + 4e-9 * c["ctx"] + 3.2e-13 * c["ctx"] ** 2
    else:
        # probability times value scale in one fp16 operand: 9e-4 seen, with 4-bit codes (smaller scales) 5e-3
        rel = 4e-3 if c["bits"] == 2 else 2e-2
    return {"rel": rel + (6.6e-3 if c["bf16_out"] else 0.0)}  # results rounded to bf16: 1.7e-3 seen


def _filter(c, n_last):
    """Algorithm 1 on token ids: the tokens that leave full precision, in the order in which they leave."""
    W, kept, gone = c["W"], [], []
    for t in range(n_last):
        if len(kept) == 3 * W:
            gone += kept[1:2 * W:2]
            kept = kept[0:2 * W:2] + kept[2 * W:]
        kept.append(t)
    return gone[:len(gone) // c["G"] * c["G"]]


def _quantised(x, top, dim):
    """x (float32 holding bf16 values) after asymmetric quantisation in groups along dim: codes 0..top, the scale rounded
    to bf16; the result in 64 bits."""
    zero = x.amin(dim, keepdim=True)
    scale = ((x.amax(dim, keepdim=True) - zero) / torch.full_like(zero, top)).to(torch.bfloat16).float()
    code = ((x - zero) / torch.where(scale > 0, scale, 1.0)).round().clamp(0, top) * (scale > 0)
    return zero.double() + code.double() * scale.double()


def exact(case, seed):
    """The attention of every step over the stores that Algorithm 1 and the quantiser leave, in 64 bits."""
    c, L, B, H, G = case, case["L"], case["B"], case["Hkv"], case["G"]
    r, steps, top = c["Hq"] // H, max(c["steps"], 1), 3.0 if c["bits"] == 2 else 15.0
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for _ in range(L):  # the queries come behind every layer's prompt
        _keys_values(c, c["ctx"], gen)
    q = _queries(c, (L,) if c["kind"] in ("decode", "image") else (steps, L), gen).view(steps, L, B, H, r, D)
    new = [_keys_values(c, c["steps"] * L, gen)[i].view(B, H, c["steps"], L, D) for i in (0, 1)] if c["steps"] else []
    gen.manual_seed(seed)
    order = torch.tensor(_filter(c, c["ctx"] + c["steps"]), device="cuda", dtype=torch.long)
    out = torch.empty(steps, L, B, H, r, D, device="cuda", dtype=torch.float64)
    for layer in range(L):
        rows = _keys_values(c, c["ctx"], gen)
        if new:
            rows = [torch.cat([x, y[:, :, :, layer]], dim=2) for x, y in zip(rows, new)]
        k, v = (x.double() for x in rows)
        grouped = [x[:, :, order].float().view(B, H, -1, G, D) for x in rows]
        low_k = _quantised(grouped[0], top, 3).view(B, H, -1, D)
        low_v = _quantised(grouped[1].view(B, H, -1, D // G, G), top, 4).view(B, H, -1, D)
        done = 0
        for step in range(steps):
            n = c["ctx"] + (step + 1 if c["steps"] else 0)
            low = _lengths(c, n)[1]
            if low > done:
                k[:, :, order[done:low]], v[:, :, order[done:low]], done = low_k[:, :, done:low], low_v[:, :, done:low], low
            s = q[step, layer].double() @ k[:, :, :n].transpose(2, 3) / math.sqrt(D)
            if c["padded"]:
                for b in range(B):
                    s[b, :, :, :c["ctx"] * 7 * b // (8 * B)] = -math.inf
            out[step, layer] = torch.softmax(s, dim=3) @ v[:, :, :n]
    out = out.view(steps, L, B, c["Hq"], D)
    if c["kind"] == "host":
        return out.cpu()
    return out[0] if c["kind"] in ("decode", "image") else out
