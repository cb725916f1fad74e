"""The allocation-free entry point lq_decode_attn_image_static.

Some callers of this library cannot allocate device memory (a server with a fixed start-up arena, code
under a foreign allocator policy, code called during stream capture), so they cannot use lq_cache_create.
They keep the cache as a canonical image in memory of their own and call this entry point, whose split-K
scratch is a fixed array inside the library.  The test feeds it the image exported from an ordinary cache
and checks, on two calls in a row (the second one finds the first one's leftovers in the shared scratch),
that the output agrees with lq_decode_attn on the same cache AND with the float64 CPU oracle fed the same
tokens, both within the tolerance of the parity tests.
Collected last on purpose: a run that stops at the first failure has run everything else before it."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import attn_tolerance
from paper_2503_19950_b200 import LogQuantCache, binding, build, decode_attn_image_static, synth

pytestmark = pytest.mark.gpu
D = 128


def _image_on_device(cache):
    img = cache.export(0)
    return {k: torch.from_numpy(v.view(np.int16) if v.dtype == np.uint16 else v).cuda()
            for k, v in img.items() if k not in ("kept_ids", "quant_ids")}


# (B, Hq, Hkv, W, G, n_tokens, bits): GQA 4, GQA 7 at G = 64, MHA below the first overflow, GQA 8, the paper's
# W = 42 with G = 64 (removed tokens that wait for a full key group sit among the bf16 rows), 4-bit codes, and
# B * Hq = 2048 heads with 2200 tokens, where the split count is clipped by the size of the scratch (4, not 5)
CASES = [(2, 8, 2, 64, 32, 64 * 9 + 5, 2), (1, 14, 2, 64, 64, 64 * 6 + 1, 2), (1, 4, 4, 32, 32, 40, 2),
         (1, 16, 2, 64, 32, 64 * 5 + 3, 2), (2, 8, 2, 42, 64, 42 * 11 + 7, 2), (2, 8, 2, 64, 32, 64 * 7 + 9, 4),
         (64, 32, 8, 128, 32, 2200, 2)]


@pytest.mark.parametrize("B,Hq,Hkv,W,G,n_tokens,bits", CASES)
def test_static_scratch_entry_point_matches_the_cache_entry_point_and_the_oracle_twice(B, Hq, Hkv, W, G, n_tokens,
                                                                                      bits):
    build.build()
    outl = synth.outlier_channels(77, Hkv, D, 3)
    k, v = synth.keys_values(77, B, Hkv, n_tokens, D, "cuda", outliers=outl)
    cache = LogQuantCache(1, B, Hq, Hkv, W, G, max_tokens=n_tokens + 8, bits=bits)
    cache.append(0, k, v)
    oc = oracle.OracleCache(B, Hq, Hkv, D, W, G, bits=bits)
    oc.append(synth.bf16_bits(k), synth.bf16_bits(v))
    image = _image_on_device(cache)
    for call in range(2):
        q = synth.queries(77, B, Hq, D, call, "cuda")
        want = torch.empty(B, Hq, D, device="cuda")
        cache.decode_attn(0, q, want)
        got = torch.full((B, Hq, D), float("nan"), device="cuda")
        status = decode_attn_image_static(image, Hq, G, q, got, bits=bits)
        assert status == binding.LQ_OK
        torch.cuda.synchronize()
        got = got.cpu().numpy().astype(np.float64)
        assert np.isfinite(got).all()
        ref = oc.attention(synth.bf16_bits(q), 1 / np.sqrt(D), n_threads=16)
        err = float(np.abs(got - ref).max())
        assert err <= attn_tolerance(ref), ("oracle", call, err)
        other = want.cpu().numpy().astype(np.float64)
        err = float(np.abs(got - other).max())
        assert err <= attn_tolerance(other), ("lq_decode_attn", call, err)


# (query heads per KV head, G, bits, n_fp, n_quant, elements by which every array starts off its 16-byte boundary, factor
# on the value scales): every head count, no and ragged bf16 rows, one tile of a key group of 64 per warp, one split and
# many, arrays that the wide copies cannot take, and scales near the end of the range
FORMS = [(1, 32, 2, 0, 32, 0, 1.0), (1, 64, 4, 9, 64 * 31, 0, 1.0), (2, 32, 2, 1, 32 * 40, 0, 1.0), (2, 64, 2, 384, 0, 0, 1.0),
         (3, 64, 2, 7, 64, 1, 1.0), (3, 32, 4, 63, 32 * 77, 0, 2.0 ** 118), (4, 32, 2, 385, 32 * 300, 0, 2.0 ** 119),
         (4, 32, 4, 8, 32 * 33, 3, 1.0), (5, 64, 2, 127, 64 * 21, 0, 1.0), (6, 32, 2, 15, 32 * 2, 5, 1.0),
         (7, 64, 4, 770, 64 * 130, 0, 1.0), (8, 32, 2, 16, 32 * 95, 0, 1.0), (8, 64, 2, 0, 64 * 9, 1, 1.0)]


@pytest.mark.parametrize("r,G,bits,n_fp,n_quant,off,factor", FORMS)
def test_random_images_against_the_same_attention_in_64_bits(r, G, bits, n_fp, n_quant, off, factor):
    """Sums of up to 10^4 fp32 terms of either sign: 2^-24 times a few of them against the root of their sum of squares,
    2e-6 seen; 1e-5 allowed."""
    build.build()
    B, H, gen = 3, 2, torch.Generator(device="cuda").manual_seed(r * 1000 + n_quant)

    def place(x):  # a copy of x that starts `off` elements behind a 16-byte boundary
        buf = torch.empty(x.numel() + 16, dtype=x.dtype, device="cuda")
        y = buf[off:off + x.numel()].view(x.shape)
        y.copy_(x)
        return y

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)

    codes = [torch.randint(0, 256, (B, H, n_quant, D * bits // 8), generator=gen, device="cuda", dtype=torch.uint8)
             for _ in range(2)]
    top = 2 ** bits - 1
    ks, vs = normal(B, H, n_quant // G, D).abs() / top, normal(B, H, n_quant, D // G).abs() / top * factor
    kz, vz = normal(B, H, n_quant // G, D) - top / 2 * ks, normal(B, H, n_quant, D // G) * factor - top / 2 * vs
    fp = [normal(B, H, n_fp, D), normal(B, H, n_fp, D) * factor]
    q = normal(B, H * r, D)
    arrays = dict(fp_k=fp[0], fp_v=fp[1], k_codes=codes[0], v_codes=codes[1], k_scale=ks, k_zero=kz, v_scale=vs, v_zero=vz)
    image = {n: place(x if x.dtype == torch.uint8 else x.view(torch.int16)) for n, x in arrays.items()}
    out = torch.full((B, H * r, D), float("nan"), device="cuda")
    assert decode_attn_image_static(image, H * r, G, place(q), out, bits=bits) == binding.LQ_OK
    code = [torch.stack([(c >> (bits * i)) & top for i in range(8 // bits)], dim=-1).flatten(3).double() for c in codes]
    keys = kz.double().repeat_interleave(G, 2) + code[0] * ks.double().repeat_interleave(G, 2)
    values = vz.double().repeat_interleave(G, 3) + code[1] * vs.double().repeat_interleave(G, 3)
    keys, values = torch.cat([fp[0].double(), keys], 2), torch.cat([fp[1].double(), values], 2)
    s = q.double().view(B, H, r, D) @ keys.transpose(2, 3) / np.sqrt(D)
    want = (torch.softmax(s, 3) @ values).view(B, H * r, D)
    assert float((out.double() - want).norm() / want.norm()) < 1e-5


@pytest.mark.parametrize("r,G,bits,n_fp,n_quant,off", [(4, 32, 2, 40, 32 * 3, 0), (4, 32, 2, 385, 32 * 60, 0), (7, 64, 4, 200, 64 * 20, 0),
                                                       (2, 32, 4, 100, 32 * 30, 1)])
def test_captured_calls_give_what_eager_calls_give(r, G, bits, n_fp, n_quant, off):
    """One split and several, wide and byte-wise fetches, two calls in a row in one graph (the second finds the first one's
    partials in the scratch), replayed on other inputs than those of the capture."""
    build.build()
    B, H, gen = 2, 2, torch.Generator(device="cuda").manual_seed(n_quant)

    def place(x):  # a copy of x that starts `off` elements behind a 16-byte boundary
        buf = torch.empty(x.numel() + 16, dtype=x.dtype, device="cuda")
        y = buf[off:off + x.numel()].view(x.shape)
        y.copy_(x)
        return y

    def bf16(*shape):
        return place(torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16).view(torch.int16))

    def codes():
        return place(torch.randint(0, 256, (B, H, n_quant, D * bits // 8), generator=gen, device="cuda", dtype=torch.uint8))

    image = dict(fp_k=bf16(B, H, n_fp, D), fp_v=bf16(B, H, n_fp, D), k_codes=codes(), v_codes=codes(),
                 k_scale=bf16(B, H, n_quant // G, D), k_zero=bf16(B, H, n_quant // G, D),
                 v_scale=bf16(B, H, n_quant, D // G), v_zero=bf16(B, H, n_quant, D // G))
    q = torch.randn(2, B, H * r, D, generator=gen, device="cuda", dtype=torch.bfloat16)
    out = torch.empty(2, B, H * r, D, device="cuda")

    def calls():
        for i in range(2):
            assert decode_attn_image_static(image, H * r, G, q[i], out[i], bits=bits) == binding.LQ_OK

    calls()   # (the first call on a device comes before any capture)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        calls()
    q.copy_(torch.randn(q.shape, generator=gen, device="cuda", dtype=torch.bfloat16))
    calls()
    want = out.clone()
    out.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    assert bool(want.isfinite().all()) and torch.equal(out, want)


def _empty_image(B):
    z16 = torch.zeros(1, dtype=torch.int16, device="cuda")
    return dict(fp_k=torch.zeros(B, 1, 1, 128, dtype=torch.int16, device="cuda"),
                fp_v=torch.zeros(B, 1, 1, 128, dtype=torch.int16, device="cuda"),
                k_codes=torch.zeros(B, 1, 0, 32, dtype=torch.uint8, device="cuda"),
                v_codes=torch.zeros(B, 1, 0, 32, dtype=torch.uint8, device="cuda"),
                k_scale=z16[:0].reshape(B, 1, 0, 128), k_zero=z16[:0].reshape(B, 1, 0, 128),
                v_scale=z16[:0].reshape(B, 1, 0, 4), v_zero=z16[:0].reshape(B, 1, 0, 4))


def test_sizes_beyond_the_scratch_are_rejected():
    build.build()
    image = _empty_image(1100)
    q = torch.zeros(1100, 8, 128, dtype=torch.bfloat16, device="cuda")
    out = torch.zeros(1100, 8, 128, device="cuda")
    assert decode_attn_image_static(image, 8, 32, q, out) == binding.LQ_ERR_CAPACITY  # 8800 > 8192 records
    assert b"scratch" in binding.load_library().lq_status_str(binding.LQ_ERR_CAPACITY)


def test_a_code_width_the_image_format_does_not_have_is_rejected():
    build.build()
    image = _empty_image(1)
    q = torch.zeros(1, 1, 128, dtype=torch.bfloat16, device="cuda")
    out = torch.zeros(1, 1, 128, device="cuda")
    for bits in (0, 3, 8):
        assert decode_attn_image_static(image, 1, 32, q, out, bits=bits) == binding.LQ_ERR_INVALID_ARG
