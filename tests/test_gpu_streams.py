"""Order on the device: what a call may assume of the work enqueued before it, on other streams, across stream captures and
after a call that failed."""
import numpy as np
import pytest
import torch

import oracle
from gpu_common import assert_images_equal, attn_tolerance
from paper_2503_19950_b200 import LQ_FLAG_OVERLAP_DECODE, LogQuantCache, LogQuantError, binding, build, synth

pytestmark = pytest.mark.gpu
B, HQ, HKV, W, G, D = 1, 8, 2, 32, 32, 128
BUSY = 60_000_000  # clock cycles of a kernel that keeps a stream busy: about 30 ms


@pytest.fixture(scope="module", autouse=True)
def _built():
    build.build()


def _filled(seed, n):
    """Keys and values of n tokens and the oracle's cache that holds them."""
    k, v = synth.keys_values(seed, B, HKV, n, D, "cuda")
    oc = oracle.OracleCache(B, HQ, HKV, D, W, G)
    oc.append(synth.bf16_bits(k), synth.bf16_bits(v))
    return k, v, oc


def _check_attention(oc, q, out):
    ref = oc.attention(synth.bf16_bits(q), 1 / np.sqrt(D))
    assert np.abs(out.cpu().numpy() - ref).max() <= attn_tolerance(ref)


@pytest.mark.parametrize("allocator", [None, "torch"])
def test_a_new_cache_on_another_stream_than_the_busy_default_one(allocator):
    """The zeros of a new cache come before its first tokens whatever the default stream is doing."""
    k, v, oc = _filled(1, 200)
    q, out = synth.queries(1, B, HQ, D, 0, "cuda"), torch.full((B, HQ, D), float("nan"), device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(BUSY)
    cache = LogQuantCache(1, B, HQ, HKV, W, G, max_tokens=256, allocator=allocator)
    cache.append(0, k, v, stream=side)
    cache.decode_attn(0, q, out, stream=side)
    side.synchronize()
    torch.cuda.synchronize()
    assert_images_equal(cache.export(0), oc.export())
    _check_attention(oc, q, out)
    assert cache.kernel_status() == 0
    cache.close()


def test_blocks_of_a_new_cache_that_the_stream_still_uses():
    """torch hands a freed block out again while kernels of its stream still read it: nothing may be written to it outside
    that stream's order, neither by the creation of a cache nor by its first padding."""
    k, v, oc = _filled(2, 200)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()

    def new_cache():
        cache = LogQuantCache(1, B, HQ, HKV, W, G, max_tokens=256, allocator="torch")
        cache.set_padding([3])
        return cache

    with torch.cuda.stream(side):
        first = new_cache()
        sizes = [t.numel() for t in first._blocks.values()]
        first.close()
        side.synchronize()
        old = [torch.full((n,), 7, dtype=torch.uint8, device="cuda") for n in sizes]
        read = [torch.empty_like(x) for x in old]
        at = {x.data_ptr() for x in old}
        torch.cuda._sleep(BUSY)
        for x, y in zip(old, read):
            y.copy_(x)
        del old, x
        cache = new_cache()
        assert at & set(cache._blocks), "no block was handed out again: the test shows nothing"
        cache.append(0, k, v)
    torch.cuda.synchronize()
    assert all(bool((y == 7).all()) for y in read)
    assert_images_equal(cache.export(0), oc.export())
    cache.close()


@pytest.mark.parametrize("allocator", [None, "torch"])
def test_a_new_cache_whose_first_calls_are_captured(allocator):
    """The zeros of a new cache are no part of a graph: they are there before its first replay and do not come again."""
    k, v, oc = _filled(3, 2)
    q, out = synth.queries(3, B, HQ, D, 0, "cuda"), torch.full((B, HQ, D), float("nan"), device="cuda")
    rows = [tuple(x[:, :, t:t + 1].contiguous() for x in (k, v)) for t in range(2)]
    torch.cuda.synchronize()
    cache = LogQuantCache(1, B, HQ, HKV, W, G, max_tokens=256, allocator=allocator)
    graphs = [torch.cuda.CUDAGraph() for _ in rows]
    for g, row in zip(graphs, rows):
        with torch.cuda.graph(g):
            cache.append(0, *row)
            cache.decode_attn(0, q, out)
    for g in (graphs[0], graphs[1], graphs[1], graphs[0], graphs[1]):
        g.replay()
    torch.cuda.synchronize()
    assert_images_equal(cache.export(0), oc.export())
    _check_attention(oc, q, out)
    assert cache.kernel_status() == 0 and cache.check_guards() == 0
    cache.close()


@pytest.mark.parametrize("window,group", [(32, 32), (42, 64)])
def test_prompts_ingested_under_capture(window, group):
    """A graph whose replay ingests a prompt and two further chunks, into one layer between eager calls that ingest the same
    and other chunks into its neighbours (whose index lists it must neither use nor overwrite)."""
    chunks = [9 * window + 5, 2 * window + 7, 70]
    n = sum(chunks)
    cache = LogQuantCache(4, B, HQ, HKV, window, group, max_tokens=n + 64)
    oracles, pieces = [], []
    for layer in range(4):
        k, v = synth.keys_values(20 + layer, B, HKV, n, D, "cuda")
        sizes = [13] * (layer == 3) + chunks   # the last layer is in another state than the others
        pieces.append([tuple(x[:, :, e - c:e].contiguous() for x in (k, v))
                       for e, c in zip(np.cumsum(sizes), sizes) if e <= n])
        oracles.append(oracle.OracleCache(B, HQ, HKV, D, window, group))
        for piece in pieces[-1]:
            oracles[-1].append(*(synth.bf16_bits(x) for x in piece))
    q, out = synth.queries(21, B, HQ, D, 0, "cuda"), torch.empty(B, HQ, D, device="cuda")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()

    def ingest(layer):
        for piece in pieces[layer]:
            cache.append(layer, *piece)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        ingest(0)
        with torch.cuda.graph(graph, stream=stream):
            ingest(1)
            cache.decode_attn(1, q, out)
        ingest(3)
        graph.replay()
        ingest(2)
    torch.cuda.synchronize()
    for layer in range(4):
        assert_images_equal(cache.export(layer), oracles[layer].export())
    _check_attention(oracles[1], q, out)
    assert cache.kernel_status() == 0
    cache.close()


def test_padding_masks_uploaded_under_capture():
    """Two layers in different states whose masks are made in one capture: every replay finds its own layer's masks."""
    lengths, pad = (150, 217), 40
    cache = LogQuantCache(2, 2, HQ, HKV, W, G, max_tokens=256)
    oracles = []
    for layer, n in enumerate(lengths):
        k, v = synth.keys_values(50 + layer, 2, HKV, n, D, "cuda")
        cache.append(layer, k, v)
        oracles.append(oracle.OracleCache(2, HQ, HKV, D, W, G))
        oracles[-1].append(synth.bf16_bits(k), synth.bf16_bits(v))
    q, out = synth.queries(51, 2, HQ, D, 0, "cuda"), torch.full((2, 2, HQ, D), float("nan"), device="cuda")
    cache.set_padding([0, pad])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for layer in range(2):
            cache.decode_attn(layer, q, out[layer])
    for _ in range(2):
        out.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        for layer in range(2):
            ref = oracles[layer].attention_subset(synth.bf16_bits(q), 1 / np.sqrt(D), pad=[0, pad])
            assert np.abs(out[layer].cpu().numpy() - ref).max() <= attn_tolerance(ref)
    assert cache.kernel_status() == 0
    cache.close()


def _two_layers(flags=0):
    """A cache of two small layers with a few steps behind them, and the calls of further steps."""
    cache = LogQuantCache(2, B, HQ, HKV, W, G, max_tokens=256, flags=flags)
    q, out = synth.queries(4, B, HQ, D, 0, "cuda"), torch.empty(B, HQ, D, device="cuda")
    k, v, _ = _filled(4, 150)
    row = tuple(x[:, :, :1].contiguous() for x in (k, v))
    for layer in range(2):
        cache.append(layer, k, v)

    def fused(layer):
        cache.append_decode_attn(layer, *row, q, out)

    def plain(layer):
        cache.decode_attn(layer, q, out)

    torch.cuda.synchronize()
    return cache, fused, plain


def test_which_launches_fetch_their_stages_early():
    """Default flags, small launches: one that follows a decode launch of the same cache and stream, unless that one wrote
    a row of the same layer."""
    cache, fused, plain = _two_layers()
    other = torch.cuda.Stream()
    count = [cache.debug_launches_prefetched()]

    def early(call, layer):
        call(layer)
        count.append(cache.debug_launches_prefetched())
        return count[-1] - count[-2]

    assert early(plain, 0) == 0      # behind the appends
    assert early(plain, 0) == 1
    assert early(plain, 1) == 1
    assert early(fused, 0) == 1
    assert early(plain, 0) == 0      # behind the launch that wrote its row
    assert early(plain, 1) == 1
    assert early(fused, 0) == 1
    assert early(plain, 1) == 1
    assert early(plain, 0) == 1      # that launch has waited for the one that wrote the row
    other.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(other):
        assert early(plain, 1) == 0  # another stream
        assert early(plain, 0) == 1
    torch.cuda.current_stream().wait_stream(other)
    assert early(plain, 0) == 0
    k, v, _ = _filled(5, 40)
    cache.append(0, k, v)            # an overflow step on the way
    assert early(plain, 1) == 0
    cache.profile_enable()
    assert early(plain, 0) == 0      # timed launches start alone
    cache.profile_enable(False)
    assert early(plain, 0) == 0
    assert early(plain, 1) == 1
    torch.cuda.synchronize()
    assert cache.kernel_status() == 0
    cache.close()


def test_a_launch_that_failed_was_not_there():
    """A decode call that returns an error has launched nothing: the call after it must not take it for the launch that
    stands between it and the one that wrote its row."""
    from cuda.bindings import runtime
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        cache, fused, plain = _two_layers()
        plain(1)
        fused(0)
        handle = runtime.cudaStream_t(stream.cuda_stream)
        # a capture that a forbidden synchronisation has made invalid: every launch on the stream fails until it is ended
        assert runtime.cudaStreamBeginCapture(handle, runtime.cudaStreamCaptureMode.cudaStreamCaptureModeThreadLocal)[0] == 0
        assert runtime.cudaStreamSynchronize(handle)[0] != 0
        with pytest.raises(LogQuantError) as err:
            plain(1)
        assert err.value.status == binding.LQ_ERR_CUDA
        assert runtime.cudaStreamEndCapture(handle)[0] != 0
        runtime.cudaGetLastError()
        before = cache.debug_launches_prefetched()
        plain(0)
        assert cache.debug_launches_prefetched() == before
        k, v, _ = _filled(5, 1)
        cache.append(1, k, v)        # the error of the earlier call is not reported again
        plain(1)
    torch.cuda.synchronize()
    assert cache.kernel_status() == 0
    cache.close()


def test_captured_launches_are_no_predecessors_of_eager_ones():
    """A captured launch has not run: neither the early fetch nor the overlapped form may be derived from it."""
    stream = torch.cuda.Stream()
    for flags, count in ((0, lambda c: c.debug_launches_prefetched()), (LQ_FLAG_OVERLAP_DECODE, lambda c: c.info(0).n_launches_overlapped)):
        with torch.cuda.stream(stream):
            cache, fused, plain = _two_layers(flags)
            plain(1)
            fused(0)
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                before = count(cache)
                plain(1)             # follows nothing that is part of the graph
                assert count(cache) == before
                plain(1)
            before = count(cache)
            plain(0)
            assert count(cache) == before
            plain(1)
            assert count(cache) == before + 1
            graph.replay()
        torch.cuda.synchronize()
        assert cache.kernel_status() == 0
        del graph
        cache.close()


@pytest.mark.parametrize("r", [4, 7])
@pytest.mark.parametrize("bits,group", [(2, 32), (4, 64)])
def test_small_launches_at_ordinary_lengths_are_reproducible(r, bits, group):
    """One sequence of 1100 to 2200 tokens: the partial results are summed in order, not as they arrive."""
    for n in (1100, 1250, 1500, 1800, 2200):
        cache = LogQuantCache(1, 1, 8 * r, 8, 128, group, max_tokens=n + 8, bits=bits)
        k, v = synth.keys_values(n, 1, 8, n, D, "cuda")
        cache.append(0, k, v)
        q = synth.queries(n, 1, 8 * r, D, 0, "cuda")
        outs = torch.empty(40, 1, 8 * r, D, device="cuda")
        for out in outs:
            cache.decode_attn(0, q, out)
        assert bool((outs == outs[0]).all()), n
        cache.close()


def test_the_finer_split_of_small_launches_is_for_small_launches():
    """Launches that may overlap, and timed ones, do not let the next one start early: they keep whole stages per warp."""
    n, group = 1024, 32
    k, v = synth.keys_values(9, 1, 2, n, D, "cuda")
    splits = []
    for flags in (0, LQ_FLAG_OVERLAP_DECODE):
        cache = LogQuantCache(1, 1, 8, 2, 128, group, max_tokens=n + 8, flags=flags)
        cache.append(0, k, v)
        info = cache.info(0)
        splits.append(info.n_splits)
        if not flags:
            cache.profile_enable()
            splits.append(cache.info(0).n_splits)
        cache.close()
    tiles_fp, tiles_quant = -(-info.n_fp // 16), info.n_quant // group
    assert splits == [-(-(tiles_fp + tiles_quant) // 4)] + 2 * [-(-(tiles_fp + tiles_quant // 2) // 4)]


@pytest.mark.parametrize("bits,group,n,heads", [(2, 32, 1200, (8, 2)), (2, 32, 6000, (4, 1)), (2, 64, 5000, (7, 1)), (4, 32, 3000, (8, 2)),
                                                (4, 64, 4000, (4, 4))])
@pytest.mark.parametrize("host", [False, True])
def test_small_launches_that_fetch_early_in_every_form(bits, group, n, heads, host):
    """Steps of two layers in turn, device-resident or with the rows, queries and results in pinned host memory, all of them
    behind a launch of the other layer: ordered merges and (more than 12 CTAs per pair) sums on arrival, both group sizes
    and widths, up to four and more heads per KV head."""
    hq, hkv = heads
    steps = 5
    cache = LogQuantCache(2, B, hq, hkv, 64, group, max_tokens=n + steps + 8, bits=bits)
    oracles, rows = [], []
    for layer in range(2):
        k, v = synth.keys_values(30 + layer, B, hkv, n + steps, D, "cuda")
        cache.append(layer, k[:, :, :n].contiguous(), v[:, :, :n].contiguous())
        oracles.append(oracle.OracleCache(B, hq, hkv, D, 64, group, bits=bits))
        oracles[-1].append(synth.bf16_bits(k[:, :, :n]), synth.bf16_bits(v[:, :, :n]))
        rows.append([tuple(x[:, :, n + s:n + s + 1].contiguous() for x in (k, v)) for s in range(steps)])
    assert (cache.info(0).n_splits > 12) == (n >= 3000)
    qs = [[synth.queries(31 + layer, B, hq, D, s, "cuda") for layer in range(2)] for s in range(steps)]
    outs = torch.full((steps, 2, B, hq, D), float("nan"), device="cuda")
    if host:
        pin = lambda x: torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)
        rows = [[tuple(pin(x) for x in row) for row in layer] for layer in rows]
        qs, outs = [[pin(q) for q in step] for step in qs], pin(outs)
    torch.cuda.synchronize()
    for s in range(steps):
        for layer in range(2):
            if host:
                cache.decode_step_host(layer, *rows[layer][s], qs[s][layer], outs[s, layer], sync=False)
            else:
                cache.append_decode_attn(layer, *rows[layer][s], qs[s][layer], outs[s, layer])
    torch.cuda.synchronize()
    assert cache.debug_launches_prefetched() == 2 * steps - 1   # no overflow falls into these steps
    for s in range(steps):
        for layer in range(2):
            oracles[layer].append(*(synth.bf16_bits(x) for x in rows[layer][s]))
            _check_attention(oracles[layer], qs[s][layer], outs[s, layer])
    for layer in range(2):
        assert_images_equal(cache.export(layer), oracles[layer].export())
    assert cache.kernel_status() == 0
    cache.close()
