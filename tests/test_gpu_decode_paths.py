"""Decode kernels at the sizes where their tiling, their combine and their fused append can go wrong, against the
oracle's weighted attention over the same rows.  Tolerances: 1e-5 for fp32; for bf16 the error of rounding the oracle's
own result (up to 2^-8, typically 1.7e-3) plus 5e-4, which covers the outputs that round the other way because the fp32
result differs in its last bits (a share of s values off by one unit adds 2^-7.5 sqrt(s): s < 1 %)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_07861_b200 import synth
from parity_util import rel_l2, to_device

pytestmark = pytest.mark.gpu


def _check(out, ref, dtype, what):
    tol = 1e-5 if dtype == "fp32" else rel_l2(synth.round_to(ref, "bf16"), ref) + 5e-4
    assert rel_l2(out, ref) <= tol, (what, rel_l2(out, ref), tol)


def _check_heads(out, K, V, w, q, g, dtype, what):
    for h in range(K.shape[1]):
        hs = slice(h * g, (h + 1) * g)
        _check(out[0, hs], oracle.weighted_attention(K[0, h], V[0, h], w, q[0, hs]), dtype, (what, h))


@pytest.mark.parametrize("g,splits,n_heavy,n_tail", [(1, 1, 65, 0), (2, 0, 63, 1), (4, 3, 640, 64), (5, 7, 1200, 129), (8, 64, 3000, 1)])
def test_tensor_core_decode_of_64_dim_heads(cuda_lib, g, splits, n_heavy, n_tail):
    """d = 64 on the tensor-core kernel: packed and unpacked probabilities, one split to more splits than tiles, tiles
    with one row, and the fused append of two steps (the second attends the row that the first appended)."""
    B, H, d, T = 1, 3, 64, 2
    ctx = cuda_lib.Context(n_seqs=B, n_layers=1, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype="bf16", block=64, levels=T,
                           max_tokens=(n_heavy << T) + n_tail + 8, decode_splits=splits)
    n = n_heavy + n_tail
    K, V = synth.layer_kv("llama", 33, 0, B, H, n + 2, d, "bf16")
    ctx.cache_load_level(0, T, to_device(K[:, :, :n_heavy], "bf16"), to_device(V[:, :, :n_heavy], "bf16"))
    if n_tail:
        ctx.stream_append_layer(0, to_device(K[:, :, n_heavy:n], "bf16"), to_device(V[:, :, n_heavy:n], "bf16"))
    w = np.concatenate([np.full(n_heavy, 4.0), np.ones(n_tail + 2)])
    for step in range(3):
        q = synth.queries(33, 0, step, B, H * g, d, "bf16")
        qt = to_device(q, "bf16")
        if step == 0:
            out, m = ctx.decode_attn(0, qt), n
        else:
            m = n + step
            out = ctx.stream_step(0, qt, to_device(K[:, :, m - 1], "bf16"), to_device(V[:, :, m - 1], "bf16"), qt.clone())
        assert ctx.debug_scratch_used() == 0
        _check_heads(out.float().cpu().numpy(), K[:, :, :m], V[:, :, :m], w[:m], q, g, "bf16", (g, splits, step))
    st = ctx.stats()
    assert st["device_status"] == 0 and st["decode_kernel"] == 2
    Kg, Vg, wg, idx = ctx.cache_view(0, 0, H - 1)
    assert np.array_equal(Kg.float().cpu().numpy(), K[0, H - 1]) and np.array_equal(Vg.float().cpu().numpy(), V[0, H - 1])
    assert np.array_equal(wg.cpu().numpy(), w.astype(np.float32))
    ctx.close()


@pytest.mark.parametrize("S,g,d,T,n_heavy,n_tail", [(1, 1, 64, 0, 0, 5), (3, 4, 128, 2, 64, 1), (5, 8, 64, 3, 1000, 63), (300, 2, 128, 1, 65, 0),
                                                    (40, 5, 128, 1, 0, 130)])
def test_static_decode_on_tensor_cores(cuda_lib, S, g, d, T, n_heavy, n_tail):
    """The allocation-free entry on the tensor-core kernel: no heavy rows, a single split (more streams
    than a wave of CTAs) and several; more calls than there are blocks of rows; and streams next to one that holds NaN
    (a tile never reads a neighbour's rows)."""
    n = n_heavy + n_tail
    K, V = synth.layer_kv("llama", 35, 0, 1, min(S, 6), n, d, "bf16")
    K, V = (np.concatenate([x[0]] * -(-S // 6))[:S, :n] for x in (K, V))
    poisoned = np.full((1, n, d), np.nan, np.float32)
    Kd, Vd = (to_device(np.concatenate([x, poisoned]), "bf16") for x in (K, V))
    w = np.concatenate([np.full(n_heavy, float(1 << T)), np.ones(n_tail)])
    for call in range(6):
        q = synth.queries(35, 0, call, S + 1, g, d, "bf16")
        out = cuda_lib.decode_attn_static(Kd, Vd, n_heavy, T, to_device(q, "bf16")).float().cpu().numpy()
        for s in range(0, S, max(1, S // 5)):
            _check(out[s], oracle.weighted_attention(K[s], V[s], w, q[s]), "bf16", (call, s))
    assert cuda_lib.decode_attn_static_status() == 0


@pytest.mark.parametrize("dtype,d,g,splits,n_heavy,n_tail",
                         [("fp32", 128, 1, 1, 33, 0), ("fp32", 128, 3, 0, 1000, 31), ("fp32", 128, 8, 5, 900, 33), ("fp32", 64, 2, 64, 70, 1),
                          ("fp32", 64, 5, 0, 2100, 64), ("bf16", 128, 4, 3, 600, 65), ("bf16", 64, 7, 0, 1300, 1)])
def test_cuda_core_decode(cuda_lib, dtype, d, g, splits, n_heavy, n_tail):
    """The CUDA-core kernel: every rounded group size, batches that end inside a tile, one split to more splits than
    tiles, the fused append, and the same rows through the allocation-free entry (fp32)."""
    B, H, T = 1, 3, 2
    ctx = cuda_lib.Context(n_seqs=B, n_layers=1, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=64, levels=T,
                           max_tokens=(n_heavy << T) + n_tail + 8, decode_splits=splits, gram_path=1)
    n = n_heavy + n_tail
    K, V = synth.layer_kv("llama", 37, 0, B, H, n + 2, d, dtype)
    ctx.cache_load_level(0, T, to_device(K[:, :, :n_heavy], dtype), to_device(V[:, :, :n_heavy], dtype))
    if n_tail:
        ctx.stream_append_layer(0, to_device(K[:, :, n_heavy:n], dtype), to_device(V[:, :, n_heavy:n], dtype))
    w = np.concatenate([np.full(n_heavy, 4.0), np.ones(n_tail + 2)])
    for step in range(3):
        q = synth.queries(37, 0, step, B, H * g, d, dtype)
        qt = to_device(q, dtype)
        if step == 0:
            out, m = ctx.decode_attn(0, qt), n
        else:
            m = n + step
            out = ctx.stream_step(0, qt, to_device(K[:, :, m - 1], dtype), to_device(V[:, :, m - 1], dtype), qt.clone())
        assert ctx.debug_scratch_used() == 0
        _check_heads(out.float().cpu().numpy(), K[:, :, :m], V[:, :, :m], w[:m], q, g, dtype, (g, splits, step))
    st = ctx.stats()
    assert st["device_status"] == 0 and st["decode_kernel"] == 1
    if dtype == "fp32":
        out = cuda_lib.decode_attn_static(to_device(K[0, :, :n], dtype), to_device(V[0, :, :n], dtype), n_heavy, T,
                                          to_device(q[0].reshape(H, g, d), dtype)).cpu().numpy()
        _check_heads(out.reshape(1, H * g, d), K[:, :, :n], V[:, :, :n], w[:n], q, g, dtype, "static")
        assert cuda_lib.decode_attn_static_status() == 0
    ctx.close()


def test_static_decode_on_overlapping_streams(cuda_lib):
    """Calls that overlap never share split rows: a long call on one stream beside many short ones on two others (no other
    test of this process takes a block but for the default stream's), and a captured call replayed in order with calls of
    four more streams.  Bit for bit the results of the calls alone."""
    streams = [torch.cuda.Stream() for _ in range(2)]
    more = [torch.cuda.Stream() for _ in range(4)]
    for dtype in (torch.bfloat16, torch.float32):
        gen = torch.Generator(device="cuda").manual_seed(8)
        make = lambda S, n, g: tuple(torch.randn(*s, 128, device="cuda", generator=gen).to(dtype) for s in ((S, n), (S, n), (S, g)))
        big, small = make(100, 16384, 4), [make(2, 2048 + 64 * i, 4) for i in range(8)]
        run = lambda x, out=None: cuda_lib.decode_attn_static(x[0], x[1], 1024, 1, x[2], out)
        want_big, want = run(big), [run(x) for x in small]
        torch.cuda.synchronize()
        for rep in range(5):
            with torch.cuda.stream(streams[0]):
                got_big = run(big)
            got = []
            for i in range(24):
                with torch.cuda.stream(streams[1] if i % 3 else torch.cuda.default_stream()):
                    got.append(run(small[i % 8]))
            torch.cuda.synchronize()
            assert torch.equal(got_big, want_big), (dtype, rep)
            assert all(torch.equal(got[i], want[i % 8]) for i in range(24)), (dtype, rep)
        out = torch.empty_like(small[0][2])
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            run(small[0], out)
        for rep in range(2):
            for i, st in enumerate(more):
                with torch.cuda.stream(st):
                    got = run(small[i])
                st.synchronize()
                assert torch.equal(got, want[i]), (dtype, rep, i)
                out.zero_()
                graph.replay()
                torch.cuda.synchronize()
                assert torch.equal(out, want[0]), (dtype, rep, i)
    assert all(cuda_lib.decode_attn_static_status(st) == 0 for st in [None, *streams, *more])


@pytest.mark.parametrize("d", [128, 64])
def test_combine_reports_any_split_that_does_not_arrive(cuda_lib, d):
    """Each lane of a combining warp waits for words of its own; whichever split is missing, the status word says so, and
    reset makes the context usable again."""
    ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=1, n_q_heads=1, head_dim=d, dtype="bf16", block=64, levels=1, max_tokens=4096)
    ctx.debug_late_split(-1)
    assert ctx.stats()["device_status"] == 0 and ctx.debug_scratch_used() == 0
    K = torch.randn(1, 1, 4096, d, device="cuda").bfloat16()
    for missing in (0, 1, 2, 5, 31, 32, 33, 63):
        ctx.debug_late_split(missing)
        assert ctx.stats()["device_status"] == 1, missing
        ctx.reset()
        assert ctx.stats()["device_status"] == 0 and ctx.debug_scratch_used() == 0, missing
    ctx.stream_append_layer(0, K, K)
    q = torch.randn(1, 1, d, device="cuda").bfloat16()
    out = ctx.decode_attn(0, q).float().cpu().numpy()
    k = K[0, 0].float().cpu().numpy()
    _check(out[0], oracle.weighted_attention(k, k, np.ones(4096), q[0].float().cpu().numpy()), "bf16", d)
    ctx.close()


@pytest.mark.parametrize("merged", [False, True])
def test_reset_empties_the_split_scratch(cuda_lib, merged):
    """Whatever the status word says: words that were left behind without a report would pass for the next launch's."""
    ctx = cuda_lib.Context(n_seqs=1, n_layers=2, n_kv_heads=3, n_q_heads=15, head_dim=128, dtype="bf16", block=64, levels=1,
                           max_tokens=4096)
    if merged:                                        # the scratch of the decode merged over slots exists as well
        K = torch.randn(1, 3, 500, 128, device="cuda").bfloat16()
        for layer in range(2):
            ctx.stream_append_layer(layer, K, K)
        ctx.decode_attn_merged([0, 1], [0, 1], torch.randn(1, 15, 128, device="cuda").bfloat16())
    ctx.debug_late_split(3)
    ctx.debug_set_status(0)
    assert ctx.debug_scratch_used() > 0
    ctx.reset()
    assert ctx.debug_scratch_used() == 0 and ctx.stats()["device_status"] == 0
    ctx.close()


@pytest.mark.parametrize("dtype,d,g,n_heavy,n_tail", [("bf16", 64, 8, 65, 33), ("bf16", 64, 3, 1000, 1), ("bf16", 128, 5, 97, 31), ("bf16", 128, 4, 4100, 95),
                                                      ("fp32", 64, 2, 65, 33), ("fp32", 128, 5, 97, 31)])
def test_rows_of_an_earlier_request_have_no_part(cuda_lib, dtype, d, g, n_heavy, n_tail):
    """A request whose rows held Inf and NaN leaves them behind the segments of the next one, in the tiles that the decode
    kernels read: before and after the fused append, and merged over slots."""
    H, T = 2, 2
    ctx = cuda_lib.Context(n_seqs=1, n_layers=2, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=64, levels=T, max_tokens=20000)
    bad = torch.empty(1, H, 2 * n_heavy + n_tail + 200, d, device="cuda", dtype=ctx.dtype)
    bad[:, :, 0::3], bad[:, :, 1::3], bad[:, :, 2::3] = float("nan"), float("inf"), float("-inf")
    for layer in range(2):
        ctx.cache_load_level(layer, T, bad[:, :, :n_heavy + 100].contiguous(), bad[:, :, :n_heavy + 100].contiguous())
        ctx.stream_append_layer(layer, bad, bad)
    ctx.reset()
    n = n_heavy + n_tail
    K, V = synth.layer_kv("llama", 39, 0, 1, H, n + 2, d, dtype)
    for layer in range(2):
        ctx.cache_load_level(layer, T, to_device(K[:, :, :n_heavy], dtype), to_device(V[:, :, :n_heavy], dtype))
        ctx.stream_append_layer(layer, to_device(K[:, :, n_heavy:n], dtype), to_device(V[:, :, n_heavy:n], dtype))
    w = np.concatenate([np.full(n_heavy, 4.0), np.ones(n_tail + 2)])
    for step in range(3):
        q = synth.queries(39, 0, step, 1, H * g, d, dtype)
        qt = to_device(q, dtype)
        if step == 0 and dtype == "bf16" and d == 128:       # two slots with the same rows
            _check_heads(ctx.decode_attn_merged([0, 1], [0, 1], qt).float().cpu().numpy(), K[:, :, :n], V[:, :, :n], w[:n], q, g, dtype, "merged")
        m = n + step
        if step == 0:
            out = ctx.decode_attn(0, qt)
        else:
            out = ctx.stream_step(0, qt, to_device(K[:, :, m - 1], dtype), to_device(V[:, :, m - 1], dtype), qt.clone())
        _check_heads(out.float().cpu().numpy(), K[:, :, :m], V[:, :, :m], w[:m], q, g, dtype, (g, step))
    assert ctx.stats()["device_status"] == 0
    ctx.close()


@pytest.mark.parametrize("dtype,d,g,n", [("fp32", 128, 1, 33), ("fp32", 128, 8, 1001), ("fp32", 64, 4, 130), ("bf16", 128, 4, 75)])
def test_cuda_core_decode_of_an_infinite_value(cuda_lib, dtype, d, g, n):
    """The last row of a cache, which the batches repeat past the end, holds an infinite value in two columns: there the
    result is that infinity, elsewhere what it is without it."""
    ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=1, n_q_heads=g, head_dim=d, dtype=dtype, block=64, levels=1, max_tokens=4096, gram_path=1)
    gen = torch.Generator(device="cuda").manual_seed(n)
    K, V = (torch.randn(1, 1, n, d, device="cuda", generator=gen).to(ctx.dtype) for _ in range(2))
    q = torch.randn(1, g, d, device="cuda", generator=gen).to(ctx.dtype)
    ctx.stream_append_layer(0, K, V)
    want = ctx.decode_attn(0, q).clone()
    V[0, 0, n - 1, 1], V[0, 0, n - 1, d - 1] = float("inf"), float("-inf")
    want[:, :, 1], want[:, :, d - 1] = float("inf"), float("-inf")
    ctx.reset()
    ctx.stream_append_layer(0, K, V)
    assert torch.equal(ctx.decode_attn(0, q), want)
    ctx.close()


@pytest.mark.parametrize("dtype,d,g", [("fp32", 128, 4), ("bf16", 64, 4), ("bf16", 128, 8)])
def test_replayed_decode_attends_the_rows_of_the_moment(cuda_lib, dtype, d, g):
    """A decode call captured into a graph reads the segment table at each replay: rows appended or compressed since the
    capture count, and rows of an earlier request do not."""
    H, t, n = 2, 64, 700
    ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=t, levels=2, max_tokens=2048)
    K, V = synth.layer_kv("llama", 41, 0, 1, H, n, d, dtype)
    Kd, Vd = to_device(K, dtype), to_device(V, dtype)
    q = synth.queries(41, 0, 0, 1, H * g, d, dtype)
    qt = to_device(q, dtype)
    out = torch.empty_like(qt)
    ctx.stream_append_layer(0, Kd[:, :, :100].contiguous(), Vd[:, :, :100].contiguous())
    ctx.decode_attn(0, qt, out)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.decode_attn(0, qt, out)

    def replay():
        out.zero_()
        graph.replay()
        return out.float().cpu().numpy()

    _check_heads(replay(), K[:, :, :100], V[:, :, :100], np.ones(100), q, g, dtype, "as captured")
    ctx.stream_append_layer(0, Kd[:, :, 100:].contiguous(), Vd[:, :, 100:].contiguous())
    _check_heads(replay(), K, V, np.ones(n), q, g, dtype, "appended")
    ctx.compress()
    for h in range(H):
        kv = [x.float().cpu().numpy() for x in ctx.cache_view(0, 0, h)[:3]]
        assert len(kv[2]) < n
        _check(replay()[0, h * g:(h + 1) * g], oracle.weighted_attention(*kv, q[0, h * g:(h + 1) * g]), dtype, ("compressed", h))
    ctx.reset()
    ctx.stream_append_layer(0, Kd[:, :, 5:8].contiguous(), Vd[:, :, 5:8].contiguous())
    _check_heads(replay(), K[:, :, 5:8], V[:, :, 5:8], np.ones(3), q, g, dtype, "next request")
    assert ctx.stats()["device_status"] == 0 and ctx.debug_scratch_used() == 0
    ctx.close()


@pytest.mark.parametrize("dtype,d", [("fp32", 64), ("bf16", 64), ("bf16", 128)])
def test_host_steps_behind_other_transfers(cuda_lib, dtype, d):
    """Host steps whose operands queue behind 8 GB of other transfers (0.15 s, three times the bound of the other waits)
    attend what the same steps on device tensors attend."""
    B, H, g, n = 1, 2, 4, 512
    pair = [cuda_lib.Context(n_seqs=B, n_layers=1, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=64, levels=1, max_tokens=4096)
            for _ in range(2)]
    host, dev = pair
    gen = torch.Generator(device="cuda").manual_seed(4)
    draw = lambda *s: torch.randn(*s, d, device="cuda", generator=gen).to(host.dtype)
    K, V = draw(B, H, n), draw(B, H, n)
    for ctx in pair:
        ctx.stream_append_layer(0, K, V)
    steps = [(draw(B, H * g), draw(B, H), draw(B, H)) for _ in range(6)]
    pinned = [tuple(x.cpu().pin_memory() for x in step) for step in steps]
    out = torch.empty(6, B, H * g, d, dtype=host.dtype).pin_memory()
    host.stream_step_host(0, *pinned[0], out[0])
    src = torch.zeros(1 << 28, dtype=torch.uint8).pin_memory()
    others = [(torch.cuda.Stream(), torch.empty_like(src, device="cuda")) for _ in range(4)]
    torch.cuda.synchronize()
    for _ in range(8):
        for stream, dst in others:
            with torch.cuda.stream(stream):
                dst.copy_(src, non_blocking=True)
    for i in range(1, 6):
        host.stream_step_host(0, *pinned[i], out[i])
    torch.cuda.synchronize()
    assert host.stats()["device_status"] == 0
    for i, (q, k, v) in enumerate(steps):
        want = dev.stream_step(0, q, k, v, torch.empty_like(q))
        assert torch.equal(out[i], want.cpu()), i
    for ctx in pair:
        ctx.close()


@pytest.mark.parametrize("dtype,g", [("bf16", 1), ("bf16", 4), ("bf16", 8), ("fp32", 1), ("fp32", 4), ("fp32", 8)])
def test_split_decode_over_several_waves(cuda_lib, dtype, g):
    """More streams than half of the resident CTAs, long enough that each is split in three: 480 CTAs, whose combining ones
    poll while the last of the others are not resident yet.  Plain decode, then a step with its append."""
    S, d, T, n_heavy, n_tail = 160, 128, 1, 4001, 130
    n = n_heavy + n_tail
    ctx = cuda_lib.Context(n_seqs=S, n_layers=1, n_kv_heads=1, n_q_heads=g, head_dim=d, dtype=dtype, block=64, levels=T, max_tokens=2 * n)
    gen = torch.Generator(device="cuda").manual_seed(g)
    draw = lambda *s: torch.randn(*s, d, device="cuda", generator=gen).to(ctx.dtype)
    K, V = draw(S, 1, n + 1), draw(S, 1, n + 1)
    ctx.cache_load_level(0, T, K[:, :, :n_heavy].contiguous(), V[:, :, :n_heavy].contiguous())
    ctx.stream_append_layer(0, K[:, :, n_heavy:n].contiguous(), V[:, :, n_heavy:n].contiguous())
    w = np.concatenate([np.full(n_heavy, 2.0), np.ones(n_tail + 1)])
    for m in (n, n + 1):
        q = draw(S, g)
        if m == n:
            out = ctx.decode_attn(0, q)
        else:
            out = ctx.stream_step(0, q, K[:, :, n].contiguous(), V[:, :, n].contiguous(), torch.empty_like(q))
        assert ctx.debug_scratch_used() == 0 and ctx.stats()["device_status"] == 0
        for s in (0, 1, 77, 147, 148, S - 1):
            k, v, x, o = (t.float().cpu().numpy() for t in (K[s, 0, :m], V[s, 0, :m], q[s], out[s]))
            _check(o, oracle.weighted_attention(k, v, w[:m], x), dtype, (m, s))
    ctx.close()


@pytest.mark.parametrize("dtype,d,g", [("fp32", 128, 4), ("bf16", 64, 4), ("bf16", 128, 8)])
def test_replayed_step_puts_its_token_in_the_same_place(cuda_lib, dtype, d, g):
    """A captured step: each replay attends the rows before it and the token that its operands then hold, and stores that
    token in the step's row.  Behind the capture, launches of the stream wait for the append that preceded it."""
    H, n = 2, 700
    ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=64, levels=2, max_tokens=2048)
    K, V = synth.layer_kv("llama", 43, 0, 1, H, n + 3, d, dtype)
    Kd, Vd = to_device(K, dtype), to_device(V, dtype)
    q = synth.queries(43, 0, 0, 1, H * g, d, dtype)
    qt, k, v = to_device(q, dtype), Kd[:, :, n].clone(), Vd[:, :, n].clone()
    out = torch.empty_like(qt)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx.stream_append_layer(0, Kd[:, :, :10].contiguous(), Vd[:, :, :10].contiguous())
        ctx.decode_attn(0, qt, out)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        ctx.stream_append_layer(0, Kd[:, :, 10:n].contiguous(), Vd[:, :, 10:n].contiguous())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.stream_step(0, qt, k, v, out)
    for i in (n, n + 1, n + 2):
        k.copy_(Kd[:, :, i])
        v.copy_(Vd[:, :, i])
        graph.replay()
        rows = [*range(n), i]
        _check_heads(out.float().cpu().numpy(), K[:, :, rows], V[:, :, rows], np.ones(n + 1), q, g, dtype, i)
    with torch.cuda.stream(stream):
        got = ctx.decode_attn(0, qt)
    torch.cuda.synchronize()
    _check_heads(got.float().cpu().numpy(), K[:, :, rows], V[:, :, rows], np.ones(n + 1), q, g, dtype, "behind")
    assert ctx.stats()["device_status"] == 0 and ctx.debug_scratch_used() == 0
    ctx.close()


@pytest.mark.parametrize("B,d,g,rows", [(1, 128, 4, 8192), (8, 128, 5, 1024), (2, 64, 8, 8000), (1, 128, 1, 8211)])
def test_caches_beyond_l2_decode_as_they_do_alone(cuda_lib, B, d, g, rows):
    """Layers that together exceed L2 load part of their tiles to leave it first; each gives what it gives in a context of its own."""
    import torch

    L, H = 4, 8
    gen = torch.Generator(device="cuda").manual_seed(21)
    make = lambda layers: cuda_lib.Context(n_seqs=B, n_layers=layers, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype="bf16", block=64,
                                           levels=2, max_tokens=4 * rows + 64, max_pending=64)
    q, kn, vn = (torch.randn(B, n, d, device="cuda", generator=gen).bfloat16() for n in (H * g, H, H))
    ctx, alone = make(L), make(1)
    for layer in range(L):
        K, V = (torch.randn(B, H, rows, d, device="cuda", generator=gen).bfloat16() for _ in range(2))
        outs = []
        for c, at in ((ctx, layer), (alone, 0)):
            if c is alone:
                c.reset()
            c.cache_load_level(at, 2, K, V)
            step = torch.empty_like(q)
            first = c.decode_attn(at, q)
            c.stream_step(at, q, kn, vn, step)
            outs.append([first, step, c.decode_attn(at, q)])
        assert all(torch.equal(a, b) for a, b in zip(*outs)), layer
    assert ctx.stats()["device_status"] == 0 and alone.stats()["device_status"] == 0
    ctx.close()
    alone.close()
