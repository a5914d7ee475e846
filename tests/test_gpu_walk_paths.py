"""SoftmaxBalance kernels at the block sizes where their tiling ends raggedly, against the oracle by the teacher-forced
procedure of parity_util (signs, margins, kept sets, stored rows, running correlations).  Tolerances of S: those of the other
parity tests (2e-4 on tensor cores, 5e-4 with key centering, 2e-5 on CUDA cores)."""
import numpy as np
import pytest

from paper_2502_07861_b200 import synth
from parity_util import Harness

pytestmark = pytest.mark.gpu


def _run(cuda_lib, d, dtype, t, T, center, tol, walk_kernel, **kw):
    B, H, n = 1, 2, 5 * t + 17
    K, V = synth.layer_kv("llama", 61, 0, B, H, n, d, dtype)
    K = synth.round_to(0.06 * K + (1.5 if center else 0.0), dtype)
    hz = Harness(cuda_lib, B=B, L=1, H=H, g=1, d=d, dtype=dtype, t=t, T=T, N=n, seed=6, c_override=0.75, center_keys=center, **kw)
    cut = 3 * t - 5
    hz.append_layer(0, K[:, :, :cut], V[:, :, :cut])
    hz.compress()
    hz.append_layer(0, K[:, :, cut:], V[:, :, cut:])
    hz.compress()
    tot, _ = hz.check_all(tol)
    assert tot == B * H * t * sum(5 >> l for l in range(T))
    st = hz.ctx.stats()
    assert st["device_status"] == 0 and st["walk_kernel"] == walk_kernel
    hz.ctx.close()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("t,T,center", [(128, 1, 0), (192, 2, 0), (192, 1, 1), (320, 1, 0), (1088, 1, 0), (2048, 1, 0), (2560, 1, 0),
                                        (1856, 1, 1), (2048, 1, 1)])
def test_tensor_core_walk_with_ragged_panels(cuda_lib, d, t, T, center):
    """Whole panels and a last panel of 64 tokens; d = 64 operands are a single 64-dim box."""
    _run(cuda_lib, d, "bf16", t, T, center, 5e-4 if center else 2e-4, 2)


@pytest.mark.parametrize("d,dtype,t,T,center", [(64, "fp32", 64, 2, 0), (64, "fp32", 128, 1, 1), (128, "fp32", 192, 2, 0), (128, "fp32", 640, 1, 0),
                                                (64, "fp32", 1024, 1, 0), (128, "bf16", 64, 2, 1), (64, "bf16", 320, 1, 0)])
def test_cuda_core_walk(cuda_lib, d, dtype, t, T, center):
    """One workspace tile, fewer tiles than stages and more, an odd number of row tiles (column blocks that reach past the
    call), small and large launches of the kernel-matrix kernel."""
    _run(cuda_lib, d, dtype, t, T, center, 5e-4 if center else 2e-5, 1, gram_path=1)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("t,T,center", [(128, 2, 0), (192, 1, 1), (320, 1, 0), (640, 1, 0), (1024, 1, 0)])
def test_kernel_matrix_of_fp32_rows_on_tensor_cores(cuda_lib, d, t, T, center):
    """Whole panels and a last panel of 64 tokens, columns that are among the tile's rows and others; the tolerances of FFMA."""
    _run(cuda_lib, d, "fp32", t, T, center, 5e-4 if center else 2e-5, 1)


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), 3.4e38])
def test_fp32_call_with_an_infinite_row(cuda_lib, value):
    """A row whose norm is infinite: its call is formed as on the CUDA cores, bit by bit."""
    import torch

    S, t, d = 2, 192, 64
    gen = torch.Generator(device="cuda").manual_seed(9)
    K = 0.3 * torch.randn(1, S, t, d, device="cuda", generator=gen)
    V = torch.randn(1, S, t, d, device="cuda", generator=gen)
    K[0, 0, 70, 5] = value
    views = []
    for path in (0, 1):
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="fp32", block=t, levels=1, max_tokens=t,
                               seed=3, c_override=0.75, gram_path=path)
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
        views.append(ctx.cache_view(0, 0, 0))
        assert ctx.stats()["device_status"] == 0
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*views))


@pytest.mark.parametrize("d,t,center,kind", [(64, 128, 0, "infinite"), (128, 320, 0, "infinite"), (128, 256, 1, "infinite"),
                                             (64, 192, 0, "uneven"), (128, 256, 1, "uneven")])
def test_fp32_calls_formed_by_ffma(cuda_lib, d, t, center, kind):
    """Calls whose rows are not split give the running sums of the CUDA cores bit by bit: whole panels and a last one of 64
    tokens, columns that are among the tile's rows and others, key shifts."""
    import torch

    S = 2
    gen = torch.Generator(device="cuda").manual_seed(t)
    K = 0.1 * torch.randn(1, S, t, d, device="cuda", generator=gen)
    V = torch.randn(1, S, t, d, device="cuda", generator=gen)
    if kind == "infinite":
        V[0, :, t - 1, 3] = float("inf")                # the last token's alone: every other sum stays finite
    else:
        V *= torch.where(torch.arange(t, device="cuda")[:, None] % d == torch.arange(d, device="cuda"), 1.0, 1e-4)
    runs = []
    for path in (0, 1):
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="fp32", block=t, levels=1, max_tokens=t,
                               seed=3, c_override=0.75, center_keys=center, r_value=float(d) ** 0.5, gram_path=path)
        ctx.debug_enable()
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
        runs.append([x for h in range(S) for x in ctx.debug_call(0, 0, h, 0, 0)[:2]])
        assert ctx.stats()["device_status"] == 0
        ctx.close()
    assert float(runs[0][1][: t - 1].abs().max()) > (1e-3 if kind == "infinite" else 1e-7)      # sums of something
    assert all(torch.equal(x.nan_to_num(7.0), y.nan_to_num(7.0)) for x, y in zip(*runs))


def test_cuda_core_walk_in_groups_of_calls(cuda_lib):
    """More calls than the workspace holds (512 MB: 60 calls of 2048 tokens), against the walk of each stream alone."""
    import torch

    S, t, n = 62, 2048, 2048
    gen = torch.Generator(device="cuda").manual_seed(5)
    K = 0.1 * torch.randn(1, S, n, 64, device="cuda", generator=gen)
    V = torch.randn(1, S, n, 64, device="cuda", generator=gen)
    ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=64, dtype="fp32", block=t, levels=1, max_tokens=n,
                           seed=3, c_override=0.75)
    ctx.stream_append_layer(0, K, V)
    ctx.compress()
    one = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=64, dtype="fp32", block=t, levels=1, max_tokens=n,
                           seed=3, c_override=0.75)
    for h in (0, 59, 60, 61):
        one.stream_append(0, 0, h, K[0, h], V[0, h])
        one.compress()
        assert all(torch.equal(a, b) for a, b in zip(ctx.cache_view(0, 0, h), one.cache_view(0, 0, h))), h
    assert ctx.stats()["device_status"] == 0 and one.stats()["device_status"] == 0
    ctx.close()
    one.close()


@pytest.mark.parametrize("center", [0, 1])
def test_tensor_core_walk_beyond_l2(cuda_lib, center):
    """Resident calls whose rows exceed L2 (148 of 2048 tokens) keep what the walk of each stream alone keeps."""
    import torch

    S, t, d = 150, 2048, 128
    gen = torch.Generator(device="cuda").manual_seed(11)
    K = (0.3 * torch.randn(1, S, t, d, device="cuda", generator=gen)).bfloat16()
    V = torch.randn(1, S, t, d, device="cuda", generator=gen).bfloat16()
    make = lambda: cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="bf16", block=t, levels=1,
                                    max_tokens=t, seed=3, c_override=0.75, center_keys=center)
    ctx, one = make(), make()
    ctx.stream_append_layer(0, K, V)
    ctx.compress()
    for h in (0, 1, S // 2, S - 1):
        one.stream_append(0, 0, h, K[0, h], V[0, h])
        one.compress()
        assert all(torch.equal(a, b) for a, b in zip(ctx.cache_view(0, 0, h), one.cache_view(0, 0, h))), h
    assert ctx.stats()["device_status"] == 0 and ctx.stats()["walk_kernel"] == 2 and one.stats()["device_status"] == 0
    ctx.close()
    one.close()


@pytest.mark.parametrize("d,dtype,large,small", [(128, "bf16", 3072, 128), (64, "bf16", 4096, 192), (64, "fp32", 4096, 64)])
def test_contexts_with_other_blocks_live_side_by_side(cuda_lib, d, dtype, large, small):
    """A kernel's shared-memory limit belongs to the device: the context with the large blocks compresses after one with
    small blocks was created and used, and keeps what it keeps alone."""
    import torch

    def make(t):
        return cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=1, n_q_heads=1, head_dim=d, dtype=dtype, block=t, levels=1,
                                max_tokens=t, seed=2, c_override=0.75)

    def compress(ctx):
        gen = torch.Generator(device="cuda").manual_seed(3)
        K, V = (0.3 * torch.randn(1, 1, ctx.cfg.block, d, device="cuda", generator=gen).to(ctx.dtype) for _ in range(2))
        ctx.reset()
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
        return ctx.cache_view(0, 0, 0)

    a = make(large)
    alone = compress(a)
    b = make(small)
    compress(b)
    assert all(torch.equal(x, y) for x, y in zip(alone, compress(a)))
    a.close()
    b.close()


@pytest.mark.parametrize("t", [1728, 1792, 2048])
def test_sums_do_not_depend_on_the_launch(cuda_lib, t):
    """The running correlations S_j of a call, bit for bit: alone and among 150 calls, on both sides of the block size where
    the order of the columns changes.  (Sums in another order differ in their last bits, and a token near its threshold then
    falls differently.)"""
    import torch

    S, d = 150, 128
    gen = torch.Generator(device="cuda").manual_seed(t)
    K = (0.3 * torch.randn(1, S, t, d, device="cuda", generator=gen)).bfloat16()
    V = torch.randn(1, S, t, d, device="cuda", generator=gen).bfloat16()
    pair = []
    for _ in range(2):
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="bf16", block=t, levels=1,
                               max_tokens=t, seed=3, c_override=0.75)
        ctx.debug_enable()
        pair.append(ctx)
    pair[0].stream_append_layer(0, K, V)
    pair[0].compress()
    for h in (0, 77, S - 1):
        pair[1].stream_append(0, 0, h, K[0, h], V[0, h])
        pair[1].compress()
        (eta, sums, p), alone = (ctx.debug_call(0, 0, h, 0, 0) for ctx in pair)
        assert torch.equal(sums, alone[1]) and torch.equal(eta, alone[0]) and torch.equal(p, alone[2]), h
        assert float(sums.abs().max()) > 1e-3           # sums of something
    for ctx in pair:
        assert ctx.stats()["device_status"] == 0 and ctx.stats()["walk_kernel"] == 2
        ctx.close()


def test_cuda_core_walk_with_little_memory(cuda_lib):
    """A context whose workspace (62 calls: 536 MB) finds no room beside its 230 MB of rows takes a smaller one, and keeps
    what it keeps with the whole workspace."""
    import torch

    S, t, d = 62, 2048, 64
    gen = torch.Generator(device="cuda").manual_seed(6)
    K = 0.1 * torch.randn(1, S, t, d, device="cuda", generator=gen)
    V = torch.randn(1, S, t, d, device="cuda", generator=gen)

    def kept():
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="fp32", block=t, levels=1,
                               max_tokens=t, seed=3, c_override=0.75)
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
        idx = [ctx.cache_view(0, 0, h)[3] for h in range(S)]
        st = ctx.stats()
        assert st["device_status"] == 0 and st["walk_kernel"] == 1
        ctx.close()
        return idx, st["bytes_resident"]

    want, whole = kept()
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - (500 << 20), dtype=torch.uint8, device="cuda")
    got, small = kept()
    del hog
    torch.cuda.empty_cache()
    assert small < whole - (200 << 20)
    assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_centered_call_beyond_a_fixed_radius(cuda_lib):
    """Keys that a fixed radius is far too small for: the exponential overflows, and the sum with it, on both kernel families.
    (Token 0 and token 200 share a key; token 0 is a column of token 200's panel.)"""
    import torch

    t, d = 256, 128
    gen = torch.Generator(device="cuda").manual_seed(4)
    K = torch.zeros(1, 1, t, d, device="cuda")
    K[0, 0, 0] = K[0, 0, 200] = 3.5
    V = torch.rand(1, 1, t, d, device="cuda", generator=gen)
    sums = []
    for path in (0, 1):
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=1, n_q_heads=1, head_dim=d, dtype="bf16", block=t, levels=1, max_tokens=t,
                               seed=3, c_override=0.75, center_keys=1, r_key=1.0, gram_path=path)
        ctx.debug_enable()
        ctx.stream_append_layer(0, K.bfloat16(), V.bfloat16())
        ctx.compress()
        sums.append(ctx.debug_call(0, 0, 0, 0, 0)[1])
        assert ctx.stats()["device_status"] == 0 and ctx.stats()["walk_kernel"] == 2 - path
        ctx.close()
    assert torch.isinf(sums[1][200]) and sums[0][200].abs() == sums[1][200].abs()
    assert torch.isfinite(sums[0][:200]).all()


def _pair_rows(kind, n, d, gen):
    """Two sets of n rows."""
    import torch

    a, b = (torch.randn(n, d, device="cuda", dtype=torch.float64, generator=gen) for _ in range(2))
    if kind.startswith("one channel x"):                # another channel in either row
        at = torch.arange(n, device="cuda")
        size = float(kind.split("x")[1])
        for x, c in ((a, at % (d // 2)), (b, d // 2 + at * 7 % (d // 2))):
            x[at, c] = size * (1 + torch.rand(n, device="cuda", dtype=torch.float64, generator=gen))
    elif kind == "one of two":
        a[:, 3] *= 1000
    elif kind == "one value":
        a[:], b[:] = a[:, :1].clone(), b[:, :1].clone()
    elif kind == "heavy tails":
        a, b = (x / torch.randn(n, d, device="cuda", dtype=torch.float64, generator=gen).abs() for x in (a, b))
    elif kind == "hot channels":
        scale = torch.ones(d, device="cuda", dtype=torch.float64)
        scale[:4] = 10
        a, b = (a + 0.5) * scale, (b + 0.5) * scale
    elif kind == "mean":
        a, b = 7 + 1e-3 * a, 7 + 1e-3 * b
    elif kind == "sparse":
        keep = torch.rand(n, d, device="cuda", generator=gen)
        a, b = a * (keep < 0.3), b * (keep < 0.3)
    elif kind.startswith("halves x"):                   # the large elements of either row meet small ones
        a[:, : d // 2] *= float(kind.split("x")[1])
        b[:, d // 2:] *= float(kind.split("x")[1])
    return a.float(), b.float()


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("t,first,second", [(128, 0, 1), (256, 0, 128)])
@pytest.mark.parametrize("kind", ["flat", "one channel x100", "one channel x1000", "one channel x30000", "one channel x1e6", "one of two",
                                  "one value", "heavy tails", "hot channels", "mean", "sparse", "halves x0.03", "halves x0.001"])
def test_fp32_products_are_as_precise_as_ffma(cuda_lib, d, t, first, second, kind):
    """Products of value rows against 64 bits; the limit is the error of the CUDA cores.  Tokens first + s m and second + s m have
    the m-th axis as their key (of length r_key: the kernel is 1 between them and 0 elsewhere), so that a token's running sum is
    the one product, up to the other token's sign.  Neighbours share a tile whose columns are among its rows, tokens 128 apart do not."""
    import torch

    S, n, r = 24, 64, 64.0
    step = 2 if second == 1 else 1
    gen = torch.Generator(device="cuda").manual_seed(d + t)
    i, j = (x + step * torch.arange(n, device="cuda") for x in (first, second))
    K, V = (torch.zeros(1, S, t, d, device="cuda") for _ in range(2))
    for x in (i, j):
        K[0, :, x, torch.arange(n, device="cuda")] = r
    a, b = (x.reshape(S, n, d) for x in _pair_rows(kind, S * n, d, gen))
    V[0, :, i], V[0, :, j] = a, b
    exact, size = (a.double() * b.double()).sum(-1), (a.double() * b.double()).abs().sum(-1)
    errors = []
    for path in (0, 1):
        ctx = cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=d, dtype="fp32", block=t, levels=1, max_tokens=t,
                               seed=3, gram_path=path, r_key=r, r_value=1.0)
        ctx.debug_enable()
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
        got = torch.stack([s[j] * e[i].float() for e, s, _ in (ctx.debug_call(0, 0, h, 0, 0) for h in range(S))])
        assert ctx.stats()["device_status"] == 0
        ctx.close()
        errors.append((got.double() - exact).abs() / size)
    assert float(errors[1].max()) < 3e-6                # sums of the right products
    for of in (lambda e: e.square().mean().sqrt(), torch.median):
        assert float(of(errors[0])) <= float(of(errors[1])), (float(of(errors[0])), float(of(errors[1])))
