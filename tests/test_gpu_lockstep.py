"""Compress over lockstep streams derives its calls from their index; with the call records on, the same calls travel as
lists.  Both must leave bit-identical caches behind, whatever the number of blocks, held halves, remainders, windows,
layers and batches."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _views(ctx):
    c = ctx.cfg
    return [x.clone() for s in range(c.n_seqs) for l in range(c.n_layers) for h in range(c.n_kv_heads) for x in ctx.cache_view(s, l, h)]


@pytest.mark.parametrize("d,dtype,t,T,W,center,chunks", [
    (128, "bf16", 128, 1, 0, 0, (128, 129, 511)),
    (128, "bf16", 128, 3, 37, 0, (640, 384, 100, 1500, 128, 896)),
    (128, "bf16", 256, 2, 0, 1, (256, 768, 1300)),
    (128, "bf16", 192, 2, 5, 0, (400, 192, 777)),
    (64, "fp32", 64, 3, 0, 0, (64, 65, 700, 63, 320)),
    (128, "fp32", 192, 2, 0, 0, (384, 192, 1000)),
    (64, "bf16", 64, 2, 100, 1, (333, 64, 500)),
    (128, "bf16", 2048, 2, 0, 0, (4096, 2048, 6200)),
])
@pytest.mark.parametrize("per_layer", [False, True])
def test_lockstep_compress_equals_the_listed_calls(cuda_lib, d, dtype, t, T, W, center, chunks, per_layer):
    B, L, H, g = 2, 2, 3, 2
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(t + T)
    pair = []
    for record in (False, True):
        ctx = cuda_lib.Context(n_seqs=B, n_layers=L, n_kv_heads=H, n_q_heads=H * g, head_dim=d, dtype=dtype, block=t, levels=T,
                               max_tokens=sum(chunks), max_pending=max(chunks), recent_window=W, center_keys=center, seed=9,
                               c_override=0.75)
        ctx.debug_enable(record)
        pair.append(ctx)
    for n in chunks:
        for l in range(L):
            K = (0.3 * torch.randn(B, H, n, d, device="cuda", generator=gen)).to(tdt)
            V = torch.randn(B, H, n, d, device="cuda", generator=gen).to(tdt)
            for ctx in pair:
                ctx.stream_append_layer(l, K, V)
                if per_layer:
                    ctx.compress_layer(l)
        if not per_layer:
            for ctx in pair:
                ctx.compress()
        a, b = (_views(ctx) for ctx in pair)
        assert all(torch.equal(x, y) for x, y in zip(a, b)), n
    q = torch.randn(B, H * g, d, device="cuda", generator=gen).to(tdt)
    assert torch.equal(pair[0].decode_attn(1, q), pair[1].decode_attn(1, q))
    assert pair[0].stats()["calls_run"] == pair[1].stats()["calls_run"]
    assert pair[0].stats()["walk_fails"] == pair[1].stats()["walk_fails"]
    for ctx in pair:
        assert ctx.stats()["device_status"] == 0
        ctx.close()


def test_lockstep_compress_in_several_batches(cuda_lib):
    """More calls than the pools hold at once (1 GiB of pool rows: 4096 calls of 256 rows): batches of whole streams."""
    S, t, T, n = 700, 128, 2, 1100
    pair = [cuda_lib.Context(n_seqs=1, n_layers=1, n_kv_heads=S, n_q_heads=S, head_dim=128, dtype="bf16", block=t, levels=T,
                             max_tokens=n, seed=3, c_override=0.75) for _ in range(2)]
    pair[1].debug_enable(True)
    K = (0.3 * torch.randn(1, S, n, 128, device="cuda")).to(torch.bfloat16)
    V = torch.randn(1, S, n, 128, device="cuda").to(torch.bfloat16)
    for ctx in pair:
        ctx.stream_append_layer(0, K, V)
        ctx.compress()
    for h in (0, 511, 512, 600, 699):
        assert all(torch.equal(x, y) for x, y in zip(pair[0].cache_view(0, 0, h), pair[1].cache_view(0, 0, h))), h
    for ctx in pair:
        assert ctx.stats()["device_status"] == 0
        ctx.close()
