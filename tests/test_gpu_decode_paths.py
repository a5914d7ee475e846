"""Decode kernels at the sizes where their tiling, their combine and their fused append can go wrong, against the
oracle's weighted attention over the same rows.  Tolerances are those of the other decode tests: 2e-3 for bf16 (the
final rounding), 1e-5 for fp32."""
import numpy as np
import pytest
import torch

import oracle
from paper_2502_07861_b200 import synth
from parity_util import rel_l2, to_device

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-5, "bf16": 2e-3}


def _check(out, K, V, w, q, g, tol, what):
    for h in range(K.shape[1]):
        ref = oracle.weighted_attention(K[0, h], V[0, h], w, q[0, h * g:(h + 1) * g])
        assert rel_l2(out[0, h * g:(h + 1) * g], ref) <= tol, (what, h)


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
        _check(out.float().cpu().numpy(), K[:, :, :m], V[:, :, :m], w[:m], q, g, TOL["bf16"], (g, splits, step))
    st = ctx.stats()
    assert st["device_status"] == 0 and st["decode_kernel"] == 2
    Kg, Vg, wg, idx = ctx.cache_view(0, 0, H - 1)
    assert np.array_equal(Kg.float().cpu().numpy(), K[0, H - 1]) and np.array_equal(Vg.float().cpu().numpy(), V[0, H - 1])
    assert np.array_equal(wg.cpu().numpy(), w.astype(np.float32))
    ctx.close()
