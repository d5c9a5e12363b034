"""The cluster kernel for small layers at its edges: number of sequences per cluster (1, 2, 3), leaf lengths around two
lanes per query, one to three leaves, the widest layers that fit, MLP widths that leave warps without rows."""
import numpy as np
import pytest

from parity_metrics import check_tensor

pytestmark = pytest.mark.gpu
TOL = {"f32": 1e-4, "bf16": 2e-2}


@pytest.mark.parametrize("dtype,d,H,dff,B,N,leaf,alibi", [
    ("f32", 64, 1, 64, 1, 1, 0, False), ("f32", 64, 1, 320, 7, 2, 0, True), ("f32", 128, 2, 512, 8, 63, 0, False),
    ("f32", 256, 4, 1024, 3, 65, 0, True), ("f32", 128, 2, 192, 15, 130, 32, False), ("f32", 192, 3, 768, 21, 20, 16, False),
    ("bf16", 384, 6, 1536, 2, 129, 0, False), ("bf16", 320, 5, 1280, 14, 66, 0, True), ("bf16", 128, 2, 512, 16, 64, 0, False)])
def test_small_layer_matches_oracle(dtype, d, H, dff, B, N, leaf, alibi):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    wl = inputs.Workload("small", 1, B, N, d, H, dff, dtype)
    data = inputs.make_inputs(wl, seed=77 + N)
    lw = data["layers"][0]
    rng = np.random.default_rng(N)
    for g in ("g_attn", "g_mlp", "g_kv", "g_q", "g_k"):
        lw[g] = inputs.round_to(1.0 + 0.2 * rng.standard_normal(d), dtype)
    slopes = [2.0 ** (-8.0 * (h + 1) / H) for h in range(H)] if alibi else None
    ref = layer_seq(RTConfig(d, H, 64, dff, residual_scale=0.8, alibi_slopes=slopes), RTWeights(**lw), data["x"])
    layer = rt.Layer(d, H, dff, dtype=dtype, leaf=leaf, residual_scale=0.8)
    layer.set_weights(dict(lw, alibi_slopes=slopes))
    got = layer.prefill(data["x"])
    for name, a, b in zip(("z", "k", "v"), got, ref):
        check_tensor(f"small {dtype} d={d} B={B} N={N}", name, a, b, TOL[dtype])


@pytest.mark.parametrize("B,N", [(14, 70), (15, 70), (28, 40), (32, 40), (64, 20)])
def test_batches_around_the_bound_of_the_cluster_kernel(B, N):
    # d = 384: one and two rounds of clusters, and the batches that the tensor-core leaf kernel and the group kernel take instead
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    d, H, dff = 384, 6, 1536
    data = inputs.make_inputs(inputs.Workload("bound", 1, B, N, d, H, dff, "bf16"), seed=B)
    lw = data["layers"][0]
    ref = layer_seq(RTConfig(d, H, 64, dff), RTWeights(**lw), data["x"])
    layer = rt.Layer(d, H, dff, dtype="bf16")
    layer.set_weights(lw)
    for name, a, b in zip(("z", "k", "v"), layer.prefill(data["x"]), ref):
        check_tensor(f"bound B={B}", name, a, b, TOL["bf16"])
