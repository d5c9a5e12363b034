"""The reverse loop of the backward pass at the edges of its kernels, bf16, against the gradient oracle (fp64): mat-vecs of up
to eight sequences (narrow widths where CTAs own no columns, leaves of 1, 63, 64 and 65 positions; slices of a larger batch), three-term dense
products of 9 to 32 sequences and, above, dense products over the batch (leaves of 16 positions; batches off the 128-row tiles; one to eight
parts per contraction).

Tolerance: every product takes bf16 operands or a three-term bf16 split and accumulates in fp32, so a gradient carries a few roundings of
2^-9 relative to its largest entries; 2e-2 is that of the other backward tests."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-2
G_NAMES = ("g_attn", "g_mlp", "g_kv", "g_q", "g_k")


def _check(d, H, dff, B, N, flags, gains, alibi, alpha):
    from oracle import RTConfig, RTWeights, layer_grad
    from paper_2604_21215_b200 import inputs, rt
    wl = inputs.Workload("bwd", 1, B, N, d, H, dff, "bf16")
    data = inputs.make_inputs(wl, seed=100 * B + N)
    lw, x = data["layers"][0], data["x"]
    rng = np.random.default_rng(B + N)
    for g in gains:
        lw[g] = inputs.round_to(1.0 + 0.2 * rng.standard_normal(d), "bf16")
    slopes = np.array([2.0 ** (-8.0 * (h + 1) / H) for h in range(H)]) if alibi else None
    dz = rng.standard_normal(x.shape).astype(np.float32).astype(np.float64)
    cfg = RTConfig(d, H, 64, dff, norm_flags=flags, residual_scale=alpha, alibi_slopes=slopes)
    z_ref, dx_ref, g_ref = layer_grad(cfg, RTWeights(**lw), x, dz)
    layer = rt.Layer(d, H, dff, dtype="bf16", norm_flags=flags, residual_scale=alpha)
    layer.set_weights(dict(lw, alibi_slopes=slopes) if alibi else lw)
    z = inputs.round_to(z_ref, "bf16")
    dx, g = layer.backward(x, z, dz)
    dx2, g2 = layer.backward(x, z, dz)
    assert np.array_equal(dx, dx2) and all(np.array_equal(g[n], g2[n]) for n in g)
    assert np.abs(dx - dx_ref).max() <= TOL * np.abs(dx_ref).max()
    for name, got in g.items():
        ref = g_ref[name]
        scale = np.abs(ref).max() or np.abs(dx_ref).max()               # gradients that are zero: up to the rounding of the others
        assert np.abs(got - ref).max() <= TOL * scale, name


@pytest.mark.parametrize("d,H,dff,B,N,flags,gains,alibi,alpha", [
    (128, 2, 256, 1, 1, 3, G_NAMES, False, 1.0),
    (64, 1, 128, 1, 65, 3, (), True, 1.0),
    (128, 2, 512, 4, 64, 3, G_NAMES, False, 0.5),
    (192, 3, 768, 5, 63, 3 | 8, ("g_k", "g_mlp"), True, 1.0),
    (256, 4, 640, 8, 66, 3, (), False, 1.0),
    (384, 6, 1536, 2, 130, 3, G_NAMES, False, 1.0),
    (128, 2, 256, 9, 70, 1, ("g_kv",), False, 1.0),
    (320, 5, 960, 16, 33, 3, (), True, 0.7),
    (128, 2, 384, 32, 20, 0, (), False, 1.0),
    (192, 3, 768, 12, 30, 3, (), False, 1.0),
    (256, 4, 512, 24, 35, 3 | 8, G_NAMES, True, 1.0),
    (1024, 16, 4096, 17, 6, 3, ("g_attn",), False, 1.0),
    (1024, 16, 4096, 3, 9, 3, ("g_attn",), False, 1.0)])
def test_loop_of_up_to_32_sequences(d, H, dff, B, N, flags, gains, alibi, alpha):
    _check(d, H, dff, B, N, flags, gains, alibi, alpha)


@pytest.mark.parametrize("d,H,dff,B,N,flags,gains,alibi,alpha", [
    (128, 2, 256, 33, 1, 3, G_NAMES, False, 1.0),                            # a single position: the operands outgrow one row block
    (128, 2, 384, 40, 17, 3, ("g_k", "g_kv"), True, 0.6),                    # a leaf of one position beside a full one
    (256, 4, 1024, 65, 16, 3 | 8, G_NAMES, False, 1.0),
    (512, 8, 2048, 129, 5, 3, (), True, 1.0),                                # second row tile of one row
    (1024, 16, 1024, 34, 6, 1, ("g_mlp",), False, 0.5),
    # With no norms at all this case is ill conditioned (one of the 130 sequences has gradients of 916; the fp64 oracle itself moves by 187
    # there when the weights change by up to 2^-9 of themselves), so it keeps the pre-norms; without them only half the length is used.
    (128, 2, 512, 130, 35, 1, (), False, 1.0),
    (128, 2, 512, 130, 18, 0, (), False, 0.5),
    (256, 4, 512, 300, 20, 3, G_NAMES, True, 1.0),                           # three groups
    (128, 2, 256, 1030, 18, 3, ("g_k", "g_kv"), False, 1.0)])                # too many groups: the launches of every position
def test_dense_products_over_wide_batches(d, H, dff, B, N, flags, gains, alibi, alpha):
    _check(d, H, dff, B, N, flags, gains, alibi, alpha)


def test_gains_at_any_address():
    # the backward pass has never asked for aligned gains: views into one packed array give the bits of separate arrays
    import torch
    from paper_2604_21215_b200 import inputs, rt
    d, H, dff, B, N = 256, 4, 1024, 3, 70
    wl = inputs.Workload("gains", 1, B, N, d, H, dff, "bf16")
    data = inputs.make_inputs(wl, seed=8)
    lw = data["layers"][0]
    rng = np.random.default_rng(2)
    for g in G_NAMES:
        lw[g] = inputs.round_to(1.0 + 0.2 * rng.standard_normal(d), "bf16")
    layer = rt.Layer(d, H, dff, dtype="bf16")
    layer.set_weights(lw)
    z, _, _ = layer.prefill(data["x"])
    dz = rng.standard_normal(z.shape)
    want = layer.backward(data["x"], z, dz)
    packed = torch.empty(1 + 5 * (d + 1), dtype=torch.bfloat16, device=layer.device)
    for i, g in enumerate(G_NAMES):
        view = packed[1 + i * (d + 1):][:d]                     # the first four 2, 4, 6 and 0 bytes off a multiple of eight
        view.copy_(torch.as_tensor(lw[g]))
        setattr(layer.w, g, view.data_ptr())
    got = layer.backward(data["x"], z, dz)
    assert np.array_equal(got[0], want[0])
    for n in want[1]:
        assert np.array_equal(got[1][n], want[1][n]), n
