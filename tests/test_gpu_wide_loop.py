"""Token loop of wide batches (bf16, one launch per leaf, groups of at most 128 sequences) at its edges, against the oracle (fp64): groups of
one sequence to a full row tile, uneven groups, more groups than the loop takes, layers narrower than a group has CTAs, d_ff off the powers of
two (the parts of the down projection), leaves of one position, more units of attention than a group takes in one go.

Tolerance: that of the other bf16 prefill tests (bf16 operands, fp32 accumulation, z rounded to bf16 and fed back through N positions)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TOL = 2e-2
G_NAMES = ("g_attn", "g_mlp", "g_kv", "g_q", "g_k")


def rel_err(got, ref):
    return float(np.abs(got - ref).max() / np.abs(ref).max())


@pytest.mark.parametrize("d,H,dff,B,N,leaf,flags,gains,alibi", [
    (128, 2, 128, 65, 1, 0, 3, G_NAMES, False),
    (128, 2, 384, 128, 33, 16, 3, (), True),
    (256, 4, 640, 129, 17, 16, 3, G_NAMES, False),            # groups of 65 and 64; a leaf of one position
    (384, 6, 1152, 200, 21, 64, 3 | 8, ("g_mlp", "g_k"), True),
    (128, 2, 512, 257, 20, 0, 1, ("g_attn",), False),         # groups of 86, 86 and 85
    (640, 10, 2560, 66, 34, 32, 3, G_NAMES, False),
    (1024, 16, 4096, 70, 5, 0, 3, (), False),
    (1024, 16, 2048, 300, 4, 16, 0, (), True),
    (512, 8, 1024, 1024, 3, 0, 3, ("g_kv",), False),          # eight groups of 18 SMs: several units and tiles per CTA
    (128, 2, 256, 1025, 5, 0, 3, (), False)])                 # one sequence too many: the launches of every position
def test_wide_loop_matches_oracle(d, H, dff, B, N, leaf, flags, gains, alibi):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    wl = inputs.Workload("wide", 1, B, N, d, H, dff, "bf16")
    data = inputs.make_inputs(wl, seed=B + N)
    lw = data["layers"][0]
    rng = np.random.default_rng(B)
    for g in gains:
        lw[g] = inputs.round_to(1.0 + 0.2 * rng.standard_normal(d), "bf16")
    slopes = np.array([2.0 ** (-8.0 * (h + 1) / H) for h in range(H)]) if alibi else None
    ref = layer_seq(RTConfig(d, H, 64, dff, norm_flags=flags, alibi_slopes=slopes, residual_scale=0.7), RTWeights(**lw), data["x"])
    layer = rt.Layer(d, H, dff, dtype="bf16", leaf=leaf, norm_flags=flags, residual_scale=0.7)
    layer.set_weights(dict(lw, alibi_slopes=slopes) if alibi else lw)
    got = layer.prefill(data["x"])
    for name, g_, r_ in zip(("z", "k", "v"), got, ref):
        assert np.isfinite(g_).all(), name
        assert rel_err(g_, r_) <= TOL, (name, rel_err(g_, r_))
    again = layer.prefill(data["x"])
    assert all(np.array_equal(a, b) for a, b in zip(got, again))
