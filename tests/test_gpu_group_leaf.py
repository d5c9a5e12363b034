"""The group leaf kernel (several jobs side by side, a group of SMs each) against the oracle: widths whose row slices are ragged
tiles, MLPs that are no multiple of the width, slices of at most eight and of sixteen sequences, one to several windows and leaves; and
the layers of a stack side by side: fewer and more layers than places, leaves that absorb earlier pairs with and without a tile launch."""
import numpy as np
import pytest

from parity_metrics import check_tensor

pytestmark = pytest.mark.gpu


def _gains(lw, d, seed):
    from paper_2604_21215_b200 import inputs
    rng = np.random.default_rng(seed)
    for g in ("g_attn", "g_mlp", "g_kv", "g_q", "g_k"):
        lw[g] = inputs.round_to(1.0 + 0.2 * rng.standard_normal(d), "bf16")


@pytest.mark.parametrize("d,H,dff,B,N,leaf,gains,alibi", [
    (512, 8, 2048, 17, 18, 0, False, False), (768, 12, 3072, 33, 70, 0, True, False), (640, 10, 2560, 19, 130, 0, True, True),
    (896, 14, 3584, 20, 33, 32, False, False), (1024, 16, 4096, 64, 20, 16, True, False), (1024, 16, 3872, 32, 67, 0, False, True),
    (512, 8, 96, 50, 1, 0, False, False), (512, 8, 256, 50, 1, 0, False, False), (512, 8, 96, 20, 20, 0, False, False)])
def test_slices_match_oracle(d, H, dff, B, N, leaf, gains, alibi):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    wl = inputs.Workload("groups", 1, B, N, d, H, dff, "bf16")
    data = inputs.make_inputs(wl, seed=300 + N)
    lw = data["layers"][0]
    if gains:
        _gains(lw, d, N)
    slopes = [2.0 ** (-8.0 * (h + 1) / H) for h in range(H)] if alibi else None
    ref = layer_seq(RTConfig(d, H, 64, dff, residual_scale=0.8, alibi_slopes=slopes), RTWeights(**lw), data["x"])
    layer = rt.Layer(d, H, dff, dtype="bf16", leaf=leaf, residual_scale=0.8)
    layer.set_weights(dict(lw, alibi_slopes=slopes))
    got = layer.prefill(data["x"])
    for name, a, b in zip(("z", "k", "v"), got, ref):
        check_tensor(f"groups d={d} B={B} N={N}", name, a, b, 2e-2)


@pytest.mark.parametrize("L,d,H,dff,B,N,leaf,gains,alibi", [
    (2, 512, 8, 2048, 1, 2, 0, False, False), (5, 512, 8, 1024, 3, 77, 0, True, True), (9, 448, 7, 896, 1, 17, 0, False, False),
    (3, 768, 12, 3072, 9, 300, 0, True, True), (6, 512, 8, 512, 2, 230, 16, False, True), (4, 640, 10, 1280, 16, 130, 64, True, False),
    (9, 448, 7, 896, 1, 130, 0, True, False), (4, 640, 10, 1280, 16, 200, 64, False, True)])
def test_layers_side_by_side_match_oracle(L, d, H, dff, B, N, leaf, gains, alibi):
    from oracle import RTConfig, RTWeights, stack_prefill
    from paper_2604_21215_b200 import inputs, rt
    V = 91
    wl = inputs.Workload("wave", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L))
    data = inputs.make_inputs(wl, seed=500 + N)
    if gains:
        for i, lw in enumerate(data["layers"]):
            _gains(lw, d, N + i)
    slopes = [2.0 ** (-8.0 * (h + 1) / H) for h in range(H)] if alibi else None
    ocfg = RTConfig(d, H, 64, dff, residual_scale=wl.residual_scale, alibi_slopes=slopes)
    hid_ref, logits_ref, caches_ref = stack_prefill(ocfg, [RTWeights(**lw) for lw in data["layers"]], data["emb"], None, data["ids"])
    st = rt.Stack(L, d, H, dff, V, dtype="bf16", leaf=leaf, residual_scale=wl.residual_scale)
    st.set_weights([dict(lw, alibi_slopes=slopes) for lw in data["layers"]], data["emb"])
    hid, logits = st.prefill(data["ids"])
    check_tensor(f"wave L={L} B={B} N={N}", "hidden", hid, hid_ref, 2e-2)
    assert np.abs(logits - logits_ref).max() <= 2e-2 * np.abs(logits_ref).max()
    for l, (k, v) in enumerate(st.caches_numpy(N)):
        check_tensor(f"wave L={L} layer {l}", "k", k, caches_ref[l][0], 2e-2)
        check_tensor(f"wave L={L} layer {l}", "v", v, caches_ref[l][1], 2e-2)


@pytest.mark.parametrize("L,B,N", [(6, 2, 77), (2, 16, 130)])
def test_a_workspace_for_long_prompts_serves_short_ones(L, B, N):
    import torch
    from paper_2604_21215_b200 import inputs, rt
    d, H, dff, V = 512, 8, 1024, 91
    data = inputs.make_inputs(inputs.Workload("wave", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    stacks = []
    for longest in (N, 1500):
        st = rt.Stack(L, d, H, dff, V, dtype="bf16", residual_scale=1 / np.sqrt(L))
        st.set_weights(data["layers"], data["emb"])
        st.reserve(B, longest)
        ids = torch.as_tensor(data["ids"], dtype=torch.int32, device=st.device).contiguous()
        hid = torch.empty((B, N, d), dtype=torch.bfloat16, device=st.device)
        st.prefill_device(ids, hid, None)
        torch.cuda.synchronize()
        assert st.status() == rt.RT_OK
        stacks.append((hid, [k[:N] for k in st.k_caches]))
    assert torch.equal(stacks[0][0], stacks[1][0])
    assert all(torch.equal(a, b) for a, b in zip(stacks[0][1], stacks[1][1]))


# With less workspace than all layers side by side would use, fewer of them are (two at a time, in bands), or none; nothing is written behind what was given.  Beyond 1024
# positions every form gives the same bits.
@pytest.mark.parametrize("L,d,H,B,N", [(6, 512, 8, 2, 1090), (5, 768, 12, 9, 100), (3, 1024, 16, 20, 40)])
def test_a_stack_runs_in_less_workspace(L, d, H, B, N):
    import torch
    from paper_2604_21215_b200 import inputs, rt
    V, dff = 91, 4 * d
    data = inputs.make_inputs(inputs.Workload("less", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    st = rt.Stack(L, d, H, dff, V, dtype="bf16", residual_scale=1 / np.sqrt(L))
    st.set_weights(data["layers"], data["emb"])
    want, _ = st.prefill(data["ids"])
    caches = st.caches_numpy(N)
    if N < 1024 and B <= 16:                                    # the forms differ in rounding: each against the oracle
        from oracle import RTConfig, RTWeights, stack_prefill
        ref = stack_prefill(RTConfig(d, H, 64, dff, residual_scale=1 / np.sqrt(L)), [RTWeights(**lw) for lw in data["layers"]], data["emb"], None, data["ids"])[0]
    least, full = rt.rt_workspace_bytes(st.cfg, B, N, 1), rt.rt_workspace_bytes(st.cfg, B, N, L)
    ids = torch.as_tensor(data["ids"], dtype=torch.int32, device=st.device).contiguous()
    layer_bytes = 11 * d * d * 2
    for size in (least, least + 3 * layer_bytes, (least + full) // 2 + 100, full - 1):
        if size > full:
            continue
        ws = torch.full((size + 65536,), 0x5A, dtype=torch.uint8, device=st.device)
        st.ws = ws[:size]
        hid = torch.empty((B, N, d), dtype=torch.bfloat16, device=st.device)
        st.prefill_device(ids, hid, None)
        torch.cuda.synchronize()
        assert st.status() == rt.RT_OK and bool((ws[size:] == 0x5A).all())
        got = hid.to(torch.float64).cpu().numpy()
        if N > 1024 or B > 16:
            assert np.array_equal(got, want)
            assert all(np.array_equal(a, b) for p, q in zip(st.caches_numpy(N), caches) for a, b in zip(p, q))
        else:
            check_tensor(f"workspace of {size}", "hidden", got, ref, 2e-2)


def _leaf128(L, B, N):
    from paper_2604_21215_b200 import inputs
    d, H, dff, V = 512, 8, 1024, 91
    data = inputs.make_inputs(inputs.Workload("wave", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    return d, H, dff, V, data


def test_a_stack_of_generic_layers_keeps_their_arithmetic():
    # leaves of 128 positions do not fit the tensor-core leaf kernel: the layers take the generic kernel, whose vectors stay fp32, also in a stack
    import torch
    from paper_2604_21215_b200 import rt
    L, B, N = 3, 3, 150
    d, H, dff, V, data = _leaf128(L, B, N)
    kw = dict(dtype="bf16", leaf=128, residual_scale=1 / np.sqrt(L))
    st = rt.Stack(L, d, H, dff, V, **kw)
    st.set_weights(data["layers"], data["emb"])
    hid, _ = st.prefill(data["ids"])
    x = st.emb[torch.as_tensor(data["ids"], dtype=torch.long, device=st.device)].double().cpu().numpy()
    for l in range(L):
        layer = rt.Layer(d, H, dff, **kw)
        layer.set_weights(data["layers"][l])
        x, k, v = layer.prefill(x)
        got = st.caches_numpy(N)[l]
        assert np.array_equal(got[0], k) and np.array_equal(got[1], v)
    assert np.array_equal(hid, x)


def test_a_batch_on_the_generic_kernel_keeps_its_arithmetic():
    # the same layer with 20 sequences: as five batches of four, which are too few for the group kernel
    from paper_2604_21215_b200 import rt
    B, N = 20, 140
    d, H, dff, V, data = _leaf128(1, B, N)
    x = np.random.default_rng(3).standard_normal((B, N, d))
    outs = []
    for lo, hi in ((0, B), (0, 4), (4, 8), (8, 12), (12, 16), (16, 20)):
        layer = rt.Layer(d, H, dff, dtype="bf16", leaf=128)
        layer.set_weights(data["layers"][0])
        outs.append(layer.prefill(x[lo:hi]))
    for i in range(3):
        assert np.array_equal(outs[0][i], np.concatenate([o[i] for o in outs[1:]]))


def test_layers_may_share_one_pair_of_caches():
    # a program that wants hidden states and logits only gives every layer the same caches
    import ctypes as C
    from oracle import RTConfig, RTWeights, stack_prefill
    from paper_2604_21215_b200 import inputs, rt
    L, d, H, dff, B, N, V = 5, 512, 8, 1024, 2, 100, 91
    wl = inputs.Workload("wave", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L))
    data = inputs.make_inputs(wl, seed=6)
    hid_ref, logits_ref, caches_ref = stack_prefill(RTConfig(d, H, 64, dff, residual_scale=wl.residual_scale), [RTWeights(**w) for w in data["layers"]],
                                                    data["emb"], None, data["ids"])
    st = rt.Stack(L, d, H, dff, V, dtype="bf16", residual_scale=wl.residual_scale)
    st.set_weights(data["layers"], data["emb"])
    st.reserve(B, N)
    st._kp = (C.c_void_p * L)(*[st.k_caches[0].data_ptr()] * L)
    st._vp = (C.c_void_p * L)(*[st.v_caches[0].data_ptr()] * L)
    hid, logits = st.prefill(data["ids"])
    check_tensor("shared caches", "hidden", hid, hid_ref, 2e-2)
    assert np.abs(logits - logits_ref).max() <= 2e-2 * np.abs(logits_ref).max()
    k, v = st.caches_numpy(N)[0]                                # the last layer's pairs
    check_tensor("shared caches", "k", k, caches_ref[L - 1][0], 2e-2)
    check_tensor("shared caches", "v", v, caches_ref[L - 1][1], 2e-2)


@pytest.mark.parametrize("B", [20, 48, 64])
def test_one_position_takes_the_tensor_core_kernels(B):
    # a prefill of one position has no use for packed weights: slices of the leaf kernel or dense products, not the generic kernel, which
    # would read the chain weights once for all sequences
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    d, H, dff = 512, 8, 2048
    data = inputs.make_inputs(inputs.Workload("one", 1, B, 1, d, H, dff, "bf16"), seed=B)
    lw = data["layers"][0]
    ref = layer_seq(RTConfig(d, H, 64, dff), RTWeights(**lw), data["x"])
    layer = rt.Layer(d, H, dff, dtype="bf16")
    layer.set_weights(lw)
    for name, a, b in zip(("z", "k", "v"), layer.prefill(data["x"]), ref):
        check_tensor(f"one position B={B}", name, a, b, 2e-2)
    chain_w, pre_w = (3 * d * d + 2 * d * dff) * 2, 3 * d * d * 2
    per_token = (rt.rt_plan_counters(layer.cfg, 16, 1)["model_bytes_read"] - chain_w - pre_w) // 16
    assert rt.rt_plan_counters(layer.cfg, B, 1)["model_bytes_read"] - B * per_token - pre_w == chain_w * (1 if B > 48 else -(-B // 16))


# One after the other, the layers of a short prompt share arrays of c, h, z and g that are filled together: a launch takes fresh ones, and the last ones do
# not always suffice for the next layer (64 arrays; 30 + 30 positions and 4 left, 21 x 3 and 1 left; 64 + 6 with a leaf of its own in between).
@pytest.mark.parametrize("L,B,N", [(24, 1, 3), (3, 9, 30), (2, 4, 70), (5, 20, 1)])
def test_layers_one_after_the_other_give_the_bits_of_single_layers(L, B, N):
    import torch
    from paper_2604_21215_b200 import inputs, rt
    d, H, dff, V = 640, 10, 1280, 91
    data = inputs.make_inputs(inputs.Workload("chain", L, B, N, d, H, dff, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    kw = dict(dtype="bf16", leaf=64 if N == 70 else 0, residual_scale=1 / np.sqrt(L))
    st = rt.Stack(L, d, H, dff, V, **kw)
    st.set_weights(data["layers"], data["emb"])
    hid, _ = st.prefill(data["ids"])
    ids = torch.as_tensor(np.asarray(data["ids"]), dtype=torch.int64, device="cuda")
    x = st.emb[ids].contiguous()
    for lw in data["layers"]:
        layer = rt.Layer(d, H, dff, **kw)
        layer.set_weights(lw)
        layer.reserve(B, N)
        z = torch.empty_like(x)
        layer.prefill_device(x, z)
        torch.cuda.synchronize()
        x = z
    assert (x.float().cpu().numpy() == hid).all()


# ... and so do layers that fit the cluster kernel, whose values between the phases are fp32, wherever four of them side by side do not pay
@pytest.mark.parametrize("L,d,B,N", [(8, 128, 1, 77), (8, 128, 1, 200), (4, 256, 8, 48), (2, 384, 1, 200)])
def test_stacks_of_small_layers_give_the_bits_of_single_layers(L, d, B, N):
    import torch
    from paper_2604_21215_b200 import inputs, rt
    V = 91
    data = inputs.make_inputs(inputs.Workload("small", L, B, N, d, d // 64, 4 * d, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    kw = dict(dtype="bf16", residual_scale=1 / np.sqrt(L))
    st = rt.Stack(L, d, d // 64, 4 * d, V, **kw)
    st.set_weights(data["layers"], data["emb"])
    hid, _ = st.prefill(data["ids"])
    x = st.emb[torch.as_tensor(np.asarray(data["ids"]), dtype=torch.int64, device="cuda")].double().cpu().numpy()
    for i, lw in enumerate(data["layers"]):
        layer = rt.Layer(d, d // 64, 4 * d, **kw)
        layer.set_weights(lw)
        x, k, v = layer.prefill(x)
        got = st.caches_numpy(N)[i]
        assert np.array_equal(got[0], k) and np.array_equal(got[1], v), i
    assert np.array_equal(hid, x)


# Layers side by side take every sum in the order of the leaf kernel and their earlier pairs in the parts of Algorithm 1's tiles: a long stack is its layers
# one by one, to the bit.  Lengths that end inside a leaf, slopes in some layers only, six and eight places.
@pytest.mark.parametrize("L,d,H,B,N,gains", [(8, 512, 8, 2, 1100, True), (6, 768, 12, 9, 1050, False), (2, 1024, 16, 1, 1089, True), (17, 512, 8, 1, 1030, False)])
def test_long_stacks_give_the_bits_of_single_layers(L, d, H, B, N, gains):
    import torch
    from paper_2604_21215_b200 import inputs, rt
    V = 91
    data = inputs.make_inputs(inputs.Workload("long", L, B, N, d, H, 4 * d, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    if gains:
        for i, lw in enumerate(data["layers"]):
            _gains(lw, d, i)
    layers = [dict(lw, alibi_slopes=[2.0 ** (-8.0 * (h + 1) / H) for h in range(H)] if gains and i % 3 == 1 else None) for i, lw in enumerate(data["layers"])]
    kw = dict(dtype="bf16", residual_scale=1 / np.sqrt(L))
    cfg = rt.make_config(d, H, 4 * d, **kw)
    assert rt.rt_plan_counters(cfg, B, N, L)["kv_bytes_read"] != L * rt.rt_plan_counters(cfg, B, N, 1)["kv_bytes_read"]      # side by side
    st = rt.Stack(L, d, H, 4 * d, V, **kw)
    st.set_weights(layers, data["emb"])
    st.reserve(B, N)
    ids = torch.as_tensor(np.asarray(data["ids"]), dtype=torch.int32, device=st.device).contiguous()
    hid = torch.empty((B, N, d), dtype=torch.bfloat16, device=st.device)
    st.prefill_device(ids, hid, None)
    torch.cuda.synchronize()
    assert st.status() == rt.RT_OK
    x = st.emb[ids.long()].contiguous()
    for i, lw in enumerate(layers):
        layer = rt.Layer(d, H, 4 * d, **kw)
        layer.set_weights(lw)
        layer.reserve(B, N)
        z = torch.empty_like(x)
        layer.prefill_device(x, z)
        torch.cuda.synchronize()
        assert torch.equal(layer.k_cache, st.k_caches[i]) and torch.equal(layer.v_cache, st.v_caches[i]), i
        x = z
    assert torch.equal(x, hid)


# Up to 1024 positions, leaves that begin before position 192 meet all earlier pairs with fp32 probabilities, in stacks side by side and in those that are faster one after the
# other though four layers side by side would pay.  Distances set the probabilities here (scale 1e-5): 1 to 1 - 0.0028, most of them within half a bf16 step of 1, so
# that rounding them to bf16 would make every value of a query too large by up to 2e-3 of the pairs' share.  Layers that pass their input on, then one that gives 64
# times the value: the factor between its output and the exact one over 90 positions.  Rounded probabilities make that 6e-4.  The stored values' own roundings (8e-4 of
# each on average, of both signs; those of z and v, which all later positions share, count once for each of the 8 x 64 H columns) leave 1.41 x 8e-4 / sqrt(3584) =
# 1.9e-5, a few times that with what the recurrence carries on: bound 2e-4.
# In a workspace with room for one layer only they are kept too.
@pytest.mark.parametrize("L,H,side,least", [(8, 8, True, False), (8, 8, True, True), (2, 7, False, False)])
def test_probabilities_of_the_first_leaves_are_not_rounded(L, H, side, least):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    d, B, N, V = 64 * H, 8, 190, 91
    data = inputs.make_inputs(inputs.Workload("first", L, B, N, d, H, 4 * d, "bf16", vocab=V), seed=N)
    for i, lw in enumerate(data["layers"]):
        lw["w_down"] = np.zeros_like(lw["w_down"])
        lw["w_o"] = 64.0 * np.eye(d) * (i == L - 1)
    slopes = [1.5e-5] * H
    st = rt.Stack(L, d, H, 4 * d, V, dtype="bf16", softmax_scale=1e-5)
    assert side == (rt.rt_plan_counters(st.cfg, B, N, L)["kv_bytes_read"] != L * rt.rt_plan_counters(st.cfg, B, N, 1)["kv_bytes_read"])
    st.set_weights([dict(lw, alibi_slopes=slopes) for lw in data["layers"]], data["emb"])
    if least:
        import torch
        st.reserve(B, N)
        st.ws = st.ws[:rt.rt_workspace_bytes(st.cfg, B, N, 1)]
        out = torch.empty((B, N, d), dtype=torch.bfloat16, device=st.device)
        st.prefill_device(torch.as_tensor(data["ids"], dtype=torch.int32, device=st.device).contiguous(), out, None)
        torch.cuda.synchronize()
        assert st.status() == rt.RT_OK
        hid = out.double().cpu().numpy()
    else:
        hid, _ = st.prefill(data["ids"])
    x = np.asarray(data["emb"], dtype=np.float64)[np.asarray(data["ids"])]
    ref = layer_seq(RTConfig(d, H, 64, 4 * d, softmax_scale=1e-5, alibi_slopes=slopes), RTWeights(**data["layers"][L - 1]), x)[0]
    got, ref = hid[:, 100:], ref[:, 100:]
    factor = (got * ref).sum() / (ref * ref).sum() - 1
    assert abs(factor) <= 2e-4, factor


# The kernel of those tiles at the edges of its rows: one query, a rest of three and full leaves in the last leaf, few warps and many, slopes in some layers.
@pytest.mark.parametrize("L,d,H,B,N", [(8, 512, 8, 1, 65), (8, 512, 8, 16, 130), (4, 1024, 16, 9, 191), (2, 448, 7, 5, 187)])
def test_first_tiles_match_oracle(L, d, H, B, N):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    V = 91
    data = inputs.make_inputs(inputs.Workload("first", L, B, N, d, H, d, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    slopes = [[2.0 ** (-8.0 * (h + 1) / H) for h in range(H)] if i % 2 else None for i in range(L)]
    st = rt.Stack(L, d, H, d, V, dtype="bf16", residual_scale=1 / np.sqrt(L))
    st.set_weights([dict(lw, alibi_slopes=s) for lw, s in zip(data["layers"], slopes)], data["emb"])
    hid, _ = st.prefill(data["ids"])
    x = np.asarray(data["emb"], dtype=np.float64)[np.asarray(data["ids"])]
    for i, lw in enumerate(data["layers"]):
        x, k, v = layer_seq(RTConfig(d, H, 64, d, residual_scale=1 / np.sqrt(L), alibi_slopes=slopes[i]), RTWeights(**lw), x)
        got = st.caches_numpy(N)[i]
        check_tensor(f"first tiles layer {i}", "k", got[0], k, 2e-2)
        check_tensor(f"first tiles layer {i}", "v", got[1], v, 2e-2)
    check_tensor("first tiles", "hidden", hid, x, 2e-2)


# Distances alone (scale 0) set the weights: a layer whose second block meets the first through a tile, the parallel sweep, and layers side by side beyond position 192.
@pytest.mark.parametrize("L,N", [(1, 150), (8, 290)])
def test_distances_without_a_scale(L, N):
    from oracle import RTConfig, RTWeights, layer_seq
    from paper_2604_21215_b200 import inputs, rt
    d, H, B, V = 512, 8, 2, 91
    data = inputs.make_inputs(inputs.Workload("dist", L, B, N, d, H, d, "bf16", vocab=V, residual_scale=1 / np.sqrt(L)), seed=N)
    slopes = [2.0 ** -(h + 3) for h in range(H)]
    kw = dict(residual_scale=1 / np.sqrt(L), softmax_scale=0.0)
    st = rt.Stack(L, d, H, d, V, dtype="bf16", **kw)
    st.set_weights([dict(lw, alibi_slopes=slopes) for lw in data["layers"]], data["emb"])
    hid, _ = st.prefill(data["ids"])
    x = np.asarray(data["emb"], dtype=np.float64)[np.asarray(data["ids"])]
    for lw in data["layers"]:
        x0 = x
        x, k, v = layer_seq(RTConfig(d, H, 64, d, alibi_slopes=slopes, **kw), RTWeights(**lw), x)
    check_tensor("distances alone", "hidden", hid, x, 2e-2)
    if L == 1:
        layer = rt.Layer(d, H, d, dtype="bf16", **kw)
        layer.set_weights(dict(data["layers"][0], alibi_slopes=slopes))
        z, _, _ = layer.recompute(x0, x)
        check_tensor("distances alone", "sweep", z, x, 2e-2)
