"""The work that a program using this package has it do, as cases that can be timed and whose outputs can be compared.

Every case is one call of a public entry point of `paper_2604_21215_b200.rt` on device buffers, as a program that keeps
its weights, caches and workspace on the GPU issues it:

    prefill    Layer.prefill_device       x [B,N,d] -> z and the K/V caches of one layer
    stack      Stack.prefill_device       token ids -> last hidden states, logits of the last position, all K/V caches
    decode     rt_decode_step             one new token per sequence through a stack whose caches hold `pos` positions
    sweep      rt_layer_recompute         the parallel sweep over all positions, given the layer's outputs
    backward   Layer.backward_device      gradients of one layer given x, z and dL/dz

Layers have heads of 64 dimensions and an MLP of four times the width, as in the package's own workloads; weights are
N(0, 1/fan_in), inputs and embeddings N(0, 1), gains around one, ALiBi slopes the geometric sequence 2^(-8h/H).
"""
import math

import torch

from paper_2604_21215_b200 import rt

_WEIGHTS = ("w_q", "w_k", "w_v", "w_o", "w_up", "w_down")
_GAINS = ("g_attn", "g_mlp", "g_kv", "g_q", "g_k")
_VOCAB = 32000


def _case(op, dtype, B, N, heads, layers=1, gains=False, alibi=False, name=None):
    """N: positions of the call (decode: positions already in the caches)."""
    c = {"op": op, "dtype": dtype, "B": B, "N": N, "heads": heads, "layers": layers, "gains": gains, "alibi": alibi}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small layer in fp32: what someone checking the method, or a small experiment, runs
        _case("prefill", "f32", 1, 256, 2, name="prefill_f32_small"),
        # one user's short prompt through a whole model before the first answer token
        _case("stack", "bf16", 1, 77, 16, layers=8, gains=True, name="stack_short_prompt"),
        # one layer at the width of the 150M models, a few documents
        _case("prefill", "bf16", 4, 2048, 12, name="prefill_150m_width"),
        # one layer at the width of the 300M models, with trained gains and ALiBi distances, a length that fits no tile
        _case("prefill", "bf16", 7, 3001, 16, gains=True, alibi=True, name="prefill_300m_width_ragged"),
        # scoring or prompt processing of a full batch through a whole model: the largest case
        _case("stack", "bf16", 16, 2048, 16, layers=8, name="stack_full_batch"),
        # a batch between the small and the wide regime
        _case("prefill", "bf16", 40, 333, 12, gains=True, name="prefill_middle_batch"),
        # the forward pass of a training batch (the shape of the paper's latency table)
        _case("prefill", "bf16", 512, 512, 16, name="prefill_training_batch"),
        # generation for a full batch with ordinary contexts
        _case("decode", "bf16", 16, 1024, 16, layers=8, name="decode_full_batch"),
        # generation for one user with a long context
        _case("decode", "bf16", 1, 16001, 16, layers=8, gains=True, alibi=True, name="decode_one_long_context"),
        # rebuilding a layer's pairs and outputs from kept activations (activation checkpointing), or verifying them
        _case("sweep", "bf16", 8, 4096, 16, name="sweep_300m_width"),
        # the backward pass of a layer for a few long sequences
        _case("backward", "bf16", 4, 1500, 12, name="backward_small_batch"),
        # the backward pass of a layer for a training batch
        _case("backward", "bf16", 96, 256, 16, gains=True, name="backward_training_batch"),
    ]


def _spread(rng, lo, hi):
    """A whole number from [lo, hi], evenly spread over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    heads = rng.choice((2, 4, 6, 8, 10, 12, 12, 14, 16, 16))
    d = 64 * heads
    more = {"gains": rng.random() < 0.5, "alibi": rng.random() < 0.4}
    op = rng.choice(("prefill", "prefill", "prefill", "stack", "decode", "decode", "sweep", "backward", "backward"))
    if op == "prefill":
        kind = rng.choice(("f32", "few", "few", "middle", "wide"))
        if kind == "f32":
            return _case(op, "f32", _spread(rng, 1, 8), _spread(rng, 16, 600), rng.choice((2, 4)), **more)
        if kind == "few":
            return _case(op, "bf16", _spread(rng, 1, 16), _spread(rng, 48, 4096), heads, **more)
        if kind == "middle":
            return _case(op, "bf16", rng.randint(17, 64), _spread(rng, 48, 600), heads, **more)
        return _case(op, "bf16", _spread(rng, 65, 512), _spread(rng, 48, 512), heads, **more)
    if op == "stack":
        return _case(op, "bf16", _spread(rng, 1, 16), _spread(rng, 16, 1024), heads, layers=rng.choice((4, 6, 8)), **more)
    if op == "decode":
        N = _spread(rng, 64, 16384)
        most = min(48, max(1, 16 * 16384 * 1024 // (N * d)))            # the caches of the largest stay below 9 GB
        return _case(op, "bf16", _spread(rng, 1, most), N, heads, layers=rng.choice((4, 6, 8)), **more)
    if op == "sweep":
        N = _spread(rng, 128, 4096)
        return _case(op, "bf16", _spread(rng, 1, max(1, 32768 // N)), N, heads, **more)
    if rng.random() < 0.25:
        return _case(op, "f32", _spread(rng, 1, 8), _spread(rng, 16, 300), rng.choice((2, 4)), **more)
    if rng.random() < 0.6:
        return _case(op, "bf16", _spread(rng, 1, 16), _spread(rng, 48, 1500), heads, **more)
    return _case(op, "bf16", _spread(rng, 17, 128), _spread(rng, 48, 256), heads, **more)


def _layer_weights(c, gen, tdt, dev):
    d = 64 * c["heads"]
    f = 4 * d
    w = {}
    for n, (rows, cols) in zip(_WEIGHTS, ((d, d), (d, d), (d, d), (d, d), (f, d), (d, f))):
        w[n] = (torch.randn((rows, cols), generator=gen, device=dev) / math.sqrt(cols)).to(tdt)
    if c["gains"]:
        for n in _GAINS:
            w[n] = (1.0 + 0.1 * torch.randn((d,), generator=gen, device=dev)).to(tdt)
    if c["alibi"]:
        w["alibi_slopes"] = [2.0 ** (-8.0 * (h + 1) / c["heads"]) for h in range(c["heads"])]
    return w


def prepare(case, seed):
    c, dev = case, torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    tdt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    B, N, L, d = c["B"], c["N"], c["layers"], 64 * c["heads"]
    weights = [_layer_weights(c, gen, tdt, dev) for _ in range(L)]
    st = {"case": c}
    if c["op"] in ("stack", "decode"):
        m = rt.Stack(L, d, c["heads"], 4 * d, _VOCAB, dtype=c["dtype"], residual_scale=1.0 / math.sqrt(L))
        m.set_weights(weights, torch.randn((_VOCAB, d), generator=gen, device=dev).to(tdt),
                      (1.0 + 0.1 * torch.randn((d,), generator=gen, device=dev)).to(tdt) if c["gains"] else None)
        st["logits"] = torch.empty((B, _VOCAB), dtype=torch.float32, device=dev)
        if c["op"] == "stack":
            m.reserve(B, N)
            st["ids"] = torch.randint(0, _VOCAB, (B, N), generator=gen, device=dev, dtype=torch.int32)
            st["hidden"] = torch.empty((B, N, d), dtype=tdt, device=dev)
        else:
            # caches as a prefill leaves them: keys normalised per head, values of order one; room for the new row
            m.reserve(B, 1, N + 1)
            for k, v in zip(m.k_caches, m.v_caches):
                k.normal_(generator=gen)
                v.normal_(generator=gen)
            st["ids"] = torch.randint(0, _VOCAB, (B,), generator=gen, device=dev, dtype=torch.int32)
    else:
        m = rt.Layer(d, c["heads"], 4 * d, dtype=c["dtype"])
        m.set_weights(weights[0])
        m.reserve(B, N)
        st["x"] = torch.randn((B, N, d), generator=gen, device=dev).to(tdt)
        st["z"] = torch.empty_like(st["x"])
        if c["op"] in ("sweep", "backward"):
            # the layer's own outputs, kept from the forward pass
            m.prefill_device(st["x"], st["z"])
            m.k_cache.zero_()
            m.v_cache.zero_()
        if c["op"] == "sweep":
            st["z_out"] = torch.empty_like(st["x"])
            m.ws = torch.zeros(rt.rt_recompute_workspace_bytes(m.cfg, B, N), dtype=torch.uint8, device=dev)
        if c["op"] == "backward":
            st["dz"] = torch.randn((B, N, d), generator=gen, device=dev)
            st["dx"] = torch.empty_like(st["dz"])
            st["grads"], st["dw"] = rt.RtLayerGrads(), {}
            for n in _WEIGHTS + (_GAINS if c["gains"] else ()):
                st["dw"][n] = torch.empty(weights[0][n].shape, dtype=torch.float32, device=dev)
                setattr(st["grads"], n, st["dw"][n].data_ptr())
            m.ws = torch.zeros(rt.rt_backward_workspace_bytes(m.cfg, B, N), dtype=torch.uint8, device=dev)
    st["m"] = m
    return st


def run(state):
    c, m = state["case"], state["m"]
    if c["op"] == "prefill":
        m.prefill_device(state["x"], state["z"])
        return state["z"], m.k_cache, m.v_cache
    if c["op"] == "stack":
        m.prefill_device(state["ids"], state["hidden"], state["logits"])
        return state["hidden"], state["logits"], m.k_caches, m.v_caches
    stream = torch.cuda.current_stream(m.device).cuda_stream
    if c["op"] == "decode":
        N = c["N"]
        status = rt.rt_decode_step(m.cfg, m.n_layers, m.layers, m.emb.data_ptr(),
                                   None if m.g_final is None else m.g_final.data_ptr(), m.vocab, state["ids"].data_ptr(),
                                   c["B"], N, state["logits"].data_ptr(), m._kp, m._vp, m.N_max, m.ws.data_ptr(),
                                   m.ws.numel(), stream)
        if status != rt.RT_OK:
            raise rt.RtError(status, "rt_decode_step")
        return state["logits"], [k[N] for k in m.k_caches], [v[N] for v in m.v_caches]
    if c["op"] == "sweep":
        status = rt.rt_layer_recompute(m.cfg, m.w, state["x"].data_ptr(), state["z"].data_ptr(), c["B"], c["N"],
                                       state["z_out"].data_ptr(), m.k_cache.data_ptr(), m.v_cache.data_ptr(), m.N_max,
                                       m.ws.data_ptr(), m.ws.numel(), stream)
        if status != rt.RT_OK:
            raise rt.RtError(status, "rt_layer_recompute")
        return state["z_out"], m.k_cache, m.v_cache
    m.backward_device(state["x"], state["z"], state["dz"], state["dx"], state["grads"], m.ws)
    return state["dx"], state["dw"]


def work(case):
    c = case
    B, N, L, d = c["B"], c["N"], c["layers"], 64 * c["heads"]
    e = 2 if c["dtype"] == "bf16" else 4
    params = 4 * d * d + 2 * 4 * d * d                     # W_q, W_k, W_v, W_o, W_up, W_down
    # products per token: W_k and W_v serve the temporary and the persistent pair
    token_flops = 2 * (params + 2 * d * d)
    if c["op"] == "decode":
        nbytes = L * (params * e + 2 * B * N * d * e + 2 * B * d * e) + _VOCAB * d * e + B * d * e + B * _VOCAB * 4
        return {"bytes": nbytes, "flops": B * (L * (token_flops + 4 * (N + 1) * d) + 2 * _VOCAB * d)}
    rows = B * N
    attention = 4 * d * B * (N * (N + 1) // 2)
    if c["op"] == "prefill":
        return {"bytes": params * e + 4 * rows * d * e, "flops": rows * token_flops + attention}
    if c["op"] == "sweep":
        return {"bytes": params * e + 5 * rows * d * e, "flops": rows * token_flops + attention}
    if c["op"] == "stack":
        nbytes = L * (params * e + 2 * rows * d * e) + rows * (4 + 2 * d * e) + _VOCAB * d * e + B * _VOCAB * 4
        return {"bytes": nbytes, "flops": L * (rows * token_flops + attention) + 2 * B * _VOCAB * d}
    # backward: the intermediates once more, then two products for each of the forward pass
    nbytes = params * (e + 4) + rows * d * (2 * e + 2 * 4)
    return {"bytes": nbytes, "flops": 3 * (rows * token_flops + attention)}


def tolerance(case):
    # storage in bf16 with fp32 sums: 2^-8 for each rounding of a stored value, a few of them in a row for each output;
    # the layers of a stack add theirs up.  fp32: the order of the sums, carried on by the recurrence.
    if case["dtype"] == "f32":
        return {"rel": 1e-5}
    return {"rel": 2e-2 if case["layers"] > 1 else 1e-2}
