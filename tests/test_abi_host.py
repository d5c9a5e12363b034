"""Host-side checks that need no GPU: the library loads, exports what include/rt.h declares,
rejects bad arguments before touching the device, and its schedule enumerator agrees with
Algorithm 1 as written out by the oracle."""
import ctypes as C
import os
import re

import pytest

from oracle import alg1_tiles
from paper_2604_21215_b200 import rt

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_library_exports_every_declared_symbol():
    header = open(os.path.join(ROOT, "include", "rt.h")).read()
    declared = set(re.findall(r"\b(rt_[a-z_]+)\s*\(", header))
    assert declared, "no declarations found"
    lib = C.CDLL(rt.LIB_PATH)
    for name in declared:
        assert hasattr(lib, name), name
    assert declared == set(rt.EXPORTS)


def test_status_strings():
    assert rt.rt_status_string(rt.RT_OK) == "ok"
    assert "timed out" in rt.rt_status_string(rt.RT_ERR_TIMEOUT)


@pytest.mark.parametrize("leaf", [1, 2, 16, 64])
def test_plan_tiles_is_algorithm_1_at_block_granularity(leaf):
    for N in (1, 2, 7, 8, 64, 65, 100, 256, 1000):
        want = [(u - 1, v, s - 1, e) for (t, u, v, s, e) in alg1_tiles(N, leaf)]   # 1-based inclusive -> 0-based half-open
        assert rt.rt_plan_tiles(N, leaf) == want, (N, leaf)


def test_worked_examples_from_the_paper_through_the_library():
    tiles = {k1: (q0, q1, k0) for (q0, q1, k0, k1) in rt.rt_plan_tiles(8, 1)}
    assert tiles[4] == (4, 8, 0)      # after position 4: pairs 1..4 -> queries 5..8
    assert tiles[6] == (6, 8, 4)      # after position 6: pairs 5..6 -> queries 7..8


def test_invalid_arguments_are_rejected_on_the_host():
    cfg = rt.make_config(128, 2, 512, dtype="f32")
    w = rt.RtLayerWeights()
    # null pointers everywhere: must return before any CUDA call
    assert rt.rt_layer_prefill(cfg, w, None, 1, 16, None, None, None, 16, None, 0, None) == rt.RT_ERR_INVALID_ARG
    bad = rt.make_config(128, 3, 512, dtype="f32")           # heads * head_dim != d_model
    assert rt.rt_workspace_bytes(bad, 1, 16) == 0
    assert rt.rt_workspace_bytes(cfg, 0, 16) == 0
    cfg32 = rt.make_config(128, 4, 512, dtype="f32", head_dim=32)
    buf = (C.c_char * 4096)()
    addr = (C.addressof(buf) + 255) & ~255
    assert rt.rt_layer_prefill(cfg32, w, addr, 1, 16, addr, addr, addr, 16, addr, 1 << 40, None) == rt.RT_ERR_UNSUPPORTED
    need = rt.rt_workspace_bytes(cfg, 1, 16)
    assert need > 0
    assert rt.rt_layer_prefill(cfg, w, addr, 1, 16, addr, addr, addr, 16, addr, need - 1, None) == rt.RT_ERR_WORKSPACE
    leafbad = rt.make_config(128, 2, 512, dtype="f32", leaf=48)
    assert rt.rt_workspace_bytes(leafbad, 1, 16) == 0


def test_backward_host_checks_need_no_gpu():
    # workspace size and argument checks of the backward pass run on the host, before any CUDA call
    cfg = rt.make_config(128, 2, 512, dtype="f32")
    need = rt.rt_backward_workspace_bytes(cfg, 2, 64)
    assert need > 0 and rt.rt_backward_workspace_bytes(cfg, 4, 64) > need
    assert rt.rt_backward_workspace_bytes(rt.make_config(128, 3, 512, dtype="f32"), 2, 64) == 0
    assert rt.rt_backward_workspace_bytes(cfg, 0, 64) == 0
    w, gr = rt.RtLayerWeights(), rt.RtLayerGrads()
    assert rt.rt_layer_backward(cfg, w, None, None, None, 2, 64, None, gr, None, 0, None) == rt.RT_ERR_INVALID_ARG
    buf = (C.c_char * 4096)()
    addr = (C.addressof(buf) + 255) & ~255
    for n in ("w_q", "w_k", "w_v", "w_o", "w_up", "w_down"):
        setattr(w, n, addr)
    call = lambda c, nbytes, g=gr: rt.rt_layer_backward(c, w, addr, addr, addr, 2, 64, addr, g, addr, nbytes, None)
    assert call(cfg, need - 1) == rt.RT_ERR_WORKSPACE
    assert call(rt.make_config(128, 2, 512, dtype="f32", recur_block=8), need) == rt.RT_ERR_UNSUPPORTED
    assert call(rt.make_config(128, 4, 512, dtype="f32", head_dim=32), need) == rt.RT_ERR_UNSUPPORTED
    odd = rt.RtLayerGrads()
    odd.w_q = addr + 4                                        # gradient arrays must be 16-byte aligned
    assert call(cfg, need, odd) == rt.RT_ERR_INVALID_ARG


def test_plan_counters_follow_the_n_log_n_model():
    # K/V rows streamed by the cross tiles: one half of the rows per level above the leaf.
    cfg = rt.make_config(1024, 16, 4096, dtype="bf16", leaf=64)
    B, d, e = 1, 1024, 2
    for N in (1024, 4096, 32768):
        c = rt.rt_plan_counters(cfg, B, N)
        levels = (N // 64).bit_length() - 1
        assert c["kv_bytes_read"] == levels * (N // 2) * 2 * B * d * e
        assert c["n_leaves"] == N // 64 and c["n_tiles"] == N // 64 - 1
        assert c["flops_tile"] == sum(4 * (q1 - q0) * (k1 - k0) * d * B for (q0, q1, k0, k1) in rt.rt_plan_tiles(N, 64))
    naive = rt.make_config(1024, 16, 4096, dtype="bf16", sched="naive")
    c = rt.rt_plan_counters(naive, B, 4096)
    assert c["kv_bytes_read"] == B * d * e * 4096 * 4095


def test_plan_counters_model_the_schedule_that_runs():
    # The counters follow the chain form a shape takes: wide batches use leaves of 16 positions, the tensor-core
    # leaf kernel keeps 64-position leaves also when an SM owns two (sequence, head) pairs, blocked recurrence tiles by blocks.
    N = 2048
    wide = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16"), 96, N)
    assert wide["n_leaves"] == N // 16 and wide["n_tiles"] == len(rt.rt_plan_tiles(N, 16))
    # 17 .. 48 sequences run as slices of at most 16 through the tensor-core leaf kernel: its leaves, and the chain
    # weights staged once per slice and leaf
    split = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16"), 32, N)
    assert split["n_leaves"] == N // 64 and split["n_tiles"] == len(rt.rt_plan_tiles(N, 64))
    one = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16"), 16, N)
    chain_w = (3 * 1024 * 1024 + 2 * 1024 * 4096) * 2
    assert split["model_bytes_read"] - 2 * one["model_bytes_read"] == -(3 * 1024 * 1024 * 2)    # the pre-pass weights once, not twice
    assert one["model_bytes_read"] > (N // 64) * chain_w
    c3 = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16"), 8, N)
    assert c3["n_leaves"] == N // 64 and c3["n_tiles"] == len(rt.rt_plan_tiles(N, 64))
    c4 = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16"), 16, N)
    assert c4["n_leaves"] == N // 64 and c4["n_tiles"] == len(rt.rt_plan_tiles(N, 64))
    blk = rt.rt_plan_counters(rt.make_config(1024, 16, 4096, dtype="bf16", recur_block=128), 8, N)
    assert blk["n_leaves"] == N // 128 and blk["n_tiles"] == N // 128 - 1
    f32 = rt.rt_plan_counters(rt.make_config(128, 2, 512, dtype="f32"), 4, 256)
    assert f32["n_leaves"] == 4 and f32["n_tiles"] == 3


def test_unknown_flags_are_invalid_configurations():
    assert rt.rt_workspace_bytes(rt.make_config(128, 2, 512, dtype="f32", norm_flags=4 | 3), 1, 16) == 0
    assert rt.rt_workspace_bytes(rt.make_config(128, 2, 512, dtype="f32", flags=2), 1, 16) == 0
    assert rt.rt_workspace_bytes(rt.make_config(128, 2, 512, dtype="f32", flags=rt.RT_FLAG_BACKWARD_STEP_LAUNCHES), 1, 16) > 0


def test_decode_workspace_covers_every_slice_of_the_batch():
    # A bf16 decode step above 16 sequences runs as slices one after the other in one exchange area.  A smaller last slice can need
    # more of it than the fuller ones: each pair's attention is then split over more CTAs.  So a batch asks for no less than any of its
    # slices would alone, at any depth (16 layers share a launch: the exchange area is most of that workspace).
    for H in range(1, 17):
        cfg = rt.make_config(64 * H, H, 256 * H, dtype="bf16")
        for L in (1, 8, 16):
            alone = [rt.rt_workspace_bytes(cfg, b, 1, L) for b in range(1, 17)]
            for B in range(17, 65):
                assert rt.rt_workspace_bytes(cfg, B, 1, L) >= max(alone), (H, B, L)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_workspace_grows_with_the_shape(dtype):
    # a workspace reserved for the longest prompt, the fullest batch and the deepest stack serves every smaller call
    Bs = [1, 2, 5, 8, 9, 15, 16, 17, 23, 32, 33, 48, 49, 64, 65, 200]
    Ns = [1, 2, 16, 17, 64, 128, 129, 1000, 1024, 1025, 4096]
    Ls = [1, 2, 3, 4, 8, 24]
    for d, dff, kw in ((64, 256, {}), (128, 512, {"leaf": 16}), (384, 1536, {}), (768, 3072, {"leaf": 128}), (1024, 4096, {}),
                       (1024, 4096, {"sched": "naive"}), (1024, 8192, {}), (2048, 8192, {})):
        cfg = rt.make_config(d, d // 64, dff, dtype=dtype, **kw)
        ws = {(B, N, L): rt.rt_workspace_bytes(cfg, B, N, L) for B in Bs for N in Ns for L in Ls}
        for (B, N, L), have in ws.items():
            for axis, values in enumerate((Bs, Ns, Ls)):
                at = [B, N, L]
                i = values.index(at[axis])
                if i:
                    at[axis] = values[i - 1]
                    assert ws[tuple(at)] <= have, (d, dff, kw, tuple(at), (B, N, L))
        for size in (rt.rt_recompute_workspace_bytes, rt.rt_backward_workspace_bytes):
            ws = [[size(cfg, B, N) for N in Ns] for B in Bs]
            assert all(a <= b for row in ws for a, b in zip(row, row[1:])), (size, d, dff, kw)
            assert all(a <= b for r0, r1 in zip(ws, ws[1:]) for a, b in zip(r0, r1)), (size, d, dff, kw)


def test_layers_run_side_by_side_where_enough_of_them_are_at_work():
    # Side by side every leaf meets all earlier pairs at once, one after the other Algorithm 1's tiles do: the counters tell which.  A prompt
    # of one leaf has one layer at work at a time; deep stacks of longer prompts have all places busy; two layers never more than two.
    def side_by_side(d, B, N, L):
        cfg = rt.make_config(d, d // 64, 4 * d, dtype="bf16")
        return rt.rt_plan_counters(cfg, B, N, L)["kv_bytes_read"] != L * rt.rt_plan_counters(cfg, B, N, 1)["kv_bytes_read"]
    for d in (128, 256, 384, 512, 768, 1024):
        for B in (1, 4, 8, 9, 16):
            assert not any(side_by_side(d, B, 16, L) for L in (2, 4, 8)), (d, B)
    for d in (512, 768, 1024):
        for B in (1, 4, 16):
            assert side_by_side(d, B, 77, 8) and side_by_side(d, B, 128, 4) and side_by_side(d, B, 1024, 8), (d, B)
            assert not side_by_side(d, B, 24, 8) and not side_by_side(d, B, 32, 2), (d, B)
    assert not side_by_side(128, 1, 64, 8) and side_by_side(384, 4, 64, 8) and side_by_side(256, 16, 200, 8)
    # layers of the cluster kernel, which holds their values between the phases in fp32, are not taken off it because more than four fit side by side
    for d, B, N, L in ((64, 4, 400, 4), (128, 1, 77, 8), (128, 1, 200, 8), (128, 8, 256, 3), (256, 1, 256, 3), (256, 8, 48, 4), (384, 1, 200, 2), (192, 1, 200, 4)):
        assert not side_by_side(d, B, N, L), (d, B, N, L)
    # the others where it was measured to be faster: widths that are no multiple of 128 pay for a pre-pass per launch, wide layers of nine and more sequences gain most;
    # a leaf reads its layer's whole cache so far, so the longest prompts go one after the other (crossing measured between 16 and 32 thousand positions for two
    # layers, 33 and 65 thousand for eight, d = 1024, B = 16)
    for d, B, N, L in ((448, 1, 64, 2), (448, 4, 48, 3), (960, 4, 64, 2), (960, 1, 200, 2), (960, 4, 129, 3), (768, 1, 48, 2), (1024, 16, 32768, 2), (1024, 16, 131072, 8), (1024, 1, 400000, 8)):
        assert not side_by_side(d, B, N, L), (d, B, N, L)
    for d, B, N, L in ((1024, 16, 64, 4), (1024, 9, 129, 4), (512, 1, 77, 8), (448, 9, 200, 4), (1024, 16, 16384, 2), (1024, 16, 32768, 8), (512, 16, 32768, 8), (1024, 1, 65536, 8)):
        assert side_by_side(d, B, N, L), (d, B, N, L)


def test_a_stack_prefill_is_refused_only_below_the_workspace_of_one_layer():
    # what it has beyond that holds weights of layers side by side: the first figure is a size that once sufficed.  (Refused later on, for the missing layers.)
    buf = (C.c_char * 4096)()
    addr = (C.addressof(buf) + 255) & ~255
    for d, B, N, L, given in ((1024, 1, 77, 8, 106650880), (768, 4, 512, 8, 90797312), (1024, 16, 2048, 8, None), (128, 2, 300, 4, None), (512, 40, 100, 3, None)):
        cfg = rt.make_config(d, d // 64, 4 * d, dtype="bf16")
        least = rt.rt_workspace_bytes(cfg, B, N, 1)
        def call(size):
            return rt.rt_stack_prefill(cfg, L, None, addr, None, 10, addr, B, N, None, None, None, None, N, addr, size, None)
        assert least <= rt.rt_workspace_bytes(cfg, B, N, L)
        assert call(least - 1) == rt.RT_ERR_WORKSPACE and call(least) == rt.RT_ERR_INVALID_ARG
        assert given is None or call(given) == rt.RT_ERR_INVALID_ARG
