"""What captured calls show of their launches: orders and kernels.

Weights that a call reads before it waits for the kernel ahead of it are complete when it starts.

The caller's weights are read in place at every call.  A kernel launched with programmatic stream
serialization may start while the kernel before it is still running, so the first kernel of a call that
reads weights ahead of its wait has to be launched in stream order.  Captured into a graph, the two kinds
of launch give edges of different types, which shows the order without running anything.

The nodes of the graph show which kernels a call of a given size runs on.
"""
import ctypes
import dataclasses

import pytest
import torch

from paper_2505_18719_gb300 import inputs as I
from paper_2505_18719_gb300 import vla as V
from tests import parity as P

pytestmark = pytest.mark.gpu
WL = I.WORKLOADS["tiny_b4"]
RELAXED = 2
FULL, PROGRAMMATIC = 0, 1
GEMMS = ("gemm_tc_kernel", "gemm_tc2_kernel", "gemm_wide_kernel", "gemv_cluster_kernel", "gemv_stream_kernel")


class EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte),
                ("reserved", ctypes.c_ubyte * 5)]


class KernelNode(ctypes.Structure):
    _fields_ = [("func", ctypes.c_void_p)] + [(n, ctypes.c_uint) for n in ("gx", "gy", "gz", "bx", "by", "bz", "smem")] + \
               [(n, ctypes.c_void_p) for n in ("params", "extra", "kern", "ctx")]


def _capture(cu, stream, calls):
    assert all(c() in (0, None) for c in calls)  # every kernel is loaded before the capture
    stream.synchronize()
    graph = ctypes.c_void_p()
    st = ctypes.c_void_p(stream.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(st, RELAXED) == 0
    rcs = [c() for c in calls]
    assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) == 0
    assert all(rc in (0, None) for rc in rcs), rcs
    return graph


def _kernel_names(stream, calls):
    """The (mangled) names of the kernels that the calls launch."""
    cu = ctypes.CDLL("libcuda.so.1")
    graph = _capture(cu, stream, calls)
    n = ctypes.c_size_t(0)
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    names = []
    for node in nodes:
        kind, p, name = ctypes.c_int(-1), KernelNode(), ctypes.c_char_p()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value != 0:  # not a kernel
            continue
        assert cu.cuGraphKernelNodeGetParams_v2(ctypes.c_void_p(node), ctypes.byref(p)) == 0
        rc = (cu.cuFuncGetName(ctypes.byref(name), ctypes.c_void_p(p.func)) if p.func
              else cu.cuKernelGetName(ctypes.byref(name), ctypes.c_void_p(p.kern)))
        assert rc == 0
        names.append(name.value.decode())
    assert cu.cuGraphDestroy(graph) == 0
    return names


def _edge_types(stream, calls):
    """The edge types of a captured chain of calls, in the order of the chain."""
    cu = ctypes.CDLL("libcuda.so.1")
    graph = _capture(cu, stream, calls)
    n = ctypes.c_size_t(0)
    assert cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)) == 0
    src, dst, data = (ctypes.c_void_p * n.value)(), (ctypes.c_void_p * n.value)(), (EdgeData * n.value)()
    assert cu.cuGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(n)) == 0
    nxt = {src[i]: (dst[i], data[i].type) for i in range(n.value)}
    at = (set(nxt) - {d for d, _ in nxt.values()}).pop()
    types = []
    while at in nxt:
        at, t = nxt[at]
        types.append(t)
    assert cu.cuGraphDestroy(graph) == 0
    return types


@pytest.fixture(scope="module")
def bufs():
    from paper_2505_18719_gb300 import build
    build.build()
    V.load()
    f = lambda *s: torch.zeros(*s, device="cuda")  # noqa: E731
    b = lambda *s: torch.zeros(*s, dtype=torch.bfloat16, device="cuda")  # noqa: E731
    return {"x": f(64, 256), "z": f(64, 256), "v": f(64), "act": f(64), "w": b(512, 256), "a": b(64, 256), "lo": b(64, 256),
            "gain": b(256), "ws": f(1 << 20), "bins": torch.zeros(64, dtype=torch.int32, device="cuda"),
            "status": torch.zeros(1, dtype=torch.int32, device="cuda")}


def _ahead(t, stream):
    # a kernel that lets its dependents start early
    return lambda: V.vla_op_rmsnorm(t["x"].data_ptr(), 256, 64, 256, t["gain"].data_ptr(), 1e-6, t["a"].data_ptr(),
                                    t["lo"].data_ptr(), False, stream.cuda_stream)


def test_a_launch_that_waits_first_may_start_early(bufs):
    s = torch.cuda.Stream()
    assert _edge_types(s, [_ahead(bufs, s), _ahead(bufs, s)]) == [PROGRAMMATIC]


def test_action_head_op_starts_in_stream_order(bufs):
    t, s = bufs, torch.cuda.Stream()
    head = lambda: V.vla_op_action_head(t["x"].data_ptr(), 256, 64, 256, t["gain"].data_ptr(),  # noqa: E731
                                        t["w"].data_ptr(), 1e-6, 0, 0.0, 0, t["bins"].data_ptr(), t["v"].data_ptr(),
                                        t["act"].data_ptr(), t["z"].data_ptr(), t["status"].data_ptr(), s.cuda_stream)
    assert _edge_types(s, [_ahead(t, s), head]) == [FULL]


@pytest.mark.parametrize("M", [16, 64])
def test_decode_gemm_ops_start_in_stream_order(bufs, M):
    t, s = bufs, torch.cuda.Stream()
    c = torch.zeros(M, 512, device="cuda")
    for op in (V.vla_op_gemm_decode_bf16, V.vla_op_gemm_decode_f16):
        gemm = lambda: op(t["a"].data_ptr(), t["lo"].data_ptr(), 256, t["w"].data_ptr(), 256, c.data_ptr(), 512,  # noqa: E731
                          M, 512, 256, t["ws"].data_ptr(), 4 << 20, s.cuda_stream)
        assert _edge_types(s, [_ahead(t, s), gemm])[0] == FULL


def test_one_token_decode_and_score_start_in_stream_order(bufs):
    # a handle of one action token uploads nothing in decode and score: the head is their first kernel
    sh = dataclasses.replace(WL.shape, action_dim=1)
    s = torch.cuda.Stream()
    pol = V.Policy(sh, P.weights_to_device(I.make_weights(sh, 3)), 2, 64, 64, stream=s)
    ids = torch.zeros(2, 4, dtype=torch.int32, device="cuda")
    u = torch.full((2, 1, 256), 0.5, device="cuda")
    tok = torch.full((2, 1), sh.vocab - 1, dtype=torch.int32, device="cuda")
    i32, f32 = torch.zeros(2, 1, dtype=torch.int32, device="cuda"), [torch.zeros(2, 1, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    pol.prefill(None, ids, [4, 3])
    pol.sync()
    decode = lambda: V.vla_decode_actions(pol.h, u.data_ptr(), 1.0, 0, i32.data_ptr(), f32[0].data_ptr(),  # noqa: E731
                                          f32[1].data_ptr(), 0)
    score = lambda: V.vla_score_actions(pol.h, tok.data_ptr(), 1.0, f32[0].data_ptr())  # noqa: E731
    assert _edge_types(s, [_ahead(bufs, s), decode]) == [FULL]
    assert _edge_types(s, [_ahead(bufs, s), score]) == [FULL]
    pol.close()


@pytest.mark.parametrize("action_dim", [1, 7])
def test_gains_embeddings_and_lm_head_are_read_at_every_call(action_dim):
    # changed in place on the stream between calls, without a synchronisation: the results are those of a
    # handle made after the change, bit for bit
    sh = dataclasses.replace(WL.shape, action_dim=action_dim)
    w = P.weights_to_device(I.make_weights(sh, 3))
    ids = I.randint_i32((2, 9), 5, 6, 0, sh.vocab - 257).cuda()
    u = I.uniform_f32((2, action_dim, 256), 5, 7).cuda()
    tok = I.randint_i32((2, action_dim), 5, 8, sh.vocab - 256, sh.vocab - 1).cuda()

    def turn(pol, between=lambda: None):
        pol.reset()
        pol.prefill(None, ids, [9, 6])
        between()
        d = pol.decode(u, 1.0, forced=tok)
        between()
        return [d["logits"], pol.score(tok, 1.0)["logits"]]

    pol = V.Policy(sh, w, 2, 64, 64)
    before = turn(pol)
    torch.cuda._sleep(1_000_000)  # keeps the stream busy while the host queues the rest
    for name in ("embed", "attn_norm", "ffn_norm", "final_norm"):
        w[name].mul_(1.25)
    w["lm_head"].neg_()
    after = turn(pol)
    w["lm_head"].neg_()
    # the head alone changed between a prefill and its decode, and back before the score
    mixed = turn(pol, between=lambda: w["lm_head"].neg_())
    pol.sync()
    want = []
    for _ in range(2):  # as it was for the score of `mixed`, then as it was for its decode and for `after`
        fresh = V.Policy(sh, w, 2, 64, 64)
        want.append(turn(fresh))
        fresh.sync()
        fresh.close()
        w["lm_head"].neg_()
    assert all(torch.equal(a, b) for a, b in zip(after, want[1]))
    assert not any(torch.equal(a, b) for a, b in zip(after, before))
    assert torch.equal(mixed[0], want[1][0]) and torch.equal(mixed[1], want[0][1])
    pol.close()


@pytest.mark.parametrize("B", [42, 43, 72, 73])
def test_score_pass_runs_o_and_down_on_the_wide_gemm(B):
    # 258 to 432 score rows; 252 and 438 stay on the tile GEMMs
    sh = I.ModelShape("tiny", 2, 4096, 32, 128, 4616)
    s = torch.cuda.Stream()
    pol = V.Policy(sh, P.weights_to_device(I.make_weights(sh, 11)), B, 32, B * 2, stream=s)
    ids = torch.zeros(B, 2, dtype=torch.int32, device="cuda")
    tok = torch.full((B, sh.action_dim), sh.vocab - 1, dtype=torch.int32, device="cuda")
    lp = torch.zeros(B, sh.action_dim, device="cuda")
    torch.cuda.synchronize()
    pol.prefill(None, ids, [2] * B)
    names = _kernel_names(s, [lambda: V.vla_score_actions(pol.h, tok.data_ptr(), 1.0, lp.data_ptr())])
    gemms = [k for n in names for k in GEMMS if k in n]  # q|k|v, o, gate|up, down of each layer
    o_down = "gemm_wide_kernel" if 43 <= B <= 72 else "gemm_tc_kernel"
    assert gemms == ["gemm_tc_kernel", o_down] * (2 * sh.n_layers)
    pol.close()


@pytest.mark.parametrize("B,kernel", [(1, "gemv_cluster_kernel"), (32, "gemv_cluster_kernel"), (33, "gemv_stream_kernel"),
                                      (128, "gemv_stream_kernel"), (129, "gemm_tc_kernel")])
def test_decode_projections_kernel_by_rows(B, kernel):
    s = torch.cuda.Stream()
    pol = V.Policy(WL.shape, P.weights_to_device(I.make_weights(WL.shape, 3)), B, 32, B * 2, stream=s)
    ids = torch.zeros(B, 2, dtype=torch.int32, device="cuda")
    u = torch.full((B, WL.shape.action_dim, 256), 0.5, device="cuda")
    i32 = torch.zeros(B, WL.shape.action_dim, dtype=torch.int32, device="cuda")
    f32 = [torch.zeros(B, WL.shape.action_dim, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    pol.prefill(None, ids, [2] * B)
    names = _kernel_names(s, [lambda: V.vla_decode_actions(pol.h, u.data_ptr(), 1.0, 0, i32.data_ptr(),
                                                           f32[0].data_ptr(), f32[1].data_ptr(), 0)])
    gemms = [k for n in names for k in GEMMS if k in n]
    assert gemms == [kernel] * (6 * 4 * WL.shape.n_layers)
    pol.close()


def test_decode_of_many_envs_over_short_contexts():
    # 120 envs x 8 heads, and a model larger than L2: decode attention on the kernel for many pairs.  The logits are those of a small batch, on the other kernel: both run on
    # operand pairs (2^-21) through 24 layers
    sh = I.ModelShape("tiny", 24, 512, 8, 64, 1368)
    B, n = 120, 8
    w = P.weights_to_device(I.make_weights(sh, 3))
    ids = I.randint_i32((B, 1), 5, 6, 0, sh.vocab - 257).cuda()
    u = I.uniform_f32((B, sh.action_dim, 256), 5, 7).cuda()
    tok = I.randint_i32((B, sh.action_dim), 5, 8, sh.vocab - 256, sh.vocab - 1).cuda()
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    z, names = [], []
    for envs in (B, n):
        pol = V.Policy(sh, w, envs, 160, 1024, stream=s)
        with torch.cuda.stream(s):
            pol.prefill(None, ids, [1] * envs)
            out = pol.decode(u, 1.0, forced=tok)
            pol.sync()
            z.append(out["logits"][:n].double())
            names.append(_kernel_names(s, [lambda: V.vla_decode_actions(
                pol.h, u.data_ptr(), 1.0, tok.data_ptr(), out["tokens"].data_ptr(), out["logprobs"].data_ptr(),
                out["actions"].data_ptr(), 0)]))
        pol.close()
    assert ((z[0] - z[1]).norm() / z[1].norm()).item() < 1e-4
    short = [sum("attn_decode_short_kernel" in x for x in k) for k in names]
    assert short == [6 * sh.n_layers, 0]
    assert [sum("attn_decode" in x for x in k) for k in names] == [6 * sh.n_layers] * 2


@pytest.mark.parametrize("hd,per_sm,over,ctx,short", [
    (64, 4, 1, 112, True), (64, 4, 0, 112, False), (64, 4, 1, 113, False), (64, 5, 1, 160, True), (64, 5, 1, 161, False),
    (128, 7, 1, 128, True), (128, 7, 0, 128, False), (128, 7, 1, 129, False), (128, 24, 1, 192, True),
    (128, 24, 1, 193, False)])
def test_decode_attention_kernel_by_pairs_and_positions(hd, per_sm, over, ctx, short):
    H, s = 8, torch.cuda.Stream()
    B = (per_sm * V.vla_op_num_sms() + H - 1) // H + over
    cap = (ctx + 15) // 16 * 16
    q = torch.zeros(B, H, hd, device="cuda")
    kv = torch.zeros(1, 2, H, cap, hd, dtype=torch.float16, device="cuda")
    env, pos = (torch.full((B,), v, dtype=torch.int32, device="cuda") for v in (0, ctx - 1))
    out = torch.zeros(2, B, H * hd, dtype=torch.bfloat16, device="cuda")
    nbytes = V.vla_op_attn_decode_workspace_bytes(B, H, hd, ctx)
    ws = torch.zeros(nbytes // 4 + 1, device="cuda")
    torch.cuda.synchronize()
    names = _kernel_names(s, [lambda: V.vla_op_attn_decode(
        q.data_ptr(), kv.data_ptr(), 1, H, hd, cap, env.data_ptr(), pos.data_ptr(), B, ctx, out[0].data_ptr(),
        out[1].data_ptr(), ws.data_ptr(), nbytes, s.cuda_stream)])
    names = [n for n in names if "attn_decode" in n]
    assert len(names) == 1 and ("attn_decode_short_kernel" in names[0]) == short, names
