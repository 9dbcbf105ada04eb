"""Edge cases of the rollout path through the C ABI, each against the fp64 oracle on the tiny
model (Algorithm 1's rollout: prefill of the state, then the 7 action tokens):
  * a prefill without visual rows and with ragged text down to a single row per env (a
    prefill this small, 31 rows, runs on the weight-streaming GEMMs);
  * a context that fills the KV cache exactly (chunk + 6 decoded positions == capacity), and
    the same chunk one position short refused;
  * forced tokens at the two edge bins (ids vocab-256 and vocab-1: the last embedding row)."""
import numpy as np
import pytest
import torch

import oracle.vla_oracle as O
from paper_2505_18719_gb300 import inputs as I
from paper_2505_18719_gb300 import vla as V
from tests import parity as P

pytestmark = pytest.mark.gpu
WL = I.WORKLOADS["tiny_b4"]
SH = WL.shape
BASE = SH.vocab - SH.n_bins


@pytest.fixture(scope="module")
def weights():
    from paper_2505_18719_gb300 import build
    build.build()
    w = I.make_weights(SH, WL.weight_seed)
    return w, P.weights_to_device(w)


def _rollout(weights, visual, ids, lengths, cap, forced=None, T=1.0):
    """Prefill + decode on the GPU and in the oracle; the GPU is teacher-forced on the oracle's
    tokens (or on `forced` for both)."""
    w, wd = weights
    B = len(lengths)
    nv = 0 if visual is None else visual.shape[1]
    envs = list(range(B))
    u = I.make_turn_inputs(WL, 0).uniforms[:B]
    orc = O.Oracle(O.shape_from(SH), w, B)
    empty = torch.zeros(0, SH.d_model, dtype=torch.bfloat16)
    orc.prefill(envs, [visual[b] if visual is not None else empty for b in envs],
                [ids[b, :lengths[b]].tolist() for b in envs])
    od = orc.decode(envs, u, T, forced=forced)
    feed = forced if forced is not None else torch.as_tensor(od["tokens"], dtype=torch.int32)
    pol = V.Policy(SH, wd, B, cap, B * (nv + max(lengths) + 8))
    try:
        pol.prefill(visual.cuda() if visual is not None else None, ids.cuda(), lengths)
        g = pol.decode(u.cuda(), T, forced=feed.cuda())
        pol.sync()
        g = {k: v.cpu().numpy() for k, v in g.items() if v is not None}
        lens = [V.vla_context_length(pol.h, b) for b in envs]
    finally:
        pol.close()
    rep = P.compare_decode(0, envs, od, g)
    print(rep)
    return rep, lens


def test_text_only_prefill_with_single_row_chunks(weights):
    inp = I.make_turn_inputs(WL, 0)
    lengths = [1, 5, 16, 9]
    rep, lens = _rollout(weights, None, inp.ids, lengths, cap=64)
    assert rep.ok(), rep
    assert lens == [n + 6 for n in lengths]


def test_context_fills_the_kv_cache_exactly(weights):
    inp = I.make_turn_inputs(WL, 0)
    lengths = [16] * 4                       # 64 visual + 16 text = 80 rows per env
    rep, lens = _rollout(weights, inp.visual, inp.ids, lengths, cap=86)
    assert rep.ok(), rep
    assert lens == [86] * 4
    w, wd = weights
    pol = V.Policy(SH, wd, 4, 85, 4 * 88)
    try:
        vis, ids = inp.visual.cuda(), inp.ids.cuda()
        rc = V.vla_prefill(pol.h, 4, vis.data_ptr(), 64, ids.data_ptr(), lengths, ids.shape[1])
        assert rc == V.VLA_ERR_CAPACITY
        assert V.vla_context_length(pol.h, 0) == 0
    finally:
        pol.close()


def test_forced_edge_bins(weights):
    inp = I.make_turn_inputs(WL, 0)
    edge = torch.tensor([0, 255, 0, 255, 255, 0, 255], dtype=torch.int32)
    forced = torch.stack([BASE + edge.roll(b) for b in range(4)]).to(torch.int32)
    rep, _ = _rollout(weights, inp.visual, inp.ids, inp.lengths.tolist(), cap=128, forced=forced)
    assert rep.ok(), rep


def test_shape_whose_sections_straddle_weight_tiles(monkeypatch):
    # d = 640: q, k and v each end inside a 256-row weight tile, and d_ffn is no multiple of one
    import sys
    sh = I.ModelShape("tiny", 2, 640, 10, 64, 1712)
    monkeypatch.setattr(sys.modules[__name__], "SH", sh)
    w = I.make_weights(sh, WL.weight_seed)
    ids = I.make_turn_inputs(WL, 0).ids
    rep, _ = _rollout((w, P.weights_to_device(w)), None, ids, [1, 5, 12], 64)
    assert rep.ok(), rep


def test_decode_attention_whole_pairs_and_a_split_rest(weights):
    # 320 envs x 4 heads: more pairs than CTAs resident at once (1216), so the last 64 pairs, envs 304
    # and up, are cut into key ranges while the others take one CTA each; lengths differ, the shortest
    # leaves ranges without keys
    w, wd = weights
    B, envs = 320, [0, 303, 304, 311, 319]
    lengths = [130 - 9 * (b % 14) for b in range(B)]
    ids = I.randint_i32((B, 130), 5, 6, 0, BASE - 1)
    u = I.uniform_f32((B, SH.action_dim, SH.n_bins), 5, 7)
    orc = O.Oracle(O.shape_from(SH), w, len(envs))
    local = list(range(len(envs)))
    empty = torch.zeros(0, SH.d_model, dtype=torch.bfloat16)
    orc.prefill(local, [empty for _ in envs], [ids[b, :lengths[b]].tolist() for b in envs])
    od = orc.decode(local, u[envs], 1.0)
    feed = torch.full((B, SH.action_dim), BASE, dtype=torch.int32)
    feed[envs] = torch.as_tensor(od["tokens"], dtype=torch.int32)
    pol = V.Policy(SH, wd, B, 160, B * 131)
    try:
        pol.prefill(None, ids.cuda(), lengths)
        g = pol.decode(u.cuda(), 1.0, forced=feed.cuda())
        pol.sync()
        g = {k: v.cpu().numpy()[envs] for k, v in g.items() if v is not None}
    finally:
        pol.close()
    rep = P.compare_decode(0, local, od, g)
    assert rep.ok(), rep


@pytest.mark.parametrize("B", [42, 43, 53, 54, 64, 71, 72, 73])
def test_score_matches_decode_around_the_wide_residual_gemm(B):
    # 6 B score rows: 252 (tile GEMMs), 258 to 432 (o and down on the wide GEMM: an odd split of the rows over
    # four ranks and padded halves among them), 438 (tile GEMMs again).  The decode runs on activation
    # pairs throughout, the score pass on fp16 activations past q|k|v: 2^-11 a layer and projection
    sh = I.ModelShape("tiny", 2, 4096, 32, 128, 4616)
    w = P.weights_to_device(I.make_weights(sh, 11))
    ids = I.randint_i32((B, 9), 5, 16, 0, sh.vocab - 257)
    tokens = I.randint_i32((B, sh.action_dim), 5, 17, sh.vocab - 256, sh.vocab - 1).cuda()
    u = I.uniform_f32((B, sh.action_dim, 256), 5, 18).cuda()
    pol = V.Policy(sh, w, B, 32, B * 9)
    try:
        pol.prefill(None, ids.cuda(), [1 + b % 9 for b in range(B)])
        d = pol.decode(u, 1.0, forced=tokens)["logits"].double()
        s = pol.score(tokens, 1.0)["logits"].double()
        pol.sync()
    finally:
        pol.close()
    assert ((s - d).norm() / d.norm()).item() < 2e-3
    assert (s - d).abs().max().item() < 0.02 * d.abs().max().item()
