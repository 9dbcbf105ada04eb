"""Learning-phase quantities on the GPU (C ABI) vs the fp64 oracle: GAE (Algorithm 1) and the
clipped PPO objective (Eq. 2).  Inputs are seeded; the value head and the rollout entropy are
checked on every workload inside the parity runs (tests/parity.py)."""
import numpy as np
import pytest
import torch

import oracle.vla_oracle as O
from paper_2505_18719_gb300 import inputs as I
from paper_2505_18719_gb300 import vla as V

pytestmark = pytest.mark.gpu


def _gae_inputs(M, B, seed):
    r = I.normal_bf16((M, B), seed, 1, 1.0).float()
    v = I.normal_bf16((M + 1, B), seed, 2, 2.0).float()
    dn = (I.uniform_f32((M, B), seed, 3) < 0.1).float()
    return r, v, dn


@pytest.mark.parametrize("M,B", [(1, 1), (5, 3), (37, 65), (128, 256)])
@pytest.mark.parametrize("gamma,lam", [(0.99, 0.95), (1.0, 1.0), (0.9, 0.0)])
def test_gae_matches_oracle(M, B, gamma, lam):
    r, v, dn = _gae_inputs(M, B, 100 + M + B)
    rd, vd, dd = r.cuda(), v.cuda(), dn.cuda()
    adv = torch.full((M, B), float("nan"), device="cuda")
    ret = torch.full((M, B), float("nan"), device="cuda")
    assert V.vla_gae(rd.data_ptr(), vd.data_ptr(), dd.data_ptr(), M, B, gamma, lam, adv.data_ptr(),
                     ret.data_ptr(), 0) == 0
    torch.cuda.synchronize()
    oa, orr = O.gae(r.double(), v.double(), dn.double(), gamma, lam)
    scale = 1.0 + float(oa.abs().max())
    assert float((adv.cpu().double() - oa).abs().max()) < 2e-6 * scale * M ** 0.5
    assert float((ret.cpu().double() - orr).abs().max()) < 2e-6 * scale * M ** 0.5


@pytest.mark.parametrize("N", [1, 7, 5000])
@pytest.mark.parametrize("eps", [0.2, 0.0])
def test_ppo_clip_matches_oracle_and_is_deterministic(N, eps):
    A = 7
    lp_old = -I.uniform_f32((N, A), 200 + N, 1) * 6.0
    lp_new = lp_old + (I.uniform_f32((N, A), 200 + N, 2) - 0.5) * 0.12
    adv = I.normal_bf16((N,), 200 + N, 3, 1.0).float()
    d = [t.cuda() for t in (lp_new, lp_old, adv)]
    outs = []
    for _ in range(2):
        obj = torch.full((1,), float("nan"), device="cuda")
        rho = torch.full((N,), float("nan"), device="cuda")
        cf = torch.full((1,), float("nan"), device="cuda")
        assert V.vla_ppo_clip(d[0].data_ptr(), d[1].data_ptr(), d[2].data_ptr(), N, A, eps, obj.data_ptr(),
                              rho.data_ptr(), cf.data_ptr(), 0) == 0
        torch.cuda.synchronize()
        outs.append((obj.item(), rho.cpu(), cf.item()))
    assert outs[0][0] == outs[1][0] and torch.equal(outs[0][1], outs[1][1])
    o_obj, o_rho, o_cf = O.ppo_clip_objective(lp_new.double(), lp_old.double(), adv.double(), eps)
    assert abs(outs[0][0] - o_obj) < 1e-5 * (1.0 + abs(o_obj))
    assert float((outs[0][1].double() - o_rho).abs().max()) < 1e-5
    # a sample within fp32 rounding of |rho - 1| = eps may be counted differently
    near = int(((o_rho - 1.0).abs() - eps).abs().lt(1e-5).sum())
    assert abs(outs[0][2] - o_cf) <= (near + 0.5) / N


# chunk and lane edges of the GAE kernel: 64-step chunks (a partial one comes first), 32 envs per CTA
@pytest.mark.parametrize("M,B", [(63, 32), (64, 33), (65, 31), (129, 1), (300, 40)])
def test_gae_chunk_edges(M, B):
    test_gae_matches_oracle(M, B, 0.99, 0.95)


# tile and cluster edges of the PPO kernel (512-sample tiles on 1, 2, 4, 8 or 16 CTAs, then round-robin)
# and its three ways to read a sample: staged scalars, staged float4 (A % 4 == 0), in place (A > 16 or
# log-probs off the 16-byte boundary)
@pytest.mark.parametrize("N,A,offset", [(511, 1, 0), (513, 4, 0), (1024, 16, 0), (1537, 17, 0), (4097, 8, 0),
                                        (8193, 7, 0), (25000, 6, 0), (2000, 7, 1)])
def test_ppo_clip_tile_edges(N, A, offset):
    lp_old = torch.cat([torch.zeros(offset), (-I.uniform_f32((N, A), 300 + N, 1) * 6.0).view(-1)])
    d = (I.uniform_f32((N, A), 300 + N, 2) - 0.5) * 0.12
    lp_new = torch.cat([torch.zeros(offset), lp_old[offset:] + d.view(-1)])
    adv = I.normal_bf16((N,), 300 + N, 3, 1.0).float()
    gn, go, ga = lp_new.cuda(), lp_old.cuda(), adv.cuda()
    obj, cf, rho = (torch.full((k,), float("nan"), device="cuda") for k in (1, 1, N))
    assert V.vla_ppo_clip(gn.data_ptr() + 4 * offset, go.data_ptr() + 4 * offset, ga.data_ptr(), N, A, 0.2,
                          obj.data_ptr(), rho.data_ptr(), cf.data_ptr(), 0) == 0
    torch.cuda.synchronize()
    o_obj, o_rho, o_cf = O.ppo_clip_objective(lp_new[offset:].view(N, A).double(), lp_old[offset:].view(N, A).double(),
                                              adv.double(), 0.2)
    # A fp32 differences of values up to 6 (each within 2^-22) under an exponential of magnitude ~1
    assert float((rho.cpu().double() - o_rho).abs().max()) < A * 2.0 ** -20
    assert abs(obj.item() - o_obj) < A * 2.0 ** -20
    near = int(((o_rho - 1.0).abs() - 0.2).abs().lt(1e-5).sum())
    assert abs(cf.item() - o_cf) <= (near + 0.5) / N


# the objective's step from one CTA that reads in place to clusters that stage
@pytest.mark.parametrize("N,A", [(1, 1), (512, 7), (512, 8), (1024, 7), (1024, 1), (1024, 8), (1025, 7)])
def test_ppo_clip_small_calls(N, A):
    test_ppo_clip_tile_edges(N, A, 0)


# a device (a partition, a client with few SMs) that cannot place clusters of 16 CTAs: fewer CTAs take the tiles
@pytest.mark.parametrize("most", [8, 4, 2, 1])
def test_ppo_clip_on_smaller_clusters(most):
    try:
        assert V.vla_test_set_max_cluster(most) == 0
        for N, A in ((4097, 8), (8193, 7), (25000, 12)):
            test_ppo_clip_tile_edges(N, A, 0)
    finally:
        V.vla_test_set_max_cluster(0)


def test_learning_entry_points_reject_bad_arguments():
    x = torch.zeros(4, device="cuda")
    p = x.data_ptr()
    assert V.vla_gae(p, p, p, 0, 1, 0.9, 0.9, p) == V.VLA_ERR_ARG
    assert V.vla_gae(p, p, p, 1, 1, 1.5, 0.9, p) == V.VLA_ERR_ARG
    assert V.vla_gae(0, p, p, 1, 1, 0.9, 0.9, p) == V.VLA_ERR_ARG
    assert V.vla_ppo_clip(p, p, p, 0, 7, 0.2, p) == V.VLA_ERR_ARG
    assert V.vla_ppo_clip(p, p, p, 1, 7, -0.1, p) == V.VLA_ERR_ARG
