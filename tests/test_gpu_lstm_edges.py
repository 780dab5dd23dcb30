"""Recurrent layers as one kernel per direction at the edges of their tiles (32, 64 or 128 envs, 16 units per CTA), the step-by-step
path where not all CTAs fit the GPU, and what acting does differently: the embedding in slabs and the state reset."""
import numpy as np
import pytest
import torch

import test_gpu_lstm as base
from helpers import oracle_model, rel_l2
from oracle import oracle as orc
from paper_2509_16434_b200 import synth
from test_gpu_learner import ENC_TOL

pytestmark = pytest.mark.gpu
DEV = "cuda"


# envs per sequence group, units, steps: one env, one short / exact / one over a tile, three tiles, too many CTAs; tiles of 32, 64
# and 128 envs with a ragged last one; clusters of four that do not all fit (36 of them) beside single CTAs that do
@pytest.mark.parametrize("Be,H,T", [(1, 64, 3), (127, 64, 3), (128, 192, 4), (129, 128, 3), (257, 448, 3), (257, 1024, 3),
                                    (33, 128, 5), (161, 512, 3), (255, 1024, 3), (385, 576, 3)])
def test_sequences_at_tile_edges_match_oracle(Be, H, T, monkeypatch):
    w = synth.Workload("edge", 2 * Be, T, 8, 12, (16, 32), (3, 3), (24,), 1, 2, P=32, A=3, n_lstm=2, lstm_h=H)
    monkeypatch.setitem(base.REC, "edge", w)
    base.test_forward_through_time_matches_oracle("edge", False)
    base.test_backward_through_time_matches_oracle_on_identical_state("edge")


# one step of a recurrent policy: 1024 rows and fewer take the embedding (4096 inputs) in slabs, one more does not
@pytest.mark.parametrize("n_lstm", [0, 1])
@pytest.mark.parametrize("n", [1, 65, 1024, 1025])
def test_acting_matches_oracle(n, n_lstm):
    w = synth.Workload("act", n, 1, 64, 64, (16, 32, 64), (3, 3, 3), (40,), 1, 1, P=32, A=3, embed=32, n_lstm=n_lstm, lstm_h=64)
    md = oracle_model(w)
    lay = orc.param_layout(md)
    theta = synth.init_params(lay.total, lay.offsets, lay.shapes, 3)
    roll = synth.rollout_numpy(w, 3)
    L = base.Learner(w, n, DEV)
    L.model.load(theta)
    dev = {k: torch.as_tensor(v).to(DEV) for k, v in roll.items()}
    used = orc.round_weights(md, theta)
    if n_lstm:
        zero = np.zeros((n_lstm, n, 64), np.float32)
        mu, V, _, _ = orc.encoder_fwd_seq(md, used, roll["depth"], roll["proprio"], roll["done"], zero, zero, True)
        a, lp, val = L.act(dev["depth"][0], dev["proprio"][0], dev["eps"][0])
    else:
        mu, V, _ = orc.encoder_fwd(md, used, roll["depth"][0], roll["proprio"][0], True)
        L.act_into_buffer(0, dev["depth"][0], dev["proprio"][0], dev["eps"][0])
        a, lp, val = (L.buffer.field(f)[0] for f in (base.ppo.FIELD_ACTION, base.ppo.FIELD_LOGP, base.ppo.FIELD_VALUE))
    ls = np.asarray(theta, np.float64)[lay.offsets[-1]:lay.offsets[-1] + md.A]
    want, lp_want = orc.sample_action(mu, ls, roll["eps"].reshape(n, md.A))
    assert base.ppo.ppo_poll_status() == 0
    assert rel_l2(a.cpu().numpy(), want) <= ENC_TOL and rel_l2(val.cpu().numpy(), V) <= ENC_TOL
    assert rel_l2(lp.cpu().numpy(), lp_want) <= ENC_TOL


@pytest.mark.parametrize("layers,n,H", [(1, 1, 64), (2, 33, 64), (2, 300, 1024)])
def test_state_reset_clears_finished_envs_only(layers, n, H):
    h, c = (torch.randn((layers, n, H), device=DEV) for _ in range(2))
    done = (torch.arange(n, device=DEV) % 3 == 0).to(torch.uint8) * 7  # any non-zero flag
    want = [torch.where(done[None, :, None] != 0, torch.zeros_like(s), s) for s in (h, c)]
    base.ppo.ppo_state_reset(h, c, done)
    assert torch.equal(h, want[0]) and torch.equal(c, want[1])


# 2048 and 4096 inputs of the embedding, few and many rows
@pytest.mark.parametrize("H,n", [(64, 1), (64, 65), (64, 1025), (72, 300)])
def test_feed_forward_acting_gives_the_bits_of_the_training_forward(H, n):
    """`act`, `act_into_buffer` and the forward of a minibatch with the same frames, in one piece and in micro-batches: the
    log-probability that acting stores belongs to the mean that training starts from."""
    ppo = base.ppo
    w = synth.Workload("act", n, 2, H, 64, (16, 32, 64), (3, 3, 3), (40,), 1, 1, P=32, A=3, norm=True, embed=32)
    L, small = base.Learner(w, w.B, DEV), base.Learner(w, max(1, n // 3), DEV)
    shapes, gammas = synth.param_shapes(w)
    theta = synth.init_params(L.model.arena, [o for o, _ in L.model.tensors()], shapes, 3, ones=gammas)
    r = synth.rollout_torch(w, DEV, 3)
    depth, proprio, eps = r["depth"][0], r["proprio"][0], r["eps"][0]
    zero = torch.zeros_like(eps)  # actions are then the means
    got = []
    for X in (L, small):
        X.model.load(theta)
        a, lp, v = X.act(depth, proprio, eps)
        X.act_into_buffer(0, depth, proprio, eps)
        got += [(a, lp, v), tuple(X.buffer.field(f)[0].clone() for f in (ppo.FIELD_ACTION, ppo.FIELD_LOGP, ppo.FIELD_VALUE))]
    for other in got[1:]:
        assert all(torch.equal(x, y) for x, y in zip(got[0], other))
    both = ppo.Minibatch(r["depth"].data_ptr(), r["proprio"].data_ptr(), None, None, None, None, None, None, 2 * n)
    ppo.ppo_encoder_fwd(L.model, both, 0, 2 * n, L.mean, L.value)  # 2 n rows at once, as training takes them
    mean = L.act(depth, proprio, zero)[0]
    ppo.ppo_encoder_fwd(L.model, both, 0, 2 * n, L.mean, L.value)
    assert torch.equal(L.mean[:n], mean) and torch.equal(L.value[:n], got[0][2])
    assert ppo.ppo_poll_status() == 0


def test_recurrent_acting_stays_within_a_rounding_of_the_sequence():
    """Steps taken one by one (embedding in slabs) against the same steps as one sequence (one sum).  The two sums of an
    embedding differ in fp32; rounded to bf16 a value may fall to the other side, a step of at most 2^-8 of it, and what
    follows (gates, layers of unit gain) does not enlarge a relative difference beyond that."""
    w = synth.Workload("act_seq", 9, 3, 64, 64, (16, 32, 64), (3, 3, 3), (40,), 1, 1, P=32, A=3, norm=True, embed=32, n_lstm=2, lstm_h=128)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, w.B)
    ppo = base.ppo
    steps = []
    for t in range(w.T):
        steps.append(L.act(dev["depth"][t], dev["proprio"][t], dev["eps"][t]))
        L.reset_rollout_state(w.N, dev["done"][t])
    rows = w.T * w.N
    seq = ppo.Minibatch(dev["depth"].data_ptr(), dev["proprio"].data_ptr(), None, None, None, None, None, None, rows)
    ppo.ppo_model_set_sequence(L.model, w.T, w.N, dev["done"], L.h_init, L.c_init)
    ppo.ppo_encoder_fwd(L.model, seq, 0, rows, L.mean, L.value)
    a, lp = torch.empty((rows, w.A), device=DEV), torch.empty(rows, device=DEV)
    ppo.ppo_policy_sample(L.model, rows, L.mean, dev["eps"].reshape(rows, w.A), a, lp)
    got_a, got_lp, got_v = (torch.cat([s[i] for s in steps]) for i in range(3))
    # the same noise on both sides: actions differ by the means
    d = (got_a - a).norm() / L.mean[:rows].norm(), (got_v - L.value[:rows]).norm() / L.value[:rows].norm()
    print(f"one by one against one sequence: mean {float(d[0]):.2e}, value {float(d[1]):.2e}")
    assert float(max(d)) <= 2.0 ** -8
    assert torch.equal(got_lp, lp)  # of the action under its own mean: noise and log-sigma only
    assert ppo.ppo_poll_status() == 0


# one launch per layer and step in every shape (32 x 8, 32 x 16, 64 x 16, 128 x 16, 128 x 32 envs x units, the last in one wave and in
# two), ragged tiles, inputs of one, two and three chunks; two launches where the state's pointers are odd
@pytest.mark.parametrize("n,H,P", [(1, 64, 32), (33, 512, 160), (65, 512, 96), (161, 512, 32), (300, 512, 160), (600, 512, 96), (700, 1024, 32)])
def test_steps_one_by_one_give_the_bits_of_the_sequence(n, H, P):
    w = synth.Workload("one", n, 2, 8, 12, (16, 32), (3, 3), (24,), 1, 1, P=P, A=3, n_lstm=2, lstm_h=H)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, w.B)
    ppo = base.ppo
    roll["done"][0, 1::3] = 1
    dev["done"] = torch.as_tensor(roll["done"]).to(DEV)
    zero = torch.zeros_like(dev["eps"][0])  # actions are then the means
    got = []
    for t in range(w.T):
        got.append(L.act(dev["depth"][t], dev["proprio"][t], zero))
        L.reset_rollout_state(n, dev["done"][t])
    mean, value = (torch.cat([g[i] for g in got]) for i in (0, 2))
    rows = w.T * n
    seq = ppo.Minibatch(dev["depth"].data_ptr(), dev["proprio"].data_ptr(), None, None, None, None, None, None, rows)
    odd = [torch.zeros(L.h_init.numel() + 1, device=DEV)[1:].view_as(L.h_init) for _ in range(2)]
    for h0, c0 in ((torch.zeros_like(L.h_init), torch.zeros_like(L.c_init)), odd):
        ppo.ppo_model_set_sequence(L.model, w.T, n, dev["done"], h0, c0)
        ppo.ppo_encoder_fwd(L.model, seq, 0, rows, L.mean, L.value)
        assert torch.equal(mean, L.mean[:rows]) and torch.equal(value, L.value[:rows])
    zero_state = np.zeros((w.n_lstm, n, H), np.float32)
    mu, V, _, _ = orc.encoder_fwd_seq(md, orc.round_weights(md, theta), roll["depth"], roll["proprio"], roll["done"], zero_state, zero_state, True)
    assert ppo.ppo_poll_status() == 0
    assert rel_l2(mean.cpu().numpy(), mu) <= ENC_TOL and rel_l2(value.cpu().numpy(), V) <= ENC_TOL
