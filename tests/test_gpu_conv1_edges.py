"""First convolution at the edges of its stages: several frames per stage, frame rows that are no multiple of 16 bytes, the
last stage part empty, every filter count and kernel size, frames too wide for the shared-memory run."""
import numpy as np
import pytest

import test_gpu_learner as base
from helpers import rel_l2
from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,C1,k,norm", [(8, 10, 16, 3, False), (9, 14, 16, 5, False), (31, 42, 32, 3, False),
                                           (31, 42, 32, 5, False), (21, 26, 48, 3, False), (40, 34, 64, 3, False),
                                           (16, 18, 16, 3, True), (23, 38, 32, 5, True), (12, 20, 32, 7, False),
                                           (7, 4002, 16, 3, False), (6, 1302, 32, 5, False)])
@pytest.mark.parametrize("rows", [1, 7])
def test_first_layer_matches_oracle(H, W, C1, k, norm, rows):
    w = synth.Workload("c1", rows, 2, H, W, (C1, 32), (k, 3), (32,), 1, 1, P=8 if not norm else 32, A=3, norm=norm)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, 2 * rows, theta_scale_head=20.0)
    L.compute_gae(dev["last_value"])
    f, _, _, mu_o, V_o = base._oracle_minibatch(md, lay, theta, roll, action, logp, w, L.hyper, 5, 0, 0, 1)
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, 1, L.mb)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, 2 * rows, L.mean, L.value)
    assert ppo.ppo_poll_status() == 0
    _, _, acts = base.orc.encoder_fwd(md, base.orc.round_weights(md, theta), f["depth"], f["proprio"], True)
    n = ((H + 2 * (k // 2) - k) // 2 + 1) * ((W + 2 * (k // 2) - k) // 2 + 1) * C1
    got = L.model.activation(0, 1)[:2 * rows * n].float().cpu().numpy().reshape(2 * rows, n)
    assert rel_l2(got, acts[:, H * W:H * W + n]) <= base.ENC_TOL
    assert rel_l2(L.mean[:2 * rows].cpu().numpy(), mu_o) <= base.ENC_TOL
