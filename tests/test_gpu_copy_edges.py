"""Frames and steps whose byte counts are no multiple of the copies' 16-byte units: gather and write_step, bit-exact."""
import numpy as np
import pytest
import torch

from oracle import oracle as orc
from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth

pytestmark = pytest.mark.gpu
DEV = "cuda"


# one pixel (less than a unit), a unit and a half, odd pixel counts (every shift occurs), frames of one and of several
# 16 KB chunks, just below and above a chunk
@pytest.mark.parametrize("N,T,H,W,K", [(5, 3, 1, 1, 3), (5, 3, 3, 4, 1), (6, 4, 17, 23, 2), (4, 3, 90, 122, 3), (3, 2, 63, 129, 1),
                                       (3, 2, 64, 128, 1), (3, 2, 67, 122, 1), (2, 2, 121, 163, 2)])
def test_ragged_frames_are_copied_bit_exactly(N, T, H, W, K):
    w = synth.WORKLOADS["cfg1"].scaled(N, T=T, H=H, W=W, P=5, A=3)
    roll = synth.rollout_numpy(w, 7)
    action, logp = roll["eps"], roll["logp_jitter"]
    buf = ppo.Buffer(ppo.buffer_desc(N, T, H, W, w.P, w.A))
    d = {k: torch.as_tensor(v).to(DEV) for k, v in roll.items()}
    for t in range(T):
        ppo.ppo_buffer_write_step(buf, t, d["depth"][t], d["proprio"][t], d["eps"][t], d["logp_jitter"][t], d["value"][t],
                                  d["reward"][t], d["done"][t])
    for f, name in ((ppo.FIELD_DEPTH, "depth"), (ppo.FIELD_PROPRIO, "proprio"), (ppo.FIELD_ACTION, "eps"),
                    (ppo.FIELD_LOGP, "logp_jitter"), (ppo.FIELD_VALUE, "value"), (ppo.FIELD_REWARD, "reward"), (ppo.FIELD_DONE, "done")):
        assert buf.field(f).cpu().numpy().tobytes() == roll[name].tobytes(), name
    ppo.ppo_compute_gae(buf, d["last_value"], 0.99, 0.95, True, None)
    fields = {"depth": roll["depth"], "proprio": roll["proprio"], "action": action, "logp_old": logp, "value_old": roll["value"],
              "adv": buf.field(ppo.FIELD_ADV).cpu().numpy(), "ret": buf.field(ppo.FIELD_RET).cpu().numpy()}
    B = N * T // K
    for k in range(K):
        mb = ppo.MinibatchArrays(buf.desc, B)
        ppo.ppo_shuffle_gather_minibatch(buf, 3, 1, k, K, mb)
        idx = orc.perm(3, 1, N * T, k * B, B)
        assert np.array_equal(mb.index.cpu().numpy().view(np.uint32), idx)
        want = orc.gather(fields, idx, N)
        for name in fields:
            assert getattr(mb, name).cpu().numpy().tobytes() == want[name].tobytes(), name
    assert ppo.ppo_poll_status() == 0
