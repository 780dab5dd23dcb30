"""Different handles from different threads: every thread trains its own model on its own stream, the very first calls of the
process among them, and gets the bits that a thread alone gets."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import sys, threading
import torch
from paper_2509_16434_b200 import binding as ppo, synth
from paper_2509_16434_b200.learner import Learner

w = synth.Workload("threads", 32, 8, 32, 48, (16, 32, 128, 256), (3, 3, 3, 3), (64,), 1, 2, P=8, A=3)
THREADS = 6
shapes, gammas = synth.param_shapes(w)
learners = []
for i in range(THREADS):
    L = Learner(w, w.B, "cuda")
    offsets = [o for o, _ in L.model.tensors()]
    learners.append((L, synth.init_params(L.model.arena, offsets, shapes, i, ones=gammas), synth.rollout_torch(w, "cuda", i)))
torch.cuda.synchronize()
out, errors = {}, []
gate = threading.Barrier(THREADS)

def work(i, key, wait):
    L, theta, r = learners[i]
    try:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            L.model.load(theta)
            for m in (L.model.adam_m, L.model.adam_v):
                m.zero_()
            L.adam_t = 0
            if wait:
                stream.synchronize()
                gate.wait()
            L.write_rollout(r, r["eps"], r["logp_jitter"])
            L.train(r["last_value"], seed=i)
        stream.synchronize()
        out[key, i] = L.model.master.clone(), L.loss.clone()
    except Exception as e:
        errors.append((i, e))

threads = [threading.Thread(target=work, args=(i, "together", True)) for i in range(THREADS)]
for t in threads: t.start()
for t in threads: t.join()
assert not errors, errors
for i in range(THREADS):
    work(i, "alone", False)
assert not errors, errors
torch.cuda.synchronize()
for i in range(THREADS):
    for a, b in zip(out["together", i], out["alone", i]):
        assert torch.equal(a, b), i
assert ppo.ppo_poll_status() == 0
print("ok")
"""


def test_first_calls_from_several_threads():
    for _ in range(3):  # each child meets its first calls anew
        run = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
        assert run.returncode == 0 and run.stdout.strip() == "ok", run.stdout + run.stderr[-3000:]
