"""What a handle keeps on the device between calls (the counters of the loss, of the recurrent time loop and of the one-launch
GAE, the transposed weights of the backward pass) when the first call, or an update of the weights, is captured into a graph.
Work that is captured has not run: an eager call has to make its own, and a graph must not lean on what ran before it.

Workspaces start out as junk bytes, as memory of a caller's own arena would."""
import pytest
import torch

from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth
from paper_2509_16434_b200.learner import Learner

pytestmark = pytest.mark.gpu
DEV = "cuda"

W_PLAIN = synth.Workload("graph", 32, 8, 32, 48, (16, 32, 128, 256), (3, 3, 3, 3), (64,), 1, 2, P=8, A=3)
W_REC = synth.Workload("graph_rec", 16, 4, 32, 48, (16, 32), (3, 3), (64,), 1, 2, P=32, A=3, n_lstm=2, lstm_h=64)


def _learner(w, seed=0):
    L = Learner(w, w.B, DEV)
    L.model.workspace.fill_(0x5A)
    L.buffer.storage.fill_(0x5A)
    shapes, gammas = synth.param_shapes(w)
    L.model.load(synth.init_params(L.model.arena, [o for o, _ in L.model.tensors()], shapes, seed, ones=gammas))
    r = synth.rollout_torch(w, DEV, seed)
    L.write_rollout(r, r["eps"], r["logp_jitter"])
    L.compute_gae(r["last_value"])
    return L, r


def _captured(fn):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        fn()
    return g


def _forward_and_loss(L):
    """Forward and loss of minibatch 0."""
    w, h = L.w, L.hyper
    if L.recurrent:
        ppo.ppo_shuffle_gather_sequences(L.buffer, 1, 0, 0, w.minibatches, L.mb, L.seq_done)
        ppo.ppo_model_set_sequence(L.model, w.T, L.seq_envs, L.seq_done, L.h_init, L.c_init)
    else:
        ppo.ppo_shuffle_gather_minibatch(L.buffer, 1, 0, 0, w.minibatches, L.mb)
    ppo.ppo_model_zero_grad(L.model)
    L.loss.zero_()
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, w.B, L.mean, L.value)
    ppo.ppo_loss_fwd_bwd(L.model, L.mb, 0, w.B, w.B, L.mean, L.value, h.clip, h.vf_coef, h.ent_coef, L.loss, L.dmean, L.dvalue)


def _gradients(L):
    """The same and the backward pass, without an update."""
    _forward_and_loss(L)
    ppo.ppo_encoder_bwd(L.model, L.mb, 0, L.w.B, L.dmean, L.dvalue, True)


def _adam(L, step):
    h = L.hyper
    ppo.ppo_adam_step(L.model, h.lr, h.beta1, h.beta2, h.eps, step)


def _outputs(L):
    torch.cuda.synchronize()
    return L.loss.clone(), L.model.grad.clone(), L.mean.clone(), L.value.clone()


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("w", [W_PLAIN, W_REC], ids=["plain", "recurrent"])
def test_counters_first_used_inside_a_capture(w):
    """Forward and loss; the loss scalars and the log-sigma gradient come from the block that counts itself the last."""
    E, _ = _learner(w)  # all eager; also loads the kernels
    _forward_and_loss(E)
    want = _outputs(E)
    assert float(want[0].abs().min()) > 0 and float(want[1].norm()) > 0
    L, _ = _learner(w)
    g = _captured(lambda: _forward_and_loss(L))
    _forward_and_loss(L)  # before the graph has ever run
    assert _same(_outputs(L), want)
    for t in (L.model.grad, L.loss, L.mean, L.value):
        t.fill_(7.0)
    L.model.workspace.fill_(0x5A)  # the graph leans on nothing that ran before it
    g.replay()
    assert _same(_outputs(L), want)
    assert ppo.ppo_poll_status() == 0


@pytest.mark.parametrize("w", [W_PLAIN, W_REC], ids=["plain", "recurrent"])
def test_backward_first_used_inside_a_capture(w):
    E, _ = _learner(w)  # all eager; also loads the kernels
    _gradients(E)
    want = _outputs(E)
    assert torch.isfinite(want[1]).all() and float(want[1].norm()) > 0
    L, _ = _learner(w)
    g = _captured(lambda: _gradients(L))
    _gradients(L)  # before the graph has ever run
    assert _same(_outputs(L), want)
    L.model.grad.fill_(7.0)
    L.loss.fill_(7.0)
    g.replay()
    assert _same(_outputs(L), want)
    _gradients(L)
    assert _same(_outputs(L), want)
    assert ppo.ppo_poll_status() == 0


@pytest.mark.parametrize("w", [W_PLAIN, W_REC], ids=["plain", "recurrent"])
def test_graph_without_earlier_calls_of_its_own(w):
    """A graph captured after eager calls carries what it needs: it gives the same result on weights that were replaced and
    in a workspace that was overwritten since."""
    L, _ = _learner(w)
    _gradients(L)
    g = _captured(lambda: _gradients(L))
    M, _ = _learner(w, seed=1)
    L.model.load(M.model.master)
    L.model.workspace.fill_(0x5A)
    for a, b in ((L.buffer.storage, M.buffer.storage), (L.stats, M.stats)):
        a.copy_(b)
    g.replay()
    got = _outputs(L)
    _gradients(M)
    assert _same(got, _outputs(M))
    assert ppo.ppo_poll_status() == 0


@pytest.mark.parametrize("w", [W_PLAIN, W_REC], ids=["plain", "recurrent"])
def test_update_inside_a_graph_reaches_eager_backward(w):
    E, _ = _learner(w)
    L, _ = _learner(w)
    for X in (E, L):
        _gradients(X)
    g = _captured(lambda: _adam(L, 1))
    for step in range(3):  # the host sees one captured update, the device three
        _gradients(L)
        g.replay()
        _gradients(E)
        _adam(E, 1)
    _gradients(E)
    _gradients(L)
    torch.cuda.synchronize()
    assert torch.equal(E.model.master, L.model.master)
    assert _same(_outputs(L), _outputs(E))
    assert ppo.ppo_poll_status() == 0


def test_whole_minibatch_as_a_graph():
    w = W_PLAIN
    E, _ = _learner(w)
    L, _ = _learner(w)

    def step(X):
        _gradients(X)
        _adam(X, 1)

    step(E)
    L.model.load(L.model.master.clone())
    g = _captured(lambda: step(L))
    g.replay()
    for _ in range(2):
        g.replay()
        step(E)
    torch.cuda.synchronize()
    assert torch.equal(E.model.master, L.model.master) and torch.equal(E.model.grad, L.model.grad)
    assert ppo.ppo_poll_status() == 0


def test_one_launch_gae_first_used_inside_a_capture():
    w = W_PLAIN
    E, r = _learner(w)
    ppo.ppo_compute_gae(E.buffer, r["last_value"], w.gamma, w.lam, 2, E.stats)
    want = [E.buffer.field(f).clone() for f in (ppo.FIELD_ADV, ppo.FIELD_RET)] + [E.stats.clone()]
    L, r = _learner(w)
    g = _captured(lambda: ppo.ppo_compute_gae(L.buffer, r["last_value"], w.gamma, w.lam, 2, L.stats))
    out = lambda: [L.buffer.field(f).clone() for f in (ppo.FIELD_ADV, ppo.FIELD_RET)] + [L.stats.clone()]
    ppo.ppo_compute_gae(L.buffer, r["last_value"], w.gamma, w.lam, 2, L.stats)  # before the graph has ever run
    assert _same(out(), want)
    L.buffer.field(ppo.FIELD_SCRATCH).fill_(float("nan"))
    L.buffer.field(ppo.FIELD_ADV).fill_(7.0)
    g.replay()
    assert _same(out(), want)
    assert ppo.ppo_poll_status() == 0
