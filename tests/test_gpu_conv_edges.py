"""Convolution kernels at the edges of their tiles: odd extents, segments that do not divide a row, several small images
per tile, every chunk width, single rows and columns of outputs, micro-batches that leave the last tile part empty."""
import numpy as np
import pytest
import torch

import test_gpu_learner as base
from helpers import rel_l2
from oracle import oracle as orc
from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth

pytestmark = pytest.mark.gpu


def _net(name, H, W, conv_c, conv_k, N=6, T=2, **kw):
    return synth.Workload(name, N, T, H, W, conv_c, conv_k, (40,), 1, 2, P=16, A=3, **kw)


NETS = {
    "narrow_16_32": _net("narrow_16_32", 17, 22, (16, 32), (3, 3)),
    "chunks_of_16": _net("chunks_of_16", 37, 30, (48, 64, 32), (3, 3, 3)),
    "two_chunks": _net("two_chunks", 33, 46, (32, 64, 128), (5, 3, 3)),
    "three_groups": _net("three_groups", 30, 50, (32, 32, 96, 32), (3, 3, 3, 3)),
    "wide_rows": _net("wide_rows", 12, 530, (16, 64, 32), (3, 3, 3), N=2),
    "tall": _net("tall", 261, 14, (32, 64), (3, 3), N=2),
    "small_images": _net("small_images", 14, 18, (32, 64, 64, 64), (3, 3, 3, 3), N=14, T=3),
    "one_block": _net("one_block", 8, 8, (16, 32, 64), (3, 3, 3), N=2),
    "tall_kernels": _net("tall_kernels", 40, 44, (32, 64, 96), (3, 5, 3)),
    "many_chunks": _net("many_chunks", 20, 26, (32, 128, 256), (3, 3, 3), N=10, T=3),
    "ln_odd": _net("ln_odd", 35, 54, (16, 32, 64, 128), (3, 3, 3, 3), norm=True, embed=32),
    "ln_32": _net("ln_32", 22, 30, (32, 32, 64), (5, 3, 3), norm=True),
}


@pytest.mark.parametrize("name", list(NETS))
def test_conv_stack_matches_oracle(name, monkeypatch):
    w = NETS[name]
    monkeypatch.setitem(base.SHAPES, name, w)
    base.test_backward_matches_oracle_on_identical_activations(name)  # every gradient tensor within 2e-2
    # forward, in micro-batches that do not divide the rows
    B = w.M // w.minibatches
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, max(1, B - 1), theta_scale_head=20.0)
    L.compute_gae(dev["last_value"])
    f, _, _, mu_o, V_o = base._oracle_minibatch(md, lay, theta, roll, action, logp, w, L.hyper, 5, 0, 0, w.minibatches)
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
    mus, vs = [], []
    for r0 in range(0, B, L.microbatch):
        rows = min(L.microbatch, B - r0)
        ppo.ppo_encoder_fwd(L.model, L.mb, r0, rows, L.mean, L.value)
        mus.append(L.mean[:rows].cpu().numpy().copy())
        vs.append(L.value[:rows].cpu().numpy().copy())
    assert ppo.ppo_poll_status() == 0
    assert rel_l2(np.concatenate(mus), mu_o) <= base.ENC_TOL and rel_l2(np.concatenate(vs), V_o) <= base.ENC_TOL


def test_gate_bits_are_the_signs_of_the_activations():
    """The forward kernels' one-bit gates against the activations they stored, also where two warps share a word."""
    for name in ("two_chunks", "ln_odd", "ln_32", "three_groups"):
        w = NETS[name]
        B = w.M // w.minibatches
        L, md, lay, theta, roll, action, logp, dev = base._setup(w, B)
        L.compute_gae(dev["last_value"])
        ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
        ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, L.mean, L.value)
        Ho, Wo = orc.conv_shapes(md)
        for l, (h, wd, c) in enumerate(zip(Ho, Wo, md.conv_c), start=1):
            if c % 32 or l == len(md.conv_c):
                continue
            act = L.model.activation(0, l)[:B * h * wd * c].float().cpu().numpy().reshape(-1, c // 32, 32)
            word = L.model.activation(2, l)[:B * h * wd * c // 32].cpu().numpy().view(np.uint32).reshape(-1, c // 32)
            ch = np.arange(32)
            bits = (word[:, :, None] >> (ch // 2 + 16 * (ch % 2))) & 1
            assert np.array_equal(bits != 0, act > 0), (name, l)


# layers whose gate the input gradient reads as half words of bits (16 channels, halo kernel), as activations (48, generic kernel)
# and as bits (32)
@pytest.mark.parametrize("name", ["narrow_16_32", "ln_odd", "chunks_of_16", "two_chunks"])
def test_gate_is_open_for_positive_activations_only(name):
    """Saved activations written from outside may be anything: minus zero, negative numbers and NaN close the gate as zero
    does, in both halves of a pair and without a trace in the neighbouring channel.  The first layer's gradients, which see
    these activations through the gate alone, keep every bit."""
    w = NETS[name]
    B = w.M // w.minibatches
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, B)
    h = L.hyper
    L.compute_gae(dev["last_value"])
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, L.mean, L.value)
    L.loss.zero_()
    ppo.ppo_loss_fwd_bwd(L.model, L.mb, 0, B, B, L.mean, L.value, h.clip, h.vf_coef, h.ent_coef, L.loss, L.dmean, L.dvalue)
    act = L.model.activation(0, 1).view(torch.int16)
    saved = act.clone()
    where = torch.rand(act.shape, device=act.device, generator=torch.Generator(act.device).manual_seed(1)) < 0.3
    closed = [0x0000, 0x8000, 0x8001, 0xBF80, 0xFF80, 0x7FC0, 0x7FFF, 0xFFC0]  # 0, -0, -tiny, -1, -inf, NaN, NaN, -NaN

    def first_layer(pattern):
        act.copy_(torch.where(where, torch.tensor(pattern - 0x10000 if pattern & 0x8000 else pattern, dtype=torch.int16,
                                                  device=act.device), saved))
        ppo.ppo_model_sync_masks(L.model, B)
        ppo.ppo_model_zero_grad(L.model)
        ppo.ppo_encoder_bwd(L.model, L.mb, 0, B, L.dmean, L.dvalue, True)
        assert ppo.ppo_poll_status() == 0
        (o0, s0), (o1, s1) = L.model.tensors()[:2]
        return L.model.grad[o0:o1 + s1].clone()

    want = first_layer(closed[0])
    assert torch.isfinite(want).all() and float(want.norm()) > 0
    for pattern in closed[1:]:
        assert torch.equal(first_layer(pattern), want), hex(pattern)


# Calls of 4 M pixels of the first layer and more: odd grids, a last trip of fewer than 32 pixels, rows wider than a tile, small images, one
# and two chunks of output channels.  The last two keep the second layer's input gradient on chip.
@pytest.mark.parametrize("rows,H,W,C2", [(2901, 61, 90, 64), (953, 31, 530, 32), (15701, 30, 34, 48), (1301, 112, 110, 128),
                                         (801, 124, 164, 64), (2541, 69, 90, 32)])
def test_first_layer_gradient_of_a_whole_call_is_that_of_its_pieces(rows, H, W, C2):
    """One backward call against the same rows in four: fp32 sums of the same products in another grouping.  A sum of 4 M terms
    runs through chains of at most 200 additions, 200 x 2^-24 = 1.2e-5 of its parts; one trip of 32 pixels left out is 3e-3."""
    w = synth.Workload("whole", rows, 1, H, W, (32, C2), (3, 3), (32,), 1, 1, P=16, A=3)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, rows)
    h = L.hyper
    L.compute_gae(dev["last_value"])
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, 1, L.mb)
    n = sum(s for _, s in L.model.tensors()[:2])
    o0 = L.model.tensors()[0][0]

    def gradients(pieces, dmean=None, dvalue=None):
        ppo.ppo_model_zero_grad(L.model)
        step = -(-rows // pieces)
        for r0 in range(0, rows, step):
            k = min(step, rows - r0)
            ppo.ppo_encoder_fwd(L.model, L.mb, r0, k, L.mean, L.value)
            if dmean is None:
                L.loss.zero_()
                ppo.ppo_loss_fwd_bwd(L.model, L.mb, 0, rows, rows, L.mean, L.value, h.clip, h.vf_coef, h.ent_coef, L.loss, L.dmean,
                                     L.dvalue)
                dm, dv = L.dmean, L.dvalue
            else:
                dm, dv = dmean[r0:r0 + k].contiguous(), dvalue[r0:r0 + k].contiguous()
            ppo.ppo_encoder_bwd(L.model, L.mb, r0, k, dm, dv, True)
        assert ppo.ppo_poll_status() == 0
        return L.model.grad[o0:o0 + n].clone()

    whole = gradients(1)
    again = gradients(1)
    pieces = gradients(4, L.dmean.clone(), L.dvalue.clone())
    assert torch.equal(whole, again)
    assert torch.isfinite(whole).all() and float(whole.norm()) > 0
    assert float((whole - pieces).norm() / pieces.norm()) <= 5e-5


# odd grids, a last trip of fewer than 32 pixels, rows wider than a tile (201 x 268); an odd number of row groups in flight with short last ones
# (124 x 164, 69 x 90: of 164 and 225 pixels), a last one of 54 (162 x 108); then calls that take the two kernels, for their channels, the
# size of their tiles (348 and 353 pixels) and their own
@pytest.mark.parametrize("rows,H,W,C2,one", [(1009, 110, 146, 64, True), (801, 124, 164, 64, True), (2541, 69, 90, 64, True),
                                             (917, 162, 108, 64, True), (2541, 69, 90, 32, True), (300, 201, 268, 64, True),
                                             (1479, 90, 122, 48, False), (1479, 90, 122, 128, False), (1477, 90, 122, 16, False),
                                             (2901, 61, 90, 64, False), (953, 31, 530, 32, False), (1457, 90, 122, 64, False)])
def test_first_layer_gradient_is_that_of_the_two_kernels(rows, H, W, C2, one):
    """The same bits from the one launch as from input gradient and weight gradient by themselves, time and again, where a backward
    call makes the one; elsewhere it is refused."""
    w = synth.Workload("first", rows, 1, H, W, (32, C2), (3, 3), (32,), 1, 1, P=16, A=3)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, rows)
    L.compute_gae(dev["last_value"])
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, 1, L.mb)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, rows, L.mean, L.value)
    g = torch.Generator("cuda").manual_seed(1)
    L.dmean.normal_(generator=g)
    L.dvalue.normal_(generator=g)
    (o0, _), (o1, s1) = L.model.tensors()[:2]

    def gradients(call, *args):
        ppo.ppo_model_zero_grad(L.model)
        before = ppo.ppo_launch_count()
        call(L.model, L.mb, 0, rows, *args)
        launches = ppo.ppo_launch_count() - before
        assert ppo.ppo_poll_status() == 0
        return L.model.grad[o0:o1 + s1].clone(), launches

    whole, _ = gradients(ppo.ppo_encoder_bwd, L.dmean, L.dvalue, True)
    two, launches = gradients(ppo.ppo_selftest_first_gradient, False)
    assert torch.isfinite(two).all() and float(two.norm()) > 0
    assert launches == 3 and torch.equal(two, whole)
    if not one:
        with pytest.raises(ppo.PpoError):
            gradients(ppo.ppo_selftest_first_gradient, True)
        return
    for _ in range(5):
        again, launches = gradients(ppo.ppo_selftest_first_gradient, True)
        assert launches == 2 and torch.equal(again, two)
