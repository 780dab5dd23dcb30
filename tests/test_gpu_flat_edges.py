"""Fully connected layers at the edges of their tiles (rows and columns that no tile width divides, reductions that are no whole
number of chunks), and the gates of the last convolution."""
import ctypes as C

import pytest
import torch

import test_gpu_learner as base
from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth
from test_gpu_conv_edges import NETS, test_conv_stack_matches_oracle as conv_stack_matches_oracle

pytestmark = pytest.mark.gpu


# minibatches of 1, 33, 129 and 300 rows: one row, one past a tile of 32, one past a tile of 128, many ragged tiles; widths that are
# no multiple of 16 or 32, a first layer of 48 + 8 (one ragged chunk) and 64 + 64 columns (two whole chunks)
@pytest.mark.parametrize("N,T,fc,P,last,embed", [
    (2, 1, (40,), 8, 48, 0), (6, 11, (200, 120), 8, 48, 0), (6, 43, (72, 504, 24), 64, 64, 0), (60, 10, (200, 120), 16, 32, 0),
    (6, 11, (128, 56), 16, 32, 32), (6, 43, (200,), 8, 64, 64), (60, 10, (64, 64), 16, 32, 96)])
def test_forward_and_gradients_match_oracle(N, T, fc, P, last, embed, monkeypatch):
    w = synth.Workload("flat", N, T, 16, 24, (16, last), (3, 3), fc, 1, 2, P=P, A=3, embed=embed)
    monkeypatch.setitem(NETS, "flat", w)
    conv_stack_matches_oracle("flat", monkeypatch)  # outputs and every gradient tensor within 2e-2


@pytest.mark.parametrize("name", ["narrow_16_32", "three_groups", "many_chunks", "small_images", "one_block"])
def test_last_gate_is_open_for_positive_activations_only(name):
    """The gradient of the average pool sees the last activations through their gates alone: minus zero, negative numbers and NaN
    close them as zero does, and every gradient keeps its bits."""
    w = NETS[name]
    B = w.M // w.minibatches
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, B)
    h = L.hyper
    L.compute_gae(dev["last_value"])
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, L.mean, L.value)
    L.loss.zero_()
    ppo.ppo_loss_fwd_bwd(L.model, L.mb, 0, B, B, L.mean, L.value, h.clip, h.vf_coef, h.ent_coef, L.loss, L.dmean, L.dvalue)
    act = L.model.activation(0, len(w.conv_c)).view(torch.int16)
    saved = act.clone()
    where = torch.rand(act.shape, device=act.device, generator=torch.Generator(act.device).manual_seed(1)) < 0.3

    def gradients(pattern):
        act.copy_(torch.where(where, torch.tensor(pattern - 0x10000 if pattern & 0x8000 else pattern, dtype=torch.int16,
                                                  device=act.device), saved))
        ppo.ppo_model_sync_masks(L.model, B)
        ppo.ppo_model_zero_grad(L.model)
        ppo.ppo_encoder_bwd(L.model, L.mb, 0, B, L.dmean, L.dvalue, True)
        assert ppo.ppo_poll_status() == 0
        return L.model.grad.clone()

    want = gradients(0x0000)
    assert torch.isfinite(want).all() and float(want.norm()) > 0
    for pattern in (0x8000, 0xBF80, 0xFF80, 0x7FC0, 0xFFC0):  # -0, -1, -inf, NaN, -NaN
        assert torch.equal(gradients(pattern), want), hex(pattern)


# average pool of few rows with many pixels (one and several loads into shared memory, exactly full ones, 32 and 96 channels) beside
# the sum in fp64, rounded to bf16: n sums in fp32 are within n 2^-24 of the sum of the magnitudes, the rounding within 2^-8
@pytest.mark.parametrize("H,W,last,rows", [(44, 48, 32, 1), (64, 128, 96, 3), (90, 92, 32, 5), (45, 47, 64, 200), (130, 140, 64, 2)])
def test_pool_of_large_maps(H, W, last, rows):
    w = synth.Workload("pool", 2 * rows, 1, H, W, (16, last), (3, 3), (40,), 1, 2, P=24, A=3)
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, rows)
    L.compute_gae(dev["last_value"])
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, rows, L.mean, L.value)
    npx = ((H + 3) // 4) * ((W + 3) // 4)
    act = L.model.activation(0, 2)[:rows * npx * last].double().view(rows, npx, last)
    h0 = L.model.activation(1, 0)[:rows * (last + 24)].double().view(rows, last + 24)
    want = act.mean(1)
    assert bool(((h0[:, :last] - want).abs() <= want.abs() * 2.0 ** -8 + act.abs().sum(1) * 2.0 ** -24).all())
    assert torch.equal(h0[:, last:], L.mb.proprio[:rows].to(torch.bfloat16).double())
    assert ppo.ppo_poll_status() == 0


# weight gradient of a 16-channel layer in pairs of pixels: even widths (one pair, a tile that ends inside a row, several tiles per
# row), odd heights, one image and many; an odd width goes pixel by pixel
@pytest.mark.parametrize("H,W,N,last", [(8, 4, 2, 32), (9, 12, 6, 64), (35, 44, 6, 32), (10, 532, 2, 96), (35, 46, 6, 32)])
def test_pairs_of_pixels_match_oracle(H, W, N, last, monkeypatch):
    w = synth.Workload("pairs", N, 2, H, W, (16, last), (3, 3), (40,), 1, 2, P=16, A=3)
    monkeypatch.setitem(NETS, "pairs", w)
    conv_stack_matches_oracle("pairs", monkeypatch)


# the dense chain at its lines: 32 | 64 | 128 rows per tile in clusters of eight, clusters of four, the most rows it takes and one
# more (layer by layer); the widest slices it takes (240 columns of a CTA) and the next width, which it leaves to single layers; a
# CTA without columns of a layer between two of which it has some (120, 200, 120 in slices of 16, 32, 16)
@pytest.mark.parametrize("B,fc", [(33, (120, 200, 120)), (480, (72, 40)), (481, (200, 120)), (961, (72, 504)), (1921, (960,)), (1921, (968,)), (4224, (40,)),
                                  (4225, (40,))])
def test_dense_chain_at_its_lines_matches_oracle(B, fc, monkeypatch):
    w = synth.Workload("chain", 2 * B, 1, 8, 12, (16, 32), (3, 3), fc, 1, 2, P=40, A=3)
    monkeypatch.setitem(NETS, "chain", w)
    conv_stack_matches_oracle("chain", monkeypatch)


class _Mallinfo2(C.Structure):
    _fields_ = [(n, C.c_size_t) for n in ("arena", "ordblks", "smblks", "hblks", "hblkhd", "usmblks", "fsmblks", "uordblks", "fordblks", "keepcost")]


def _heap_bytes():
    libc = C.CDLL(None)
    libc.mallinfo2.restype = _Mallinfo2
    m = libc.mallinfo2()
    return m.uordblks + m.hblkhd


def test_a_chain_with_other_ends_is_the_chain_that_was_prepared():
    """Mean and value, and their gradients, at addresses that no call has seen: every call writes to and reads from its own, and none is
    prepared (or remembered: a prepared chain is 2 KB) again."""
    w = synth.Workload("ends", 64, 1, 8, 12, (16, 32), (3, 3), (504, 72), 1, 1, P=40, A=3)
    n, B = 256, 64
    L = base._setup(w, B)[0]
    L.compute_gae(torch.zeros(64, device="cuda"))
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, 1, L.mb)
    mean, value = torch.full((n, B, 3), -9.0, device="cuda"), torch.full((n, B), -9.0, device="cuda")
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, L.mean, L.value)
    g = torch.Generator("cuda").manual_seed(2)
    L.dmean.copy_(torch.randn((B, 3), device="cuda", generator=g))
    L.dvalue.copy_(torch.randn(B, device="cuda", generator=g))
    dmean, dvalue = torch.zeros_like(mean), torch.zeros_like(value)
    dmean[n - 1], dvalue[n - 1] = L.dmean, L.dvalue

    def gradients(dm, dv):
        ppo.ppo_model_zero_grad(L.model)
        ppo.ppo_encoder_bwd(L.model, L.mb, 0, B, dm, dv, True)

    gradients(L.dmean, L.dvalue)
    want = L.model.grad.clone()
    for i in range(8):
        ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, mean[i], value[i])
        gradients(dmean[i], dvalue[i])
    before = _heap_bytes()
    for i in range(8, n):
        ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, mean[i], value[i])
        gradients(dmean[i], dvalue[i])
    grown = _heap_bytes() - before
    assert ppo.ppo_poll_status() == 0
    assert bool((mean == L.mean).all()) and bool((value == L.value).all())
    assert torch.equal(L.model.grad, want) and float(want.norm()) > 0
    assert grown < 64 * 1024, grown


# 48 outputs: behind 16, 32 and 48 channels, odd extents, rows of several segments, many small images, as the last layer
@pytest.mark.parametrize("H,W,N,conv", [(17, 22, 6, (16, 48, 32)), (35, 54, 4, (32, 48, 64)), (12, 530, 2, (16, 48)), (14, 18, 60, (48, 48, 16))])
def test_48_channels_from_halo_tiles_match_oracle(H, W, N, conv, monkeypatch):
    w = synth.Workload("c48", N, 2, H, W, conv, (3,) * len(conv), (40,), 1, 2, P=16, A=3)
    monkeypatch.setitem(NETS, "c48", w)
    conv_stack_matches_oracle("c48", monkeypatch)


# weight gradients in pairs of column tiles (148 SMs): 15 tiles of pixels per CTA (single) and 16 (pairs) with a ragged last one, the
# bias in a tile of its own, in a free block (192 inputs) and beside an empty tile (256), two groups of output columns (512)
@pytest.mark.parametrize("H,N,conv", [(64, 420, (32, 128, 128)), (64, 421, (32, 128, 128)), (32, 1290, (64, 192, 128)),
                                      (64, 215, (32, 128, 512)), (64, 850, (32, 64, 256, 256))])
def test_pairs_of_column_tiles_match_oracle(H, N, conv, monkeypatch):
    w = synth.Workload("cpairs", N, 1, H, H, conv, (3,) * len(conv), (40,), 1, 1, P=16, A=3)
    monkeypatch.setitem(NETS, "cpairs", w)
    conv_stack_matches_oracle("cpairs", monkeypatch)


# convolutions whose pixel tiles go in pairs: fewer tiles than SMs (147, single) and as many, odd numbers of tiles, rows of two tiles
# each, tiles of several images; 128, 192 (above) and 256 columns forward, 4 x 256 back
@pytest.mark.parametrize("H,W,N,conv", [(64, 64, 294, (32, 128, 128)), (64, 64, 296, (32, 128, 128)), (8, 532, 41, (64, 128)),
                                        (34, 30, 601, (64, 256, 256))])
def test_pairs_of_pixel_tiles_match_oracle(H, W, N, conv, monkeypatch):
    w = synth.Workload("ppairs", N, 1, H, W, conv, (3,) * len(conv), (40,), 1, 1, P=16, A=3)
    monkeypatch.setitem(NETS, "ppairs", w)
    conv_stack_matches_oracle("ppairs", monkeypatch)
