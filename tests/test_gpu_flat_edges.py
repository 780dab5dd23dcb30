"""Fully connected layers at the edges of their tiles (rows and columns that no tile width divides, reductions that are no whole
number of chunks), and the gates of the last convolution."""
import ctypes as C

import numpy as np
import pytest
import torch

import test_gpu_learner as base
from helpers import rel_l2
from paper_2509_16434_b200 import binding as ppo
from paper_2509_16434_b200 import synth
from test_gpu_conv_edges import NETS, test_conv_stack_matches_oracle as conv_stack_matches_oracle

pytestmark = pytest.mark.gpu


def _all_rows_match_oracle(w):
    """The forward of a whole minibatch in one call, row by row: a row is within the encoder's tolerance of itself, or of a row of
    average size where it is smaller."""
    B = w.M // w.minibatches
    L, md, lay, theta, roll, action, logp, dev = base._setup(w, B, theta_scale_head=20.0)
    L.compute_gae(dev["last_value"])
    f, _, _, mu_o, V_o = base._oracle_minibatch(md, lay, theta, roll, action, logp, w, L.hyper, 5, 0, 0, w.minibatches)
    ppo.ppo_shuffle_gather_minibatch(L.buffer, 5, 0, 0, w.minibatches, L.mb)
    L.mean.fill_(-9.0)
    L.value.fill_(-9.0)
    ppo.ppo_encoder_fwd(L.model, L.mb, 0, B, L.mean, L.value)
    assert ppo.ppo_poll_status() == 0
    got = np.concatenate([L.mean[:B].cpu().numpy(), L.value[:B, None].cpu().numpy()], 1).astype(np.float64)
    want = np.concatenate([mu_o, np.asarray(V_o).reshape(-1, 1)], 1)
    norm = np.linalg.norm(want, axis=1)
    err = np.linalg.norm(got - want, axis=1) / np.maximum(norm, np.sqrt(np.mean(norm ** 2)))
    print(f"rows of {B}: largest error {err.max():.2e}")
    assert err.max() <= base.ENC_TOL, int(err.argmax())


# minibatches of 1, 33, 129 and 300 rows: one row, one past a tile of 32, one past a tile of 128, many ragged tiles; widths that are
# no multiple of 16 or 32, a first layer of 48 + 8 (one ragged chunk) and 64 + 64 columns (two whole chunks)
@pytest.mark.parametrize("N,T,fc,P,last,embed", [
    (2, 1, (40,), 8, 48, 0), (6, 11, (200, 120), 8, 48, 0), (6, 43, (72, 504, 24), 64, 64, 0), (60, 10, (200, 120), 16, 32, 0),
    (6, 11, (128, 56), 16, 32, 32), (6, 43, (200,), 8, 64, 64), (60, 10, (64, 64), 16, 32, 96)])
def test_forward_and_gradients_match_oracle(N, T, fc, P, last, embed, monkeypatch):
    w = synth.Workload("flat", N, T, 16, 24, (16, last), (3, 3), fc, 1, 2, P=P, A=3, embed=embed)
    monkeypatch.setitem(NETS, "flat", w)
    conv_stack_matches_oracle("flat", monkeypatch)  # outputs and every gradient tensor within 2e-2
    _all_rows_match_oracle(w)


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
CHAIN_LINES = [(33, (120, 200, 120)), (480, (72, 40)), (481, (200, 120)), (961, (72, 504)), (1921, (960,)), (1921, (968,)), (4224, (40,)),
               (4225, (40,))]


@pytest.mark.parametrize("B,fc", CHAIN_LINES)
def test_dense_chain_at_its_lines_matches_oracle(B, fc, monkeypatch):
    w = synth.Workload("chain", 2 * B, 1, 8, 12, (16, 32), (3, 3), fc, 1, 2, P=40, A=3)
    monkeypatch.setitem(NETS, "chain", w)
    conv_stack_matches_oracle("chain", monkeypatch)
    _all_rows_match_oracle(w)


# (widths that the chain takes: a layer reads 64 values or more)
@pytest.mark.parametrize("B,fc", [(1, (72,)), (33, (120, 200, 120)), (480, (72, 72)), (481, (200, 120)), (960, (504, 72)), (961, (72, 504)), (1920, (120,)),
                                  (1921, (960,)), (1921, (968,)), (4224, (64,)), (4225, (64,))])
def test_dense_chain_gives_the_bits_of_single_layers(B, fc):
    """B rows in one call against the same rows among 4226, which no chain takes, and (forward) in pieces of 480, which clusters of
    eight take: outputs and hidden layers are the same bits.  Back, only the rows of the last tile of 32 carry a gradient, so that
    none of it can be lost in the rest; the input gradients are the same bits, and the weight gradients sum the same terms (at most 32
    rows x 24 pixels) in other groups: 768 roundings of 2^-24 are 4.6e-5 of the sum of their sizes."""
    R = 4226
    w = synth.Workload("bits", R, 1, 8, 12, (16, 32), (3, 3), fc, 1, 1, P=40, A=3)
    L = base.Learner(w, R, "cuda")
    shapes, gammas = synth.param_shapes(w)
    L.model.load(synth.init_params(L.model.arena, [o for o, _ in L.model.tensors()], shapes, 3, ones=gammas))
    r = synth.rollout_torch(w, "cuda", 3)
    rows = ppo.Minibatch(r["depth"].data_ptr(), r["proprio"].data_ptr(), None, None, None, None, None, None, R)
    g = torch.Generator("cuda").manual_seed(4)
    first = (B - 1) // 32 * 32
    dmean, dvalue = torch.zeros((R, 3), device="cuda"), torch.zeros(R, device="cuda")
    dmean[first:B] = torch.randn((B - first, 3), device="cuda", generator=g)
    dvalue[first:B] = torch.randn(B - first, device="cuda", generator=g)

    def run(n):
        L.mean.fill_(-9.0)
        L.value.fill_(-9.0)
        ppo.ppo_encoder_fwd(L.model, rows, 0, n, L.mean, L.value)
        out = [L.mean.clone(), L.value.clone()] + [L.model.activation(1, l)[:B * k].clone() for l, k in enumerate([72] + list(fc))]
        ppo.ppo_model_zero_grad(L.model)
        ppo.ppo_encoder_bwd(L.model, rows, 0, n, dmean, dvalue, True)
        return out, L.model.grad.clone()

    (mean, value, *hidden), grad = run(B)
    (mean_all, value_all, *hidden_all), grad_all = run(R)
    assert bool((mean[B:] == -9.0).all()) and bool((value[B:] == -9.0).all())
    assert torch.equal(mean[:B], mean_all[:B]) and torch.equal(value[:B], value_all[:B])
    assert all(torch.equal(a, b) for a, b in zip(hidden, hidden_all))
    for r0 in range(0, B, 480):
        n = min(480, B - r0)
        ppo.ppo_encoder_fwd(L.model, rows, r0, n, L.mean, L.value)
        assert torch.equal(L.mean[:n], mean[r0:r0 + n]) and torch.equal(L.value[:n], value[r0:r0 + n])
    assert ppo.ppo_poll_status() == 0
    errs = [rel_l2(grad[o:o + s].cpu().numpy(), grad_all[o:o + s].cpu().numpy()) for o, s in L.model.tensors()[:-1]]
    print(f"gradients of rows {first} to {B}: largest difference {max(errs):.1e}")
    assert float(grad.norm()) > 0 and max(errs) <= 5e-5


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
