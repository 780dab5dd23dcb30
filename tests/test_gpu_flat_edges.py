"""Fully connected layers at the edges of their tiles (rows and columns that no tile width divides, reductions that are no whole
number of chunks)."""
import pytest

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
