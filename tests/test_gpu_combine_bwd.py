"""Backward of the combine with the gate's backward in it: one or two slots a token (rows of fewer vectors than a piece, of one, of several,
ragged), up to eight, more than one pass of eight; against the oracle."""
import pytest

from oracle import margin
from paper_2502_16927_b200 import workloads as wl

import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bf16,r,k,capacity", [(True, 64, 1, 0.0), (True, 320, 2, 0.8), (True, 576, 1, 0.0), (True, 1088, 2, 0.0), (True, 192, 9, 0.0),
                                               (False, 36, 1, 0.0), (False, 300, 2, 0.7), (False, 128, 8, 0.0), (False, 140, 10, 0.8)])
def test_slots_a_token_and_row_lengths(bf16, r, k, capacity):
    w = wl.Workload("cb", T=333, d=128, r=r, h=64, E=12, k=k, dtype=wl.DTYPE_BF16 if bf16 else wl.DTYPE_F32, act=wl.ACT_GELU_ERF, seed=600 + r)
    inp = wl.make_inputs(w)
    margin.enforce_margin(w, inp, 1e-3)
    parity.compare_full(w, inp, parity.run_full(w, inp, capacity_factor=capacity), capacity_factor=capacity)
