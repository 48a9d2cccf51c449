"""The probe of the packed pair loop (libbldtt_pipes.so) returns plausible rates: at
most the MUFU unit's (one rsqrt an evaluation, 16 a clock and SM; Yukawa an exp2
more, 32), and within a factor of two of it."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2012_06925_gb300 import build as builder

pytestmark = pytest.mark.gpu


def test_pair_loop_rates():
    lib = ctypes.CDLL(builder.build_pipes())
    out = np.zeros(2)
    s = torch.cuda.current_stream()
    rc = lib.pipes_pair_loop(out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), ctypes.c_void_p(s.cuda_stream))
    assert rc == 0
    print("evaluations per clock and SM: Coulomb %.2f, Yukawa %.2f" % tuple(out))
    assert 8.0 <= out[0] <= 16.2 and 5.0 <= out[1] <= 10.8
