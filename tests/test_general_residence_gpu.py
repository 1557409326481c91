"""The general plan's field wherever it lives: on the device, there off the
8-byte boundary that the kernels read it at, and on the host; the same bits.
(A field on another device goes through a copy as host fields do; one device
cannot show it.)"""
import ctypes

import numpy as np
import pytest
import torch

import paper_1705_06284_gb300 as fbs
from test_general_gpu import _edges, _field

pytestmark = pytest.mark.gpu


def test_same_bits_from_anywhere():
    shape, Ls = (18, 32, 24), (10.0, 12.0, 11.0)
    f = _field(shape, "complex", 53).astype(np.complex64)
    with fbs.GeneralPlan(shape, Ls, _edges(shape, Ls, 3)) as plan:
        B, P = plan.bispectrum(f)
        flat = torch.from_numpy(f.view(np.float32).ravel())
        room = torch.zeros(flat.numel() + 1, device="cuda")
        for off in (0, 1):
            room[off:off + flat.numel()] = flat.cuda()
            torch.cuda.synchronize()
            b, p = np.zeros(2 * plan.ntrip), np.zeros(2 * plan.nbins)
            at = ctypes.c_void_p(room.data_ptr() + 4 * off)
            assert fbs.lib().fbs_gplan_bispectrum(ctypes.c_void_p(plan._h), at, ctypes.c_void_p(b.ctypes.data),
                                                  ctypes.c_void_p(p.ctypes.data)) == 0
            assert np.array_equal(b.view(np.complex128), B) and np.array_equal(p.view(np.complex128), P, equal_nan=True)
