"""A training step that cannot be launched leaves the update count alone.  Here
nothing can: without a GPU the first call of the runtime fails.  (Host pointers
stand in for device buffers, so the test runs only where no GPU is.)"""
import ctypes
import os

import numpy as np
import pytest
import torch

from paper_2508_11790_gb300 import learned as LR


@pytest.mark.skipif(torch.cuda.is_available() or os.path.exists("/dev/nvidiactl"), reason="needs a machine without a GPU")
@pytest.mark.parametrize("H", [8, 300])
def test_failed_step_is_not_counted(H):
    L = LR._lib()
    n = int(L.bs_mlp_param_count(4, H, 2))
    f = [np.zeros(n, np.float32) for _ in range(5)]
    a = [np.zeros(16 * H, np.float32) for _ in range(8)]
    X, T = np.zeros(64, np.float32), np.zeros(32, np.float32)
    p = lambda v: v.ctypes.data
    m = LR._Mlp(4, H, 2, 7, *[p(v) for v in f])
    w = LR._Work(16, *[p(v) for v in a])
    assert L.bs_mlp_train_step(ctypes.byref(m), p(X), p(T), 16, ctypes.byref(w), 1e-3, None, None) != 0
    assert m.step == 7
