"""Max-pooling for the window sizes with a kernel of their own (2, 3) and others,
overlapping and apart, with NaN (ignored unless a window holds nothing else),
infinities and both zeros."""
import numpy as np
import pytest
import torch

import paper_1512_06473_gb300 as q
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,C,H,W,k,s", [
    (1, 1, 1, 1, 1, 1), (2, 3, 2, 2, 2, 2), (1, 5, 7, 9, 2, 1), (3, 33, 13, 13, 3, 2),
    (2, 7, 11, 6, 3, 3), (1, 2, 9, 9, 3, 5), (2, 4, 12, 10, 4, 2), (1, 3, 9, 8, 5, 3),
])
def test_windows(N, C, H, W, k, s):
    x = synth.normal((N, C, H, W), 1.0, 60 + k).ravel()
    x[::5], x[1::7], x[2::11], x[3::13] = np.nan, np.inf, -np.inf, 0.0
    x = x.reshape(N, C, H, W)
    y = q.maxpool(torch.from_numpy(x).cuda(), k, s).cpu().numpy()
    win = np.lib.stride_tricks.sliding_window_view(x, (k, k), (2, 3))[:, :, ::s, ::s]
    ref = np.fmax.reduce(win.reshape(*win.shape[:4], k * k), axis=-1)
    assert np.array_equal(y, ref, equal_nan=True)
