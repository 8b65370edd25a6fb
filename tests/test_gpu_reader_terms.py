"""Populations read from 16-bit storage are the sum, in FP64, of the rest
equilibrium, the stored part, the shift and the deferred terms c . X / 2 (f, face
velocities) and w(theta) c . K (g).  X and K of a stepped state are replaced by
powers of two far below the FP32 resolution of the shift (2^-40, 2^-30) and by
zero: the two readings must differ by the terms themselves.

Bounds: every sum has at most four FP64 roundings, of values up to the largest
population (or 1); a term of g also has the FP32 roundings of its products,
2^-21 of the sum of magnitudes."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import gpu_handle

pytestmark = pytest.mark.gpu

SP_K, SP_THR, SP_X = 10, 13, 14
C = np.array([[i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1] for i in range(27)])


@pytest.mark.parametrize("M,precision,shape,steps", [(2, "bf16", (3, 4, 11), 3), (3, "fp16", (4, 3, 33), 2), (8, "bf16", (3, 3, 40), 3)])
def test_deferred_terms_are_added_in_fp64(M, precision, shape, steps):
    import torch
    wl = W.random_mixture(M=M, shape=shape, seed=15 + M, velocity=0.02)
    h = gpu_handle(wl, precision)
    h.init_fields(wl.X, wl.u, wl.T, wl.P)
    h.step(steps)
    h.synchronize()
    planes = h.scratch_buf[: 20 * wl.nodes * 4].view(torch.float32).view(20, wl.nodes)
    th = planes[SP_THR].cpu().numpy().astype(np.float64).reshape(shape)
    X, K = 2.0 ** -40 * np.array([1, 2, 4]), 2.0 ** -30 * np.array([1, 2, 4])
    read = []
    for on in (0.0, 1.0):
        for d in range(3):
            planes[SP_X + d] = on * float(X[d])
            planes[SP_K + d] = on * float(K[d])
        torch.cuda.synchronize()
        read.append(h.populations())
    diff = read[1] - read[0]
    eps = 4 * 2.0 ** -53 * max(1.0, float(np.abs(read[0]).max()))
    assert (diff[:M] == 0).all()
    for i, c in enumerate(C):
        th_s = np.roll(th, (c[2], c[1], c[0]), axis=(0, 1, 2))                       # of the sender n - c
        f = 0.5 * float(c @ X) if np.abs(c).sum() == 1 else 0.0
        assert np.abs(diff[M, i] - f).max() <= 2 * eps, i
        w = np.prod([np.where(c[d] == 0, 1.0 - th_s, 0.5 * th_s) for d in range(3)], axis=0)
        tol = 2 * eps + 2.0 ** -21 * w * float(np.abs(c) @ K)
        assert (np.abs(diff[M + 1, i] - w * float(c @ K)) <= tol).all(), i
    h.close()
