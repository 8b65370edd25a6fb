"""Populations read from 16-bit storage are the sum, in FP64, of the rest
equilibrium, the stored part, the shift and the deferred terms c . X / 2 (f, face
velocities) and w(theta) c . K (g).  The deferred terms of a stepped state are
taken out of the scratch planes and the populations read again: the difference
is the terms themselves, not their rounding against the shift.

Tolerances: a term of f is an FP32 value, and two FP64 sums are rounded to
2^-53 of the population each (four units allowed); a term of g adds its own
FP32 products, five roundings of 2^-24 (2^-21 of the sum of magnitudes)."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import gpu_handle

pytestmark = pytest.mark.gpu

SP_K, SP_THR, SP_X = 10, 13, 14
C = np.array([[i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1] for i in range(27)])


@pytest.mark.parametrize("M,precision,shape,steps", [(2, "bf16", (3, 4, 11), 3), (3, "fp16", (4, 3, 33), 2), (8, "bf16", (2, 3, 40), 3)])
def test_deferred_terms_are_added_in_fp64(M, precision, shape, steps):
    import torch
    wl = W.random_mixture(M=M, shape=shape, seed=15 + M, velocity=0.02)
    h = gpu_handle(wl, precision)
    h.init_fields(wl.X, wl.u, wl.T, wl.P)
    h.step(steps)
    N = wl.nodes
    with_terms = h.populations()
    h.synchronize()
    planes = h.scratch_buf[: 20 * N * 4].view(torch.float32).view(20, N)
    side = planes.cpu().numpy().astype(np.float64).reshape((20,) + shape)
    planes[SP_X:SP_X + 3] = 0
    planes[SP_K:SP_K + 3] = 0
    torch.cuda.synchronize()
    without = h.populations()
    X, K, th = side[SP_X:SP_X + 3], side[SP_K:SP_K + 3], side[SP_THR]
    assert np.abs(X).max() > 0 and np.abs(K).max() > 0
    for i, c in enumerate(C):
        at = lambda a: np.roll(a, (c[2], c[1], c[0]), axis=(-3, -2, -1))     # of the sender n - c
        eps = 4 * 2.0 ** -53 * np.abs(with_terms[:, i])
        diff = with_terms[:, i] - without[:, i]
        assert (diff[:M] == 0).all()
        f = 0.5 * sum(c[d] * at(X[d]) for d in range(3)) if np.abs(c).sum() == 1 else np.zeros(shape)
        assert (np.abs(diff[M] - f) <= eps[M]).all(), i
        w = np.prod([np.where(c[d] == 0, 1.0 - at(th), 0.5 * at(th)) for d in range(3)], axis=0)
        terms = [w * c[d] * at(K[d]) for d in range(3)]
        assert (np.abs(diff[M + 1] - sum(terms)) <= eps[M + 1] + 2.0 ** -21 * sum(np.abs(t) for t in terms)).all(), i
    h.close()
