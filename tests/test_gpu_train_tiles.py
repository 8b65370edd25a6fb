"""The training gradient at the edges of its row tiles: 16-row tiles up to
one tile per SM, 32-row tiles beyond, ragged last tiles, several tiles per
block, and each padded (features, outputs) size the kernels are built for.

Tolerance: the kernels sum at most a few hundred products in a row (a tile's
rows, the layer widths, the blocks' partials), so the rounding is below
300 * 2^-24 = 1.8e-5 of the terms' absolute sum; 1e-4 of the largest entry
allows for a cancellation of five."""

import numpy as np
import pytest

from oracle import closure as CL
from paper_2004_11286_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,n", [(8, 1), (8, 15), (8, 17), (8, 2432), (8, 2433), (8, 6000), (2, 33), (4, 47), (6, 95)])
def test_gradient_row_tiles(M, n):
    import torch
    from paper_2004_11286_gb300 import binding
    F, Out, _ = CL.closure_dims(M)
    wl = W.random_mixture(M=M, shape=(2, 2, 2), seed=7)
    h = binding.from_workload(wl)
    w = W.closure_initial_weights(M, seed=n)
    h.set_closure_weights(w)
    rng = np.random.Generator(np.random.PCG64(n))
    x = rng.uniform(-1, 1, (n, F)).astype(np.float32)
    t = rng.uniform(-1, 1, (n, Out)).astype(np.float32)
    loss, g = h.closure_loss_grad(torch.as_tensor(x, device="cuda"), torch.as_tensor(t, device="cuda"))
    w64, x64, t64 = (a.astype(np.float64) for a in (w, x, t))
    assert abs(loss - CL.loss(w64, x64, t64, M)) <= 1e-5 * loss
    for a, b in zip(CL.unpack(g.cpu().numpy(), M), CL.unpack(CL.gradients(w64, x64, t64, M), M)):
        assert np.abs(a - b).max() <= 1e-4 * max(np.abs(b).max(), 1e-12)
    h.close()
