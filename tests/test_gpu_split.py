"""The collide whose warps share out a node's lattices, against the oracle:
every species count it is built for (two and three on small grids; grids past
that line, with a thread per node, are held to the same), grids that end inside a 32-node tile or
fill none, walls, both couplings, and the FP64 re-solve of ill-conditioned
systems (a condition bound of 1 sends every node there).

Tolerances are the precision contract's: 1e-12 (FP64), 1e-5 (FP32) of the
largest population, lattice by lattice."""

import numpy as np
import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import TOL, gpu_handle, oracle_params, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision,shape,kw", [
    (4, "fp32", (1, 1, 5), {}), (4, "fp64", (3, 4, 5), {}), (5, "fp32", (3, 4, 11), {}), (5, "fp64", (2, 3, 7), {"coupling": "weak"}),
    (6, "fp32", (2, 4, 8), {"coupling": "weak"}), (6, "fp64", (1, 3, 33), {"walls_x": True}),
    (7, "fp32", (3, 3, 13), {"walls_x": True}), (8, "fp32", (4, 4, 9), {}), (8, "fp64", (2, 3, 9), {}),
    (4, "fp32", (3, 4, 5), {"fp64_cond_bound": 1.0}), (7, "fp32", (3, 4, 5), {"fp64_cond_bound": 1.0}),
    (8, "fp32", (3, 4, 5), {"fp64_cond_bound": 1.0, "coupling": "weak"}),
    (4, "fp32", (3, 4, 5), {"omega_fixed": 1.2, "omega1_fixed": 0.9}),
    (2, "fp64", (3, 5, 7), {"coupling": "weak"}), (3, "fp32", (2, 3, 35), {"coupling": "weak"}), (3, "fp64", (1, 2, 40), {"walls_x": True}),
    (3, "fp32", (3, 4, 5), {"fp64_cond_bound": 1.0}),
    # past the small-grid lines: 6144 nodes in FP64, 15,600 in FP32
    (2, "fp64", (12, 16, 32), {}), (3, "fp64", (12, 16, 32), {"walls_x": True}), (3, "fp64", (12, 17, 33), {"coupling": "weak"}),
    (3, "fp32", (24, 25, 26), {}), (3, "fp32", (24, 25, 26), {"walls_x": True, "coupling": "weak"}),
])
def test_split_collide(M, precision, shape, kw):
    wl = W.random_mixture(M=M, shape=shape, seed=20 + M, velocity=0.03)
    okw = {k: v for k, v in kw.items() if k != "fp64_cond_bound"}
    prm = oracle_params(wl, **okw)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    pops = pops * W.perturbation(pops.shape, 0.01, 4)
    h = gpu_handle(wl, precision, **kw)
    h.set_populations(pops)
    h.step(3)
    got, ref = h.populations(), O.run(pops, prm, 3)
    for L in range(M + 2):
        assert rel(got[L], ref[L]) < TOL[precision], L
    h.close()
