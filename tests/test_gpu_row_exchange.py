"""16-bit storage: what a population lacks is formed by the lane at its
sender's x and handed to the neighbouring lane; at warp edges and grid-row
ends it is formed for that receiver alone.  Rows shorter than, equal to and
longer than a warp, grids that end inside a warp, walls, both couplings and
odd species counts, two steps (both streaming parities) against the oracle.

Tolerance: the state's non-equilibrium part is at most 2 % of a population
(1 % noise, and the first step's relaxation), stored with a relative rounding
of 2^-9 (BF16) in each of two steps: 8e-5 of the largest population; 2e-4
allowed.  A wrong sender would be off by its equilibrium's difference, which
the composition's 50 % modes make 1e-2 and more."""

import numpy as np
import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import gpu_handle, oracle_params, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision,shape,walls,coupling", [
    (2, "bf16", (3, 4, 1), False, "strong"), (2, "bf16", (2, 3, 2), False, "strong"),
    (2, "fp16", (3, 3, 31), False, "strong"), (2, "bf16", (2, 3, 32), False, "weak"),
    (3, "bf16", (2, 3, 33), False, "strong"), (3, "bf16", (2, 2, 70), True, "strong"),
    (3, "fp16", (3, 2, 11), True, "weak"), (1, "bf16", (2, 3, 129), False, "strong"),
    (5, "bf16", (3, 3, 33), False, "strong"), (8, "fp16", (2, 3, 11), False, "weak"), (4, "bf16", (2, 2, 35), True, "strong"),
])
def test_row_exchange(M, precision, shape, walls, coupling):
    wl = W.random_mixture(M=M, shape=shape, seed=11 + M, velocity=0.02)
    prm = oracle_params(wl, coupling=coupling, walls_x=walls)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    pops = pops * W.perturbation(pops.shape, 0.01, 3)
    h = gpu_handle(wl, precision, coupling=coupling, walls_x=walls)
    h.set_populations(pops)
    h.step(2)
    got, ref = h.populations(), O.run(pops, prm, 2)
    for L in range(M + 2):
        assert rel(got[L], ref[L]) < 2e-4, L
    h.close()
