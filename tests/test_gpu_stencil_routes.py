"""The stencil passes on either side of their size line: a thread per node and
field on small grids, four nodes of a row per thread or (rows of no multiple
of four) one node per thread beyond, against the oracle after three steps
(the third uses both passes' terms of the first two).

Tolerances are the precision contract's, of the largest population."""

import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import TOL, gpu_handle, oracle_params, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shape,walls", [
    ("fp32", (32, 32, 32), False), ("fp32", (32, 33, 32), False), ("fp32", (32, 32, 33), True), ("fp32", (31, 33, 36), True),
    ("fp64", (32, 64, 64), False), ("fp64", (32, 65, 64), False), ("fp64", (32, 64, 65), True),
])
def test_stencil_routes(precision, shape, walls):
    wl = W.random_mixture(M=1, shape=shape, seed=5, velocity=0.03)
    prm = oracle_params(wl, walls_x=walls)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    h = gpu_handle(wl, precision, walls_x=walls)
    h.set_populations(pops)
    h.step(3)
    got, ref = h.populations(), O.run(pops, prm, 3)
    for L in range(3):
        assert rel(got[L], ref[L]) < TOL[precision], L
    h.close()
