"""A network that is rejected at every node against the exact step, from four
species with 16-bit storage.  There the exact step takes the split collide and
the network's a thread per node: the same equations in another order.  After a
step from one state each stored part is the 16-bit rounding of values that
differ by FP32 arithmetic, so the two differ by at most one unit in the last
place of the stored part (two unit roundoffs, 2^-8 BF16 and 2^-11 FP16, of its
magnitude) and FP32 arithmetic of each (1e-5 of the lattice's largest
population)."""

import numpy as np
import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import TOL, gpu_handle, oracle_params
from test_gpu_row_exchange import _stored_part

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision", [(4, "bf16"), (5, "fp16"), (8, "bf16")])
def test_rejected_network_agrees_to_one_unit_of_the_stored_part(M, precision):
    wl = W.random_mixture(M=M, shape=(5, 6, 7), seed=21 + M, velocity=0.03)
    prm = oracle_params(wl)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm) * W.perturbation((M + 2, 27) + wl.shape, 0.01, 3)
    ha = gpu_handle(wl, precision)
    hb = gpu_handle(wl, precision, closure="mlp", closure_bound=1e-30)
    ha.set_populations(pops)
    hb.set_populations(pops)
    post, part = _stored_part(ha.populations(), prm)
    ha.step(1)
    hb.step(1)
    a, b = ha.populations(), hb.populations()
    unit = 2.0 ** (-8 if precision == "bf16" else -11)
    tol = 2 * unit * O.stream(part, False)
    for L in range(M + 2):
        assert (np.abs(a[L] - b[L]) <= tol[L] + 2 * TOL["fp32"] * np.abs(post[L]).max()).all(), L
    print(M, precision, "largest difference of the largest population: %.2e" % (np.abs(a - b).max() / np.abs(a).max()))
    assert hb.closure_stats() == (0, wl.nodes)
    ha.close()
    hb.close()
