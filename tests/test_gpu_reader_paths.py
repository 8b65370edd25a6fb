"""The readers of 16-bit states form a sender's terms by rows and exchange them
between lanes; the conservation sums gather every sender's record for itself,
in another form of the same equations.  Grid totals of the two agree: each
node's 27 deviations are summed in FP32 (27 roundings of 2^-24 of values no
larger than the node's density, in both), and the form of the shift is good to
FP32 rounding of its dozen operations: 2 (27 + 12) 2^-24 < 5e-6 of the total
density."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import gpu_handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision,shape,walls", [(2, "bf16", (3, 5, 33), False), (3, "fp16", (4, 3, 11), True),
                                                     (5, "bf16", (2, 3, 70), False), (8, "fp16", (3, 3, 45), True)])
def test_moments_against_diagnostics(M, precision, shape, walls):
    wl = W.random_mixture(M=M, shape=shape, seed=60 + M, velocity=0.03)
    slaved = W.slaved_species(wl)
    h = gpu_handle(wl, precision, walls_x=walls)
    h.init_fields(wl.X, wl.u, wl.T, wl.P)
    for n in (3, 1):
        h.step(n)
        m, s = h.moments_dict(), h.diagnostics()
        total = m["rho"].sum()
        for a in range(M):
            if a != slaved:
                assert abs((m["Y"][a] * m["rho"]).sum() - s[a]) < 5e-6 * total, a
        assert abs(total - s[M]) < 5e-6 * total
        for d in range(3):
            assert abs((m["rho"] * m["u"][d]).sum() - s[M + 1 + d]) < 5e-6 * total, d
    h.close()
