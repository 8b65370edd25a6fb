"""16-bit storage: what a population lacks is formed by the lane at its
sender's x and handed to the neighbouring lane; at warp edges and grid-row
ends it is formed for that receiver alone.  Rows shorter than, equal to and
longer than a warp, grids that end inside a warp, walls, both couplings and
odd species counts, one step from each streaming parity against the oracle.

The oracle steps the state as the library reports it (decoded by the readers,
which form each sender's terms directly), so one rounding lies between the
two: the stored part of each population, its post-collision value less the
sender's equilibrium and deferred terms, to the unit roundoff 2^-8 (BF16) or 2^-11 (FP16) of
itself, both taken from the oracle population by population, and FP32
arithmetic, 1e-5 of the lattice's largest population."""

import numpy as np
import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import TOL, gpu_handle, oracle_params

pytestmark = pytest.mark.gpu

C = np.array([[i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1] for i in range(27)], dtype=np.float64)


def _stored_part(pops, prm):
    """Post-collision populations, and the magnitude of what 16-bit storage holds of them."""
    post, a = O.collide(pops, prm, return_aux=True)
    M = prm.M
    part = post.copy()
    part[:M] -= a["feq_s"]
    part[M] -= a["feq"]
    part[M + 1] -= a["geq"]
    face = (np.abs(C).sum(axis=1) == 1)[:, None, None, None]
    part[M] -= 0.5 * face * np.einsum("id,d...->i...", C, a["Xc"])
    theta = a["R"] * a["T"]
    K = 0.5 * (2.0 - a["omega1"]) * a["P"] / theta * sum(prm.Cp_a[s] * a["T"] * a["gradY"][s] for s in range(M))
    w = np.prod([np.where(C[:, d][:, None, None, None] == 0, 1.0 - theta, 0.5 * theta) for d in range(3)], axis=0)
    part[M + 1] -= w * np.einsum("id,d...->i...", C, K)
    return post, np.abs(part)


@pytest.mark.parametrize("M,precision,shape,walls,coupling", [
    (2, "bf16", (3, 4, 1), False, "strong"), (2, "bf16", (2, 3, 2), False, "strong"),
    (2, "fp16", (3, 3, 31), False, "strong"), (2, "bf16", (2, 3, 32), False, "weak"),
    (3, "bf16", (2, 3, 33), False, "strong"), (3, "bf16", (2, 2, 70), True, "strong"),
    (3, "fp16", (3, 2, 11), True, "weak"), (1, "bf16", (2, 3, 129), False, "strong"),
    (5, "bf16", (3, 3, 33), False, "strong"), (8, "fp16", (2, 3, 11), False, "weak"), (4, "bf16", (2, 2, 35), True, "strong"),
    # more nodes than the small-grid line of two and three species
    (2, "bf16", (15, 31, 33), False, "strong"), (3, "fp16", (16, 31, 31), True, "strong"),
])
def test_row_exchange(M, precision, shape, walls, coupling):
    wl = W.random_mixture(M=M, shape=shape, seed=11 + M, velocity=0.02)
    prm = oracle_params(wl, coupling=coupling, walls_x=walls)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    pops = pops * W.perturbation(pops.shape, 0.01, 3)
    h = gpu_handle(wl, precision, coupling=coupling, walls_x=walls)
    h.set_populations(pops)
    unit = 2.0 ** (-8 if precision == "bf16" else -11)
    for _ in range(2):
        post, part = _stored_part(h.populations(), prm)
        h.step(1)
        err = np.abs(h.populations() - O.stream(post, walls))
        tol = unit * O.stream(part, walls)
        for L in range(M + 2):
            assert (err[L] <= tol[L] + TOL["fp32"] * np.abs(post[L]).max()).all(), L
    h.close()
