"""Slabs smaller than the size lines by which the step chooses its kernels, cut
from grids above them: the undivided grid and the slabs take different stencil
passes (whose sums are the same operation by operation) and would take
different collides (the slabs know the whole grid's size), and the interiors
must agree bit for bit.  The stencil lines are 32,768 nodes (FP32 fields) and
131,072 (FP64) with rows of a multiple of four, 24,576 with others; the collide
lines, in nodes an SM: 32 (FP64, two and three species), and in FP32 96 (three
and five species) and 384 (four)."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import binding, workloads as W
from paper_2004_11286_gb300.slabs import SlabSet, reference_state

from gpu_helpers import gpu_handle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision,shape,walls", [
    # stencils: rows of a multiple of four, and not
    (2, "fp32", (64, 32, 32), False), (2, "fp32", (64, 32, 33), True), (1, "fp64", (64, 64, 64), True),
    (1, "fp64", (64, 27, 37), False), (2, "bf16", (64, 32, 36), False),
    # collides
    (2, "fp64", (24, 16, 16), False), (3, "fp64", (24, 17, 15), True), (3, "fp32", (48, 20, 20), False),
    (4, "fp32", (64, 32, 31), False), (4, "fp32", (16, 32, 128), False), (5, "fp32", (24, 28, 28), False),
])
def test_slabs_on_the_other_side_of_a_size_line(M, precision, shape, walls):
    wl = W.random_mixture(M=M, shape=shape, seed=90 + M, velocity=0.02)
    Y, T, rho = reference_state(wl.X, wl.T, wl.P, wl.molar_mass, wl.R_U)
    one = gpu_handle(wl, precision, walls_x=walls)
    one.set_reference(Y, T, rho)
    one.init_fields(wl.X, wl.u, wl.T, wl.P)

    def make(s, dev):
        return binding.LbmMix(wl.molar_mass, wl.cv_molar, wl.D, mu=wl.mu, lam=wl.lam, shape=s, precision=precision,
                              slaved=W.slaved_species(wl), R_U=wl.R_U, walls_x=walls, device=dev)

    slabs = SlabSet(make, wl.shape, 4, wl.molar_mass, wl.cv_molar, wl.R_U, slaved=W.slaved_species(wl))
    slabs.init_fields(wl.X, wl.u, wl.T, wl.P)
    for n in (1, 4):
        one.step(n)
        slabs.step(n)
        a, b = slabs.populations(), one.populations()
        assert np.array_equal(a, b), float(np.abs(a - b).max())
    one.close()
    slabs.close()


def test_grid_nodes_arguments():
    wl = W.random_mixture(M=2, shape=(3, 4, 5), seed=1)
    h = gpu_handle(wl, "fp32")
    with pytest.raises(binding.LbmError) as e:
        h.set_grid_nodes(-1)
    assert e.value.status == 1
    h.set_grid_nodes(10 ** 9)
    h.set_grid_nodes(0)
    h.close()
    b = binding.LbmBatch([binding.workload_params(wl, precision="fp32")])
    with pytest.raises(binding.LbmError) as e:
        b.domain(0).set_grid_nodes(100)
    assert e.value.status == 6
    b.close()
