"""A node's result does not depend on which lane of which warp computes it.
With 16-bit storage a sender's terms are formed by the lane at its x and handed
on, or, at warp edges and ends of grid rows, for one receiver alone; both must
give the same bits.  Two consequences, on grids whose rows and planes are no
multiples of a warp: a state uniform in y and z stays so, and slabs (which
shift every node's place) reproduce the undivided grid."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import binding, workloads as W
from paper_2004_11286_gb300.slabs import SlabSet, reference_state

from gpu_helpers import gpu_handle

pytestmark = pytest.mark.gpu

CASES = [(1, "fp16", 13, False), (2, "bf16", 11, False), (2, "fp16", 33, True), (3, "bf16", 33, False),
         (3, "fp16", 11, True), (4, "bf16", 70, True), (5, "fp16", 33, False), (8, "bf16", 11, False), (8, "fp16", 45, True),
         (2, "fp32", 33, False), (4, "fp64", 11, True)]


@pytest.mark.parametrize("M,precision,nx,walls", CASES)
def test_uniform_in_y_and_z_stays_uniform(M, precision, nx, walls):
    wl = W.random_mixture(M=M, shape=(3, 5, nx), seed=30 + M, velocity=0.02)
    line = lambda a: np.ascontiguousarray(np.broadcast_to(a[..., :1, :1, :], a.shape))
    h = gpu_handle(wl, precision, walls_x=walls)
    h.init_fields(line(wl.X), line(wl.u), line(wl.T), line(wl.P))
    for n in (1, 1, 9):
        h.step(n)
        p = h.populations()
        # velocity by velocity: a population that moves in y or z stays with its own line
        assert np.array_equal(p, np.broadcast_to(p[..., :1, :1, :], p.shape))
        m = h.moments_dict()
        for k in ("rho", "u", "T", "X"):
            assert np.array_equal(m[k], np.broadcast_to(m[k][..., :1, :1, :], m[k].shape)), k
    h.close()


@pytest.mark.parametrize("M,precision,nx,walls", CASES)
def test_slabs_shift_no_bit(M, precision, nx, walls):
    wl = W.random_mixture(M=M, shape=(11, 5, nx), seed=70 + M, velocity=0.02)
    Y, T, rho = reference_state(wl.X, wl.T, wl.P, wl.molar_mass, wl.R_U)
    one = gpu_handle(wl, precision, walls_x=walls)
    one.set_reference(Y, T, rho)
    one.init_fields(wl.X, wl.u, wl.T, wl.P)

    def make(shape, dev):
        return binding.LbmMix(wl.molar_mass, wl.cv_molar, wl.D, mu=wl.mu, lam=wl.lam, shape=shape, precision=precision,
                              slaved=W.slaved_species(wl), R_U=wl.R_U, walls_x=walls, device=dev)

    slabs = SlabSet(make, wl.shape, 2, wl.molar_mass, wl.cv_molar, wl.R_U, slaved=W.slaved_species(wl))
    slabs.init_fields(wl.X, wl.u, wl.T, wl.P)
    for n in (1, 8):
        one.step(n)
        slabs.step(n)
        a, b = slabs.populations(), one.populations()
        assert np.array_equal(a, b), float(np.abs(a - b).max())
    ma, mb = slabs.moments_dict(), one.moments_dict()
    for k in ("rho", "u", "T", "P", "X"):
        assert np.array_equal(ma[k], mb[k]), k
    one.close()
    slabs.close()
