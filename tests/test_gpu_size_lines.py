"""Kernels that only grids beyond the step's size lines reach, against the
oracle: the per-node and row-blocked stencils with variable heats and with the
opposed-jets frame (more than 32,768 nodes in FP32, 65,536 in FP64 and 24,576
where rows are no multiple of four), the frame of the collide with a thread per
node (grids beyond the split collide's line), that collide from four species
(small grids that are told they are a slab of a large one), and the split collide's blocks at their second and later tiles
(more 32-node tiles than blocks fit the device) in FP64 and with 16-bit storage.

Tolerances: the precision contract's for FP64 and FP32; with 16-bit storage
those of test_gpu_row_exchange.py, one rounding of each stored part."""

import types

import numpy as np
import pytest

import oracle as O
from paper_2004_11286_gb300 import workloads as W

from gpu_helpers import TOL, gpu_handle, oracle_params, rel
from test_gpu_row_exchange import _stored_part

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,precision,shape", [(2, "fp32", (32, 32, 33)), (2, "fp32", (32, 32, 36)), (1, "fp64", (33, 63, 64))])
def test_variable_heats_beyond_the_stencil_line(M, precision, shape):
    wl = W.random_mixture(M=M, shape=shape, seed=510 + M, velocity=0.03)
    cvp = W.variable_heats(wl.molar_mass, seed=M)
    prm = oracle_params(wl, cv_poly=cvp)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    h = gpu_handle(wl, precision, cv_poly=cvp)
    h.set_populations(pops)
    h.step(3)
    got, ref = h.populations(), O.run(pops, prm, 3)
    for L in range(M + 2):
        assert rel(got[L], ref[L]) < TOL[precision], L
    h.close()


def _jets(M, shape):
    """The opposed jets with the first M of their species, and the oracle's parameters."""
    nz, ny, nx = shape
    wl, inl = W.opposed_jets(nx=nx - 2, ny=ny - 2, nz=nz, U=0.02, nozzle=(0.25, 0.75))
    if M < 4:
        cut = lambda X: X[:M] / X[:M].sum(axis=0)
        wl = W.Workload(wl.name, wl.molar_mass[:M], wl.cv_molar[:M], wl.D[:M, :M], wl.mu[:M], wl.lam[:M], cut(wl.X), wl.u,
                        wl.T, wl.P, wl.steps)
        inl = types.SimpleNamespace(y0=inl.y0, y1=inl.y1, X=np.stack([cut(x) for x in inl.X]), u=inl.u, T=inl.T, P=inl.P)
    prm0 = oracle_params(wl)
    inlet = tuple(O.init_populations(inl.X[k][:, None], np.array([[inl.u[k]], [0.0], [0.0]]), np.array([inl.T[k]]),
                                     np.array([inl.P[k]]), prm0)[..., 0] for k in range(2))
    prm = oracle_params(wl, frame=O.Frame(y0=inl.y0, y1=inl.y1, inlet=inlet))
    grid = types.SimpleNamespace(y0=inl.y0 + 1, y1=inl.y1 + 1, X=inl.X, u=inl.u, T=inl.T, P=inl.P)
    framed = W.Workload(wl.name, wl.molar_mass, wl.cv_molar, wl.D, wl.mu, wl.lam, W.with_frame(wl.X), W.with_frame(wl.u),
                        W.with_frame(wl.T), W.with_frame(wl.P), wl.steps)
    return wl, framed, grid, prm


@pytest.mark.parametrize("M,precision,shape", [
    (4, "fp32", (1, 182, 184)), (4, "fp32", (1, 182, 183)),     # frame, then row-blocked / per-node stencils
    (4, "fp32", (1, 243, 244)), (3, "fp32", (1, 125, 124)), (3, "fp64", (1, 74, 75)),   # frame of the thread per node
    (2, "fp64", (2, 50, 52)), (2, "fp32", (1, 20, 14)), (3, "fp32", (3, 12, 11)),
])
def test_jets_on_every_route(M, precision, shape):
    wl, framed, grid, prm = _jets(M, shape)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    h = gpu_handle(framed, precision, jets=grid)
    h.init_fields(framed.X, framed.u, framed.T, framed.P)
    h.step(4)
    got, ref = h.populations()[..., 1:-1, 1:-1], O.run(pops, prm, 4)
    for L in range(M + 2):
        assert rel(got[L], ref[L]) < TOL[precision], L
    h.close()


@pytest.mark.parametrize("M,precision,shape,kw", [
    (2, "fp64", (3, 4, 11), {}), (3, "fp64", (2, 3, 33), {"walls_x": True}), (3, "fp32", (2, 5, 33), {"coupling": "weak"}),
    (4, "fp32", (2, 3, 33), {}), (4, "fp32", (2, 2, 128), {}), (4, "fp32", (1, 2, 256), {"fp64_cond_bound": 1.0}),
    (5, "fp32", (2, 3, 33), {"coupling": "weak"}), (5, "fp32", (2, 3, 35), {"walls_x": True}), (5, "fp32", (2, 2, 128), {}),
    (6, "fp32", (2, 2, 128), {}), (6, "fp32", (1, 3, 256), {"coupling": "weak"}),
])
def test_thread_per_node_collide_of_large_grids(M, precision, shape, kw):
    wl = W.random_mixture(M=M, shape=shape, seed=40 + M, velocity=0.03)
    prm = oracle_params(wl, **{k: v for k, v in kw.items() if k != "fp64_cond_bound"})
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm) * W.perturbation((M + 2, 27) + wl.shape, 0.01, 4)
    got = []
    for whole in (0, 2_000_000):
        h = gpu_handle(wl, precision, **kw)
        h.set_grid_nodes(whole)
        h.set_populations(pops)
        h.step(3)
        got.append(h.populations())
        h.close()
    ref = O.run(pops, prm, 3)
    assert not np.array_equal(*got)              # another kernel, another order of the sums
    for p in got:
        for L in range(M + 2):
            assert rel(p[L], ref[L]) < TOL[precision], L


@pytest.mark.parametrize("M,shape", [(4, (21, 31, 33)), (8, (17, 33, 35))])
def test_split_collide_past_the_first_tile_fp64(M, shape):
    wl = W.random_mixture(M=M, shape=shape, seed=25 + M, velocity=0.03)
    prm = oracle_params(wl)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm)
    h = gpu_handle(wl, "fp64")
    h.set_populations(pops)
    h.step(2)
    got, ref = h.populations(), O.run(pops, prm, 2)
    for L in range(M + 2):
        assert rel(got[L], ref[L]) < TOL["fp64"], L
    h.close()


@pytest.mark.parametrize("M,precision,shape,walls", [(4, "bf16", (21, 31, 33), False), (4, "fp16", (21, 31, 33), True),
                                                     (7, "bf16", (17, 33, 35), False)])
def test_split_collide_past_the_first_tile_16_bit(M, precision, shape, walls):
    wl = W.random_mixture(M=M, shape=shape, seed=27 + M, velocity=0.02)
    prm = oracle_params(wl, walls_x=walls)
    pops = O.init_populations(wl.X, wl.u, wl.T, wl.P, prm) * W.perturbation((M + 2, 27) + wl.shape, 0.01, 3)
    h = gpu_handle(wl, precision, walls_x=walls)
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
