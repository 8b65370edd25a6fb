"""A batched domain's state is that of the same domain stepped alone, whichever
launch plan runs the batch.  Where a domain's step takes the split collide (from
four species) the batch runs the same tiles: bit for bit, at every precision,
rows of a multiple of four and not.  Where it takes a thread per node the batch
compiles the same function apart, and the two agree to the precision
contract's rounding (1e-12 FP64, 1e-5 FP32): domains on both sides of the size
lines by which a step chooses its collide, in one batch."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import binding, workloads as W

from gpu_helpers import TOL, gpu_handle, rel

pytestmark = pytest.mark.gpu


def _compare(M, precision, shapes, agree):
    wls = [W.random_mixture(M=M, shape=s, seed=7 * M + k, velocity=0.02) for k, s in enumerate(shapes)]
    ref = []
    for w in wls:
        h = gpu_handle(w, precision)
        h.init_fields(w.X, w.u, w.T, w.P)
        h.step(7)
        ref.append(h.populations())
        h.close()
    for mode, blocks in ((0, None), (0, 3), (1, None)):
        b = binding.LbmBatch([binding.workload_params(w, precision=precision, slaved=W.slaved_species(w)) for w in wls])
        for d, w in enumerate(wls):
            b.domain(d).init_fields(w.X, w.u, w.T, w.P)
        b.set_mode(mode, branches=2)
        c = b.config()
        if blocks:
            b.set_config(blocks, 128, 5)
        assert c["tiles_collide"] == sum(-(-w.nodes // c["collide_block"]) for w in wls)
        b.step(5)
        b.step(2)
        b.synchronize()
        for d in range(len(wls)):
            assert agree(b.domain(d).populations(), ref[d]), (mode, blocks, shapes[d])
        b.close()


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("M", range(4, 9))
def test_split_domains_have_the_single_domains_bits(M, precision):
    _compare(M, precision, [(3, 5, 33), (4, 3, 12), (2, 7, 9)], np.array_equal)


@pytest.mark.parametrize("M,precision,shapes", [
    (2, "fp64", [(3, 4, 11), (18, 17, 17), (12, 18, 24)]), (3, "fp64", [(18, 17, 17), (3, 4, 12)]),
    (3, "fp32", [(3, 5, 33), (25, 25, 24), (25, 24, 25)]), (4, "fp32", [(3, 4, 11), (40, 38, 39)]),
    (5, "fp32", [(25, 25, 24), (3, 4, 11)]), (1, "fp32", [(3, 5, 33), (4, 3, 12)]),
])
def test_domains_on_both_sides_of_a_size_line(M, precision, shapes):
    _compare(M, precision, shapes, lambda a, b: max(rel(a[L], b[L]) for L in range(M + 2)) < TOL[precision])
