"""Batched domains walked by few persistent blocks: a block that takes many
tiles in turn reuses its shared-memory stage, in which 16-bit storage also
writes other lanes' columns.  The tiles' work does not depend on which block
takes them, so the result is the same bit for bit as with a block per tile."""

import numpy as np
import pytest

from paper_2004_11286_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _batch(M, shapes, precision):
    from paper_2004_11286_gb300 import binding
    wls = [W.random_mixture(M=M, shape=s, seed=40 + k, velocity=0.02) for k, s in enumerate(shapes)]
    b = binding.LbmBatch([binding.workload_params(w, precision=precision, slaved=W.slaved_species(w)) for w in wls])
    for d, w in enumerate(wls):
        b.domain(d).init_fields(w.X, w.u, w.T, w.P)
    return b


@pytest.mark.parametrize("M,precision", [(1, "fp16"), (2, "bf16"), (3, "bf16"), (3, "fp32"), (4, "bf16"), (8, "fp16")])
def test_few_blocks_give_what_a_block_per_tile_gives(M, precision):
    shapes = [(5, 6, 33), (4, 7, 11), (6, 5, 70)]
    got = []
    for blocks in (None, 2):
        b = _batch(M, shapes, precision)
        b.set_mode(0)
        c = b.config()
        b.set_config(blocks or c["tiles_collide"], 256, c["tiles_256"], use_graph=False)
        b.step(6)
        b.synchronize()
        got.append([b.domain(d).populations().copy() for d in range(len(shapes))])
        b.close()
    for one, few in zip(*got):
        assert np.array_equal(one, few)
