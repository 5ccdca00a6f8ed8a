"""The one-launch Gram-Schmidt step of short vectors against the separate launches.

A batch takes the separate launches of every member, and its step equals the member's
own bit for bit: the sizes below leave one entry, a part of a virtual block of 256, one
block and one more, a block in a CTA's second half (from 17 blocks) and both sides of
the 6,144-entry rule; both reorthogonalisation modes; bases of up to 32 vectors
(the longer ones with the block-Jacobi second stage).
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (127, 1, 1), (128, 1, 1), (43, 3, 1), (16, 16, 8), (27, 19, 4), (32, 32, 3), (439, 7, 1)]


@pytest.mark.parametrize("orth", [0, 1])
@pytest.mark.parametrize("stage2", [0, 1])
def test_own_step_equals_the_batched_one(orth, stage2):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_00548_gb300 import build
    build.build()
    from paper_1606_00548_gb300.sim import Batch, Simulator
    cases = [synth.oil_water_case(nx=a, ny=b, nz=c, sigma=0.6, seed=140 + k, nsteps=1, orth=orth, stage2=stage2, gmres_m=32,
                                  wells=[synth.well(0, 0, 0, 0, 1, 230.0)])
             for k, (a, b, c) in enumerate(SHAPES)]
    A, B = [Simulator(c) for c in cases], [Simulator(c) for c in cases]
    batch = Batch(A, mode=0)
    sts, infos = batch.step(0.2)
    assert all(s == 0 for s in sts), (sts, batch.last_error())
    for shape, a, b, i in zip(SHAPES, A, B, infos):
        st, ib = b.step(0.2)
        assert st == 0 and (ib.newton_iterations, ib.linear_iterations) == (i.newton_iterations, i.linear_iterations), shape
        for u, v in zip(a.get_state(), b.get_state()):
            assert np.array_equal(u, v), shape
    batch.close()
