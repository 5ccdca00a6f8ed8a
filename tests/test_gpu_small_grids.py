"""The one-launch CPR application of small grids against the separate launches.

Both call the same row functions in the same order, so the results are equal bit
for bit; the cell counts are one cell, a single level (dense inverse only), grids
that leave CTAs of the cluster without cells, and both sides of the 5,120-cell
rule.  A batch of small members takes the same applications as clusters of one
launch (up to eight) or as rows of the batched launches (more), each equal to the
member's own step.
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_00548_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("model,precision", [(2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (5, 3, 1), (16, 16, 1), (17, 19, 4), (31, 15, 11), (32, 32, 5)])
@pytest.mark.parametrize("stage2,cycles,stages", [(1, 1, 2), (0, 1, 2), (1, 2, 3), (0, 3, 3)])
def test_small_apply_equals_the_oracle_form(torch_cuda, model, precision, nx, ny, nz, stage2, cycles, stages):
    """fused_coarse = 0 takes the separate launches: their 7-point sweeps round alike; coarse levels
    may use other lanes per row only where the level sizes differ, which they do not here, and the
    dense solve is the same warp sum"""
    torch = torch_cuda
    from paper_1606_00548_gb300.sim import Simulator
    make = synth.oil_water_case if model == 2 else synth.black_oil_case
    out = []
    for fused in (0, 1):
        g = Simulator(make(nx=nx, ny=ny, nz=nz, sigma=0.8, seed=95, wells=[synth.well(0, 0, 0, 0, 0, 180.0)], stage2=stage2,
                           amg_cycles=cycles, cpr_stages=stages, amg_coarse_max=40), precision=precision, fused_coarse=fused)
        g.assemble(2.0)
        g.precond_setup()
        r = torch.tensor(np.random.default_rng(4).standard_normal(g.N * g.b), device="cuda")
        z = torch.full_like(r, float("nan"))
        torch.cuda.synchronize()
        g.precond_apply(r, z)
        out.append(z.cpu().numpy())
        g.close()
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("n", [3, 9])
def test_batches_of_small_members(torch_cuda, n):
    """n small members beside a larger one, each bit for bit its own sim_step"""
    from paper_1606_00548_gb300.sim import Batch, Simulator
    shapes = [(8 + 3 * k, 7 + k, 3 + k % 4) for k in range(n)] + [(40, 33, 6)]
    cases = [synth.oil_water_case(nx=a, ny=b, nz=c, sigma=0.7, seed=120 + k, nsteps=1) for k, (a, b, c) in enumerate(shapes)]
    A, B = [Simulator(c) for c in cases], [Simulator(c) for c in cases]
    batch = Batch(A, mode=0)
    sts, infos = batch.step(0.5)
    assert all(s == 0 for s in sts), (sts, batch.last_error())
    for a, b, i in zip(A, B, infos):
        st, ib = b.step(0.5)
        assert (ib.newton_iterations, ib.linear_iterations) == (i.newton_iterations, i.linear_iterations)
        for u, v in zip(a.get_state(), b.get_state()):
            assert np.array_equal(u, v)
    batch.close()
