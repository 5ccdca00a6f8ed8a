"""Several V-cycles per stage P on grids above the one-launch rule (5,120 cells).

5,491 cells in the mixed form start the coarse cluster cycle at level 0, where the
cycles' corrections are added by a launch of their own; 5,491 cells in FP64 and 8,091 in
both forms add them in the last smoothing sweep.  fused_coarse = 0 takes the separate
launches of every level.  The two differ by the rounding of an application: a few
thousand operations' worth of the precision's epsilon at most.
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-4)])
@pytest.mark.parametrize("dims", [(17, 19, 17), (29, 31, 9)])
@pytest.mark.parametrize("cycles,stages", [(2, 2), (3, 2), (3, 3)])
def test_cycles_add_up(precision, tol, dims, cycles, stages):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_00548_gb300 import build
    build.build()
    from paper_1606_00548_gb300.sim import Simulator
    out = []
    for fused in (0, 1):
        g = Simulator(synth.black_oil_case(nx=dims[0], ny=dims[1], nz=dims[2], sigma=0.8, seed=96, amg_cycles=cycles,
                                           cpr_stages=stages), precision=precision, fused_coarse=fused)
        g.assemble(2.0)
        g.precond_setup()
        r = torch.tensor(np.random.default_rng(4).standard_normal(g.N * g.b), device="cuda")
        z = torch.full_like(r, float("nan"))
        torch.cuda.synchronize()
        for _ in range(2):             # the second application finds the first one's buffers
            g.precond_apply(r, z)
        out.append(z.cpu().numpy())
        g.close()
    assert np.isfinite(out[0]).all()
    assert np.linalg.norm(out[0] - out[1]) <= tol * np.linalg.norm(out[0])
