"""Sizes on both sides of the lines that choose a launch: the chunks of the aggregate
numbering (256 nodes up to 2^18 nodes, 1,024 above), the lanes of a coarse row (16 up to
256 rows, 8 up to 1,024, 4 up to 131,072) and the one-launch application (5,120 cells).
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth
from test_gpu_amg_setup import compare_hierarchies, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(255, 1, 1), (256, 1, 1), (257, 1, 1), (512, 512, 1), (2405, 109, 1)])
def test_chunks_of_the_numbering(torch_cuda, nx, ny, nz):
    """one node less than a chunk, one chunk, one more; 2^18 nodes and one more"""
    big = nx * ny * nz > 1000
    case = synth.oil_water_case(nx=nx, ny=ny, nz=nz, sigma=0.0 if big else 1.0, seed=91, wells=[], amg_coarse_max=256 if big else 8)
    assert compare_hierarchies(case, 1.0, rough=0.5 if big else 0.0) >= 2


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-4)])
@pytest.mark.parametrize("nx,ny,nz", [(569, 9, 1), (17, 17, 18)])
@pytest.mark.parametrize("cycles,stages", [(1, 2), (2, 3)])
def test_application_above_the_one_launch_rule(torch_cuda, precision, tol, nx, ny, nz, cycles, stages):
    """5,121 and 5,202 cells with the coarse levels in one cluster launch and as launches of
    their own; an application is a few thousand operations of the precision's epsilon"""
    torch = torch_cuda
    from paper_1606_00548_gb300.sim import Simulator
    out = []
    for fused in (0, 1):
        g = Simulator(synth.black_oil_case(nx=nx, ny=ny, nz=nz, sigma=0.8, seed=97, amg_cycles=cycles, cpr_stages=stages,
                                           wells=[synth.well(0, 0, 0, 0, 0, 180.0)]), precision=precision, fused_coarse=fused)
        g.assemble(2.0)
        g.precond_setup()
        r = torch.tensor(np.random.default_rng(4).standard_normal(g.N * g.b), device="cuda")
        z = torch.full_like(r, float("nan"))
        torch.cuda.synchronize()
        for _ in range(2):
            g.precond_apply(r, z)
        out.append(z.cpu().numpy())
        g.close()
    assert np.isfinite(out[0]).all()
    assert np.linalg.norm(out[0] - out[1]) <= tol * np.linalg.norm(out[0])


def test_lanes_of_a_row_do_not_change_the_product(torch_cuda):
    """Levels around 256 and 1,024 rows: the application with the device's hierarchy against the
    same V-cycle and stage F in the oracle (both FP64; 1e-10 of the largest entry, a few
    thousand operations)"""
    torch = torch_cuda
    import oracle
    from paper_1606_00548_gb300.sim import Simulator
    from gpu_util import gpu_J_from_ora, to_cm, to_il
    seen = []
    for n in (300, 700, 1100, 2900, 6200):
        case = synth.oil_water_case(nx=n, ny=5, nz=1, sigma=1.0, seed=98, wells=[], amg_coarse_max=16)
        g, o = Simulator(case), oracle.Oracle(case)
        N, b = g.N, g.b
        o.assemble(1.0)
        g.set_jacobian(gpu_J_from_ora(o.jacobian(), N, b))
        o.precond_setup()
        g.precond_setup()
        seen += [L["n"] for L in g.amg_levels()[1:]]
        r = np.random.default_rng(5).standard_normal(N * b)
        zo = o.precond_apply(r)
        z = torch.empty(N * b, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        g.precond_apply(torch.tensor(to_cm(r, N, b), device="cuda"), z)
        assert np.abs(to_il(z.cpu().numpy(), N, b) - zo).max() <= 1e-10 * np.abs(zo).max(), n
        g.close()
    assert any(s <= 256 for s in seen) and any(256 < s <= 1024 for s in seen) and any(1024 < s < 131072 for s in seen)
