"""The Krylov reductions at the edges of their launch grids.

A reduction over n entries runs min(ceil(n / 256), 152) blocks of 256 threads
(304 from 2^21 entries), a thread taking 4, 2 or 1 entries of its stride at a
time by the number of basis vectors, and the last block to finish folds the
partials.  The sizes below leave one entry, one short of a block, one block
and one more, one wave of blocks and one more, and both sides of 2^21; 32
basis vectors (33 values with w . w) are the longest.
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


@pytest.mark.parametrize("nx,ny,nz,orth", [
    (1, 1, 1, 0), (127, 1, 1, 0), (128, 1, 1, 0), (43, 3, 1, 1), (152, 128, 1, 0), (151, 43, 3, 0), (19457, 1, 1, 1),
    (1024, 32, 32, 0), (1023, 32, 32, 0)])
def test_norms_and_residuals_of_a_solve(torch_cuda, nx, ny, nz, orth):
    """||b|| and ||b - J x|| as the solver reports them against torch's norms of the same vectors.
    A sum of n squares in any order is within n 2^-53 of the exact one, so two of them differ by
    2 n 2^-53 relative at most and their roots by n 2^-53 <= 2.4e-10; the residual's entries carry
    the product's rounding too (63 products per row), 1e-6 of a residual at 1e-8 of ||b||."""
    torch = torch_cuda
    from paper_1606_00548_gb300.sim import Simulator
    case = synth.oil_water_case(nx=nx, ny=ny, nz=nz, sigma=0.0, k=200.0,
                                wells=[synth.well(0, 0, 0, 0, 1, 230.0)], gmres_m=32, orth=orth)
    g = Simulator(case)
    n = g.N * g.b
    g.assemble(1.0)
    b = torch.randn(n, generator=torch.Generator(device="cuda").manual_seed(nx), device="cuda", dtype=torch.float64)
    x, y = torch.empty_like(b), torch.empty_like(b)
    st, info = g.linear_solve(b, x)
    assert st == 0 and info.converged
    nb = float(torch.linalg.vector_norm(b))
    assert abs(info.b_norm - nb) <= n * 2.0 ** -53 * nb + 1e-15 * nb
    g.spmv(x, y)
    r = float(torch.linalg.vector_norm(b - y))
    assert r <= 1.000001e-8 * nb
    assert abs(info.r_norm - r) <= 1e-6 * 1e-8 * nb
    g.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_long_basis_matches_oracle(torch_cuda, precision):
    """block-Jacobi FGMRES(32) on a system it needs several full cycles for: every basis length
    from 1 to 32 occurs; the iteration count is the oracle's within 1 and the solutions agree to
    the tolerance times the conditioning."""
    torch = torch_cuda
    import oracle
    from paper_1606_00548_gb300.sim import Simulator
    from gpu_util import gpu_J_from_ora, rel_err, to_cm, to_il
    case = synth.oil_water_case(nx=13, ny=11, nz=3, sigma=0.5, seed=71, precond=1, gmres_m=32, gmres_max_restarts=60)
    g, o = Simulator(case, precision=precision), oracle.Oracle(case)
    N, b = g.N, g.b
    o.assemble(0.2); g.assemble(0.2)
    g.set_jacobian(gpu_J_from_ora(o.jacobian(), N, b))
    rhs = np.random.default_rng(5).standard_normal(N * b)
    xo, io = o.linear_solve(rhs)
    bd = torch.tensor(to_cm(rhs, N, b), device="cuda", dtype=torch.float64)
    xd = torch.empty_like(bd)
    st, ig = g.linear_solve(bd, xd)
    assert io.converged and ig.converged and ig.iterations > 32
    if precision == 0:
        assert abs(ig.iterations - io.iterations) <= 1
    assert rel_err(to_il(xd.cpu().numpy(), N, b), xo) <= 1e-5
