"""Weight gradients on grids where a CTA takes several bricks.

wgrad_tc_kernel deals bricks of 128 x 1 x 4 cells to two CTAs per SM.  The grids below give
a CTA 2 to 9 of them, one brick more for some than for others, and lines of x that do not
fill a brick, two of them with a second brick column, and bricks of 1 to 4 lines in z; the
last has whole bricks only.  Reference, rounding and bounds are those of the smaller grids
(test_gpu_learned.py): the same roundings in FP64, so what is left is FP32 accumulation and
the rare BF16 flip.
"""
import numpy as np
import pytest

from test_gpu_learned import reference, torch_cuda, unflatten  # noqa: F401

pytestmark = pytest.mark.gpu


def bricks(nx, ny, nz):
    return ((nx + 127) // 128) * ((nz + 3) // 4) * ny


@pytest.mark.parametrize("nx,ny,nz,each", [(5, 41, 61, 2), (131, 155, 6, 2), (7, 59, 63, 3), (3, 155, 64, 8), (17, 163, 61, 8),
                                           (128, 43, 60, 2)])
def test_gradients_of_many_bricks_match_reference(torch_cuda, nx, ny, nz, each):
    torch = torch_cuda
    from paper_1606_00548_gb300.sim import Net
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    assert bricks(nx, ny, nz) // ctas == each and bricks(nx, ny, nz) % ctas != 0
    net = Net(nx, ny, nz, seed=3)
    rng = np.random.default_rng(4)
    p = net.get_params()
    p[:] = 0.5 * p + 0.05 * rng.standard_normal(p.size).astype(np.float32)
    net.set_params(p)
    x = rng.standard_normal((nz, ny, nx, 4)).astype(np.float32)
    t = rng.standard_normal((nz, ny, nx, 1)).astype(np.float32)
    # a trend along y: a slab taken for a neighbour's is seen in the gradients
    x += np.linspace(-1.0, 2.0, ny, dtype=np.float32)[None, :, None, None]
    t -= np.linspace(-1.0, 2.0, ny, dtype=np.float32)[None, :, None, None]
    loss, grads = net.loss_grad(torch.tensor(x.reshape(-1, 4), device="cuda"), torch.tensor(t.reshape(-1), device="cuda"))
    _, loss_ref, grads_ref = reference(x.astype(np.float64), t.astype(np.float64), unflatten(net.get_params()))
    assert loss == pytest.approx(loss_ref, rel=2e-3)
    for l, (got, ref) in enumerate(zip(unflatten(grads), grads_ref)):
        for a, b in zip(got, ref):
            err = np.abs(a - b)
            assert err.max() <= 2e-2 * np.abs(b).max(), (l, err.max(), np.abs(b).max())
            assert np.median(err) <= 2e-3 * np.abs(b).max()
    net.close()
