"""Device memory of a handle and of its preconditioner set-up, and the hierarchy where the
set-up builds its products in other places than usual.

A product's width is known only when it has been built.  With few Krylov directions
(gmres_m) there is no room for it beside the levels, and its width is counted first; in
the FP32-preconditioned two-phase form the second product of a level is built in the pool.
The hierarchy is the same in all of them.
"""
import ctypes

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
    torch.zeros(1, device="cuda")
    return torch


class Pool:
    """the device's default memory pool"""
    USED, USED_HIGH = 7, 8             # cudaMemPoolAttrUsedMemCurrent, ...High

    def __init__(self):
        lib = [line.split()[-1] for line in open("/proc/self/maps") if "libcudart" in line][0]
        self.rt, self.p = ctypes.CDLL(lib), ctypes.c_void_p()
        assert self.rt.cudaDeviceGetDefaultMemPool(ctypes.byref(self.p), 0) == 0

    def get(self, attr):
        v = ctypes.c_uint64()
        assert self.rt.cudaMemPoolGetAttribute(self.p, attr, ctypes.byref(v)) == 0
        return v.value

    def reset_high(self):
        assert self.rt.cudaMemPoolSetAttribute(self.p, self.USED_HIGH, ctypes.byref(ctypes.c_uint64(0))) == 0


def rough_case(model, nx, ny, nz, m):
    make = synth.oil_water_case if model == 2 else synth.black_oil_case
    case = make(nx=nx, ny=ny, nz=nz, sigma=0.0, gmres_m=m, **({} if model == 2 else dict(corr_len=0.0)))
    k = np.exp(4.6 + np.random.default_rng(1).standard_normal(nx * ny * nz))
    case.update(kx=k, ky=k.copy(), kz=0.1 * k)
    return case


# bytes a cell of a handle and of its set-up at its largest, when each product's width was
# counted by a launch of its own before the product was allocated (measured at 16.8M cells;
# the mixed black-oil form at 4.1M)
BEFORE = {(3, 0, 30): 3303 + 188, (3, 1, 30): 2777 + 177, (2, 0, 30): 1943 + 179, (2, 1, 30): 1635 + 179,
          (2, 0, 2): 1079 + 179}


@pytest.mark.parametrize("model,precision,m", sorted(BEFORE))
def test_setup_needs_no_more_memory_than_with_counted_widths(torch_cuda, model, precision, m):
    from paper_1606_00548_gb300.sim import Simulator
    dims = (256, 128, 128)
    N = dims[0] * dims[1] * dims[2]
    case = rough_case(model, *dims, m)
    pool = Pool()
    torch_cuda.cuda.synchronize()
    free = torch_cuda.cuda.mem_get_info()[0]
    g = Simulator(case, precision=precision)
    handle = free - torch_cuda.cuda.mem_get_info()[0]
    g.assemble(1.0)
    torch_cuda.cuda.synchronize()
    used = pool.get(pool.USED)
    pool.reset_high()
    g.precond_setup()
    high, held = pool.get(pool.USED_HIGH) - used, pool.get(pool.USED) - used
    print(f"b {model} precision {precision} m {m}: handle {handle / N:.0f}, set-up {high / N:.0f}, held {held / N:.0f} B a cell")
    g.close()
    assert handle + high <= BEFORE[model, precision, m] * N


@pytest.mark.parametrize("model,precision,m", [(2, 0, 2), (2, 1, 2), (2, 1, 30), (3, 1, 7), (3, 0, 1)])
def test_hierarchy_does_not_depend_on_where_it_is_built(torch_cuda, model, precision, m):
    """452,907 cells: a first product of about 190k rows, a second of about 80k"""
    from paper_1606_00548_gb300.sim import Simulator
    levels = []
    for mm, prec in ((30, 0), (m, precision)):
        g = Simulator(rough_case(model, 91, 79, 63, mm), precision=prec)
        g.assemble(1.0)
        g.precond_setup()
        g.precond_setup()              # the second finds the first one's memory
        levels.append(g.amg_levels())
        g.close()
    a, b = levels
    assert [(L["n"], L["width"]) for L in a] == [(L["n"], L["width"]) for L in b] and len(a) > 3
    for l, (p, q) in enumerate(zip(a, b)):
        if l + 1 < len(a):
            assert np.array_equal(p["agg"], q["agg"]), l
        if l:
            assert np.array_equal(p["col"], q["col"]) and np.array_equal(p["val"], q["val"]), l
