"""The numbering of aggregates over more than 4,096 chunks of 1,024 nodes, where one block
scans the chunks' sums before they are written: 4,096 chunks (added up by every block) and
4,097 (scanned), bit for bit the oracle's hierarchy.
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth
from gpu_util import gpu_J_from_ora
from test_gpu_amg_setup import torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


def test_both_sides_of_the_line(torch_cuda):
    import oracle
    from paper_1606_00548_gb300.sim import Simulator
    for nx, ny in ((2048, 2048), (2049, 2048)):          # 2^22 nodes and 2,048 more
        case = synth.oil_water_case(nx=nx, ny=ny, nz=1, sigma=0.0, seed=91, wells=[], gmres_m=3)
        g, o = Simulator(case), oracle.Oracle(case)
        N, b = g.N, g.b
        o.assemble(1.0)
        J = o.jacobian()
        J *= np.exp(0.5 * np.random.default_rng(3).standard_normal(J.shape))
        o.set_jacobian(J)
        g.set_jacobian(gpu_J_from_ora(J, N, b))
        o.precond_setup()
        g.precond_setup()
        lo, lg = o.amg_levels(), g.amg_levels()
        assert [L["n"] for L in lo] == [L["n"] for L in lg]
        for l, (a, c) in enumerate(zip(lo, lg)):
            if l + 1 < len(lo):
                assert np.array_equal(a["agg"], c["agg"]), l
            if l:
                n, rp = a["n"], np.asarray(a["rowptr"])
                cnt = np.diff(rp)
                assert c["width"] == cnt.max()
                row = np.repeat(np.arange(n), cnt)
                k = np.arange(rp[-1]) - rp[row]
                val = np.zeros((c["width"], n))
                val[k, row] = a["val"][:rp[-1]]
                assert np.array_equal(c["col"][k, row], a["col"][:rp[-1]]) and np.array_equal(c["val"], val), l
        g.close()
        del o
