"""Assembly at the edges of its kernels: more wells than the well kernel has
warps (16), perforation counts around a warp's 32, pressures and bubble points
on, between and beyond the PVT nodes, saturations at and beyond the ends of the
relative-permeability curves, general Corey exponents, and equal potentials (the
upstream tie) in both directions along each axis.

Residual and Jacobian against the oracle, 1e-11 of their largest entry: both sides
round at most a few hundred operations of operands no larger than that (2e-14 each
at most), in different orders.
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth
from gpu_util import ora_J_from_gpu, to_cm, to_il

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_00548_gb300 import build
    build.build()
    return torch


def wells(nx, ny, nz, n, rates):
    """n wells along the diagonals, of one layer up to all; every third rate-controlled"""
    out, seen = [], set()
    for k in range(n):
        i, j = (7 * k) % nx, (5 * k + k // nx) % ny
        if (i, j) in seen:
            continue
        seen.add((i, j))
        inj = k % 2
        ctrl = (1 if inj else 2) if rates and k % 3 == 0 else 0
        out.append(synth.well(i, j, 0, min(nz - 1, k % nz), inj, 240.0 if inj else 170.0, ctrl=ctrl, rate=(3e4 if inj else -2e4)))
    return out


def compare(case, x, ph, dt):
    import oracle
    from paper_1606_00548_gb300.sim import Simulator
    g, o = Simulator(case), oracle.Oracle(case)
    N, b = g.N, g.b
    o.set_iterate(x, ph); o.assemble(dt)
    g.set_iterate(to_cm(x, N, b), ph); g.assemble(dt)
    Ro, Jo = o.residual(), o.jacobian()
    assert np.abs(to_il(g.residual(), N, b) - Ro).max() <= 1e-11 * np.abs(Ro).max() + 1e-300
    Jg = ora_J_from_gpu(g.jacobian(), N, b)
    assert np.abs(Jg - Jo).max() <= 1e-11 * np.abs(Jo).max()
    assert abs(g.cnv(dt) - o.cnv(dt)) <= 1e-11 * o.cnv(dt) + 1e-300
    if case["wells"]:
        qo = o.well_component_rates()
        assert np.abs(g.well_component_rates() - qo).max() <= 1e-11 * np.abs(qo).max()
        for a, r in zip(g.well_system(), o.well_system()):
            assert np.abs(a - np.asarray(r).reshape(a.shape)).max() <= 1e-11 * max(np.abs(r).max(), 1e-300)


@pytest.mark.parametrize("model", [2, 3])
@pytest.mark.parametrize("nz,n,rates", [(1, 1, False), (31, 3, True), (33, 20, True), (40, 60, True)])
def test_many_wells(torch_cuda, model, nz, n, rates):
    make = synth.oil_water_case if model == 2 else synth.black_oil_case
    case = make(nx=11, ny=9, nz=nz, sigma=0.8, seed=81, wells=wells(11, 9, nz, n, rates))
    N, b = 11 * 9 * nz, model
    rng = np.random.default_rng(6)
    x = np.zeros((N, b))
    x[:, 0] = case["init"]["p"] + rng.uniform(-15, 15, N)
    x[:, 1] = rng.uniform(0.12, 0.6, N)
    ph = np.ones(N, np.int8)
    if b == 3:
        ph = (rng.uniform(size=N) < 0.5).astype(np.int8)
        x[:, 2] = np.where(ph == 1, rng.uniform(0.0, 0.25, N), x[:, 0] - rng.uniform(5, 40, N))
    compare(case, x.reshape(-1), ph, 2.0)


@pytest.mark.parametrize("exponent", [2.0, 3.5])
@pytest.mark.parametrize("model", [2, 3])
def test_property_edges(torch_cuda, model, exponent):
    """every combination of pressure, saturation and third unknown at nodes and ends"""
    fl = synth.oil_water_fluid() if model == 2 else synth.black_oil_fluid()
    fl.update(nw=exponent, now=exponent, ng=exponent, nog=exponent)
    nx, ny, nz = 13, 9, 8
    N = nx * ny * nz
    if model == 2:
        case = synth.oil_water_case(nx=nx, ny=ny, nz=nz, sigma=0.5, seed=82, fluid=fl, wells=[])
    else:
        case = synth.black_oil_case(nx=nx, ny=ny, nz=nz, sigma=0.5, seed=82, wells=[])
        case["fluid"].update({k: exponent for k in ("nw", "now", "ng", "nog")})
    ps = [20.0, 50.0, 75.0, 100.0, 149.99999, 150.0, 200.0, 399.0, 400.0, 430.0]
    sws = [0.0, 0.05, 0.1, 0.3, 0.89, 0.9, 0.95, 1.0]
    rng = np.random.default_rng(7)
    x = np.zeros((N, model))
    x[:, 0] = rng.choice(ps, N)
    x[:, 1] = rng.choice(sws, N)
    ph = np.ones(N, np.int8)
    if model == 3:
        ph = (rng.uniform(size=N) < 0.5).astype(np.int8)
        x[:, 2] = np.where(ph == 1, rng.choice([0.0, 0.05, 0.2, 0.75, 0.9], N), np.minimum(x[:, 0], rng.choice(ps, N)))
    compare(case, x.reshape(-1), ph, 5.0)
    # equal pressures: no flow across lateral faces, upstream ties everywhere
    x[:, 0] = 180.0
    compare(case, x.reshape(-1), ph, 5.0)
