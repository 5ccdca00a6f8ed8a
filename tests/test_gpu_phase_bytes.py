"""The bytes a Newton call reports for its set-up and solve: the model stated in sim.h, with
each coarse row counting the columns it has (its level's width is the longest row's, two
to three times the mean).
"""
import numpy as np
import pytest

from paper_1606_00548_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("model,precision,coarse_max,stages", [(2, 0, 8, 2), (3, 0, 256, 2), (3, 1, 40, 2), (3, 1, 40, 3),
                                                               (2, 0, 1024, 2)])
def test_reported_bytes_are_the_entries(model, precision, coarse_max, stages):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1606_00548_gb300 import build
    build.build()
    from paper_1606_00548_gb300.sim import Simulator
    make = synth.oil_water_case if model == 2 else synth.black_oil_case
    dims = (9, 7, 5) if coarse_max == 1024 else (37, 29, 11)      # the last: one level
    g = Simulator(make(nx=dims[0], ny=dims[1], nz=dims[2], sigma=1.0, seed=93, amg_coarse_max=coarse_max, cpr_stages=stages),
                  precision=precision)
    N, b, t = float(g.N), g.b, 4 if precision else 8
    st, info = g.newton_step(2.0)
    levels = g.amg_levels()
    rows = [float(L["n"]) for L in levels]
    e = [7 * N] + [float((L["col"] >= 0).sum()) for L in levels[1:]]
    assert len(levels) == 1 or e[1] < 0.7 * levels[1]["width"] * rows[1]
    setup = N * (7 * b * b * (8 + 2 * t) + 56 + b * b * t)
    apply = N * (8 * b + b * t + t) + rows[-1] ** 2 * 8 + 2 * rows[-1] * t
    for l in range(len(levels) - 1):
        setup += 4 * e[l] * 12 + e[l + 1] * 12 + 4 * rows[l]
        apply += 3 * e[l] * (t if l == 0 else 4 + t) + 6 * rows[l] * t
    stage_f = N * (8 * b + b * b * t + 7 * b * t + t + b * t) + N * (8 * b * b * t + 4 * b * t)
    apply += stage_f if stages == 2 else 2 * stage_f + N * 7 * b * b * t
    assert info.phase.setup_bytes == pytest.approx(setup, rel=1e-12)
    k, n = info.linear_iterations, b * N
    cycles = [30] * ((k - 1) // 30) + [(k - 1) % 30 + 1]          # restarts after 30 vectors
    spmv = (7 * b * b + b) * 8 * N + b * N * t
    solve = sum(sum(spmv + apply + (3.0 * (j + 1) + 7) * n * 8 for j in range(c)) + c * n * t + 2 * n * 8 + spmv + 3 * n * 8
                for c in cycles)
    assert info.phase.solve_bytes == pytest.approx(solve, rel=1e-12)
    g.close()
