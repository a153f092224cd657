"""The FP32 staged sweep against the marching sweep (chosen by naming a tile) in
the forms test_gpu_staged leaves out: the approximate solvers, fallback mode 2,
cells that the fallback mends in either mode, and flux registers.  Fields,
counters and registers are the same bits."""
import numpy as np
import pytest

import paper_1307_2265_gb300 as ez
from gpu_helpers import active, batch_from_patches, gpu_patches, white_patch, with_registers
from test_gpu_staged_faces import DX, OPTIONS, SIZES, _split_flow

pytestmark = pytest.mark.gpu


def _run(flow, tile, registers, flags, **kw):
    if flow == "split":
        patches, dt = [_split_flow(n, 60 + i) for i, n in enumerate(SIZES)], 1.4 * DX / 7.5
    else:
        patches, dt = [white_patch(n, seed=60 + i) for i, n in enumerate(SIZES)], 0.3 * DX / 4.0
    b = batch_from_patches(patches, [DX] * 3, flags=flags)
    if registers:
        with_registers(b)
    for d in range(3):
        ez.ppm_sweep(b, d, dt, 0, ez.Params(precision=ez.FP32, tile=(tile,) * 3, **kw))
    freg = b.freg.cpu().numpy() if registers else np.zeros(0)
    return [active(f) for U in gpu_patches(b) for f in U] + [freg], b.read_status()


@pytest.mark.parametrize("registers", [False, True])
@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("options", [0, OPTIONS])
@pytest.mark.parametrize("fallback", [1, 2])
@pytest.mark.parametrize("solver", [ez.SOLVER_TWOSHOCK, ez.SOLVER_HLL, ez.SOLVER_HLLC])
@pytest.mark.parametrize("flow", ["white", "split"])
def test_staged_equals_march(flow, solver, fallback, options, flags, registers):
    kw = dict(solver=solver, fallback=fallback, options=options)
    (staged, s), (march, m) = _run(flow, 0, registers, flags, **kw), _run(flow, 128, registers, flags, **kw)
    assert s == m
    assert flow == "white" or s["hll_cells"] > 0
    for a, c in zip(staged, march):
        assert np.array_equal(a, c, equal_nan=True)
