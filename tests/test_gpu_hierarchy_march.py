"""The marching sweep with flux registers in a hierarchy (named tiles: a small
hierarchy's levels are staged otherwise): two subcycled FP32 root steps give the
staged sweep's levels bit for bit, plain and with the reconstruction options,
and are as close to the FP64 oracle."""
import numpy as np
import pytest

import paper_1307_2265_gb300 as ez
from oracle import hierarchy as H
from paper_1307_2265_gb300 import hierarchy as gh
from test_gpu_hierarchy import _l1_by_level, fp64_reference  # noqa: F401  (fixture)
from test_gpu_staged_faces import OPTIONS

pytestmark = pytest.mark.gpu


def _levels(layout, fields, tile, steps, options=0):
    hier = gh.Hierarchy(layout, fields, 1.0 / 16)
    for _ in range(steps):
        hier.root_step(ez.Params(precision=ez.FP32, tile=(tile,) * 3, options=options))
    hier.stream.synchronize()
    return [[hier.patch_fields(l, i) for i in range(len(lev["n"]))] for l, lev in enumerate(hier.levels)]


@pytest.mark.parametrize("options", [0, OPTIONS])
@pytest.mark.parametrize("tile", [64, 256])
def test_march_equals_staged(fp64_reference, tile, options):  # noqa: F811
    layout, fields, _, logs, _ = fp64_reference
    march = _levels(layout, fields, tile, len(logs), options)
    staged = _levels(layout, fields, 0, len(logs), options)
    for A, B in zip(march, staged):
        for pa, pb in zip(A, B):
            for a, b in zip(pa, pb):
                assert np.array_equal(H._active(a), H._active(b))


def test_march_close_to_oracle(fp64_reference):  # noqa: F811
    layout, fields, ref, logs, floor = fp64_reference
    err = _l1_by_level(_levels(layout, fields, 128, len(logs)), ref)
    assert np.all(err <= np.maximum(4.0 * floor, 2e-6)), err
