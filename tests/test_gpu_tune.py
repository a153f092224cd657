"""The autotuner's choice is no slower than not tuning: for a batch of few
pencils, where the library's default is another kernel than the named tiles',
and for one that fills the device."""
import pytest

import paper_1307_2265_gb300 as ez
from gpu_helpers import batch_from_patches, white_patch
from paper_1307_2265_gb300 import tune

pytestmark = pytest.mark.gpu


def _step_ms(b, params, reps=20):
    import torch
    for s in range(3):
        ez.step(b, params, s, b.dt_dev)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for s in range(reps):
        ez.step(b, params, s, b.dt_dev)
    e1.record()
    e1.synchronize()
    return e0.elapsed_time(e1) / reps


@pytest.mark.parametrize("options", [0, ez.OPT_STEEPEN | ez.OPT_FLATTEN])
@pytest.mark.parametrize("sizes", [[(32, 32, 32)], [(64, 64, 64)] * 24])
def test_tuned_step_is_not_slower_than_the_default(sizes, options):
    b = batch_from_patches([white_patch(n, seed=5 + i) for i, n in enumerate(sizes)], [1.0 / 64] * 3,
                           flags=ez.PATCH_PERIODIC)
    params = ez.Params(precision=ez.FP32, options=options)
    tiles, ms = tune.autotune_tiles(b, params)
    assert all(0 in ms[d] for d in range(3))
    b.dt_dev.fill_(1e-5)
    tuned = min(_step_ms(b, ez.Params(precision=ez.FP32, options=options, tile=tiles)) for _ in range(3))
    default = min(_step_ms(b, params) for _ in range(3))
    assert tuned <= 1.25 * default, (tiles, tuned, default)
