"""FP32 staged sweep beside failing cells (Sec. 4.1.2): a re-fluxed face enters
its two cells and the flux register as one value.  Every cell's update is
(U + G_left) - G_right, bit for bit, with G the applied increments that the
all-face registers hold, so what leaves a cell is what its neighbour gets."""
import numpy as np
import pytest

import paper_1307_2265_gb300 as ez
from gpu_helpers import active, batch_from_patches, gpu_patches, with_registers
from paper_1307_2265_gb300 import synth

pytestmark = pytest.mark.gpu
OPTIONS = ez.OPT_STEEPEN | ez.OPT_FLATTEN | ez.OPT_DIFFUSE
SIZES = [(60, 21, 18), (333, 3, 5), (2, 270, 3), (5, 2, 300), (1, 1, 1)]
DX, U0 = 1.0 / 64, 6.0


def _split_flow(n, seed, gamma=5.0 / 3.0):
    """Cells of random density that move at 3 to 6 either way along each axis."""
    rng = np.random.default_rng(seed)
    sh = n[::-1]
    vel = [rng.choice([-1.0, 1.0], sh) * U0 * rng.uniform(0.5, 1.0, sh) for _ in range(3)]
    prims = (np.exp(rng.normal(0, 0.5, sh)), *vel, rng.uniform(0.2, 0.6, sh))
    return [synth.embed(f) for f in synth.prims_to_conserved(*prims, gamma)]


def _increments(batch, i, d):
    """All-face register of patch i along axis d: (n_a2, n_a1, n_d + 1, 5)."""
    n = [int(v) for v in batch.table["n"][i]]
    o = int(batch.table["freg_all"][i])
    for a in range(d):
        o += (n[a] + 1) * np.prod([n[b] for b in range(3) if b != a], dtype=int) * 5
    a1, a2 = [b for b in range(3) if b != d]
    size = (n[d] + 1) * n[a1] * n[a2] * 5
    return batch.freg[o:o + size].cpu().numpy().reshape(n[a2], n[a1], n[d] + 1, 5)


@pytest.mark.parametrize("d", [0, 1, 2])
@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("fallback,options", [(1, 0), (1, OPTIONS), (2, 0), (2, OPTIONS)])
def test_cells_share_their_faces(fallback, options, flags, d):
    patches = [_split_flow(n, 60 + i) for i, n in enumerate(SIZES)]
    b = with_registers(batch_from_patches(patches, [DX] * 3, flags=flags))
    dt = 1.4 * DX / 7.5     # beyond the CFL limit: mode 1 has cells to mend too
    ez.ppm_sweep(b, d, dt, 0, ez.Params(precision=ez.FP32, fallback=fallback, options=options))
    assert b.read_status()["hll_cells"] > 0
    fields = [0, 1 + d, 1 + (1 if d == 0 else 0), 1 + (1 if d == 2 else 2), 4]   # of the register's components
    for i, (new, old) in enumerate(zip(gpu_patches(b), patches)):
        G = _increments(b, i, d)
        for c, f in enumerate(fields):
            u = np.moveaxis(active(old[f]), 2 - d, -1)
            want = (u + G[..., :-1, c]) - G[..., 1:, c]
            assert np.array_equal(np.moveaxis(active(new[f]), 2 - d, -1), want, equal_nan=True), (i, f)
