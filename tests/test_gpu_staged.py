"""The staged sweep (one tile of whole pencils, or of windows of long ones, in
shared memory) at its edges: one-cell axes, pencils of exactly one tile, one
position more, many windows, ragged batches, wrapped and ghosted patches.  FP64
equals the oracle bit for bit; FP32 equals the marching sweep (chosen by naming
a tile) bit for bit, counters included."""
import numpy as np
import pytest

import oracle
import paper_1307_2265_gb300 as ez
from gpu_helpers import active, batch_from_patches, gpu_evolve, gpu_patches, oracle_evolve_batch, white_patch

pytestmark = pytest.mark.gpu

BATCHES = {
    "cells": [(1, 1, 1), (2, 1, 3), (1, 5, 1)],
    "tile": [(250, 2, 3), (2, 250, 1), (1, 3, 250)],
    "over": [(251, 3, 2), (3, 251, 2), (2, 1, 251)],
    "windows": [(700, 1, 2), (2, 333, 3), (1, 2, 520)],
    "ragged": [(38, 33, 17), (8, 64, 9), (129, 5, 6), (7, 7, 7)],
}


def _patches(sizes, mach):
    return [white_patch(n, seed=40 + i, mach=mach) for i, n in enumerate(sizes)]


@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("mach", [1.0, 12.0])
@pytest.mark.parametrize("name", sorted(BATCHES))
def test_fp64_equals_oracle(name, mach, flags):
    dx = [1.0 / 64] * 3
    patches = _patches(BATCHES[name], mach)
    ora = [[f.copy() for f in U] for U in patches]
    oracle_evolve_batch(ora, dx, 2, oracle.Params())
    b = batch_from_patches(patches, dx, flags=flags)
    gpu_evolve(b, ez.Params(precision=ez.FP64), 2)
    for G, O in zip(gpu_patches(b), ora):
        for g, o in zip(G, O):
            assert np.array_equal(active(g), active(o))


@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("mach", [1.0, 12.0])
@pytest.mark.parametrize("options", [0, ez.OPT_STEEPEN | ez.OPT_FLATTEN | ez.OPT_DIFFUSE])
@pytest.mark.parametrize("name", sorted(BATCHES))
def test_fp32_equals_march(name, options, mach, flags):
    dx = [1.0 / 64] * 3
    out = []
    for tile in ((0, 0, 0), (128, 128, 128)):
        b = batch_from_patches(_patches(BATCHES[name], mach), dx, flags=flags)
        gpu_evolve(b, ez.Params(precision=ez.FP32, tile=tile, options=options), 2)
        out.append((gpu_patches(b), b.read_status()))
    assert out[0][1] == out[1][1]
    for G, M in zip(out[0][0], out[1][0]):
        for g, m in zip(G, M):
            assert np.array_equal(active(g), active(m), equal_nan=True)


OPTIONS = ez.OPT_STEEPEN | ez.OPT_FLATTEN | ez.OPT_DIFFUSE


@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("mach", [1.0, 12.0])
@pytest.mark.parametrize("name", ["over", "windows", "ragged"])
def test_fp64_options_and_fallback_2_equal_oracle(name, mach, flags):
    dx = [1.0 / 64] * 3
    patches = _patches(BATCHES[name], mach)
    ora = [[f.copy() for f in U] for U in patches]
    oracle_evolve_batch(ora, dx, 2, oracle.Params(options=OPTIONS, fallback=2))
    b = batch_from_patches(patches, dx, flags=flags)
    gpu_evolve(b, ez.Params(precision=ez.FP64, options=OPTIONS, fallback=2), 2)
    for G, O in zip(gpu_patches(b), ora):
        for g, o in zip(G, O):
            assert np.array_equal(active(g), active(o))


@pytest.mark.parametrize("flags", [0, ez.PATCH_PERIODIC])
@pytest.mark.parametrize("mach", [1.0, 12.0])
@pytest.mark.parametrize("name", ["over", "windows", "ragged"])
def test_fp64_dual_equals_oracle(name, mach, flags):
    """The gas energy's resynchronisation reaches across a window's edge."""
    dx = [1.0 / 64] * 3
    patches = _patches(BATCHES[name], mach)
    P = oracle.Params(options=oracle.OPT_DUAL | OPTIONS)
    rng = np.random.default_rng(9)
    ges = [(U[4] - 0.5 * (U[1] ** 2 + U[2] ** 2 + U[3] ** 2) / np.where(U[0] > 0, U[0], 1.0)) *
           rng.uniform(0.5, 1.5, U[0].shape) for U in patches]
    b = batch_from_patches(patches, dx, flags=flags)
    import torch
    b.ge = torch.from_numpy(np.concatenate([g.ravel() for g in ges])).to(b.device)
    for s in range(2):
        dt = 0.3 / max(oracle.cfl_rate(U, dx, P) for U in patches)
        for U, g in zip(patches, ges):
            oracle.step_periodic_dual(U, g, dx, dt, s, P)
        b.dt_dev.fill_(dt)
        ez.step(b, ez.Params(precision=ez.FP64, options=ez.OPT_DUAL | OPTIONS), s, b.dt_dev)
    for i, (G, O) in enumerate(zip(gpu_patches(b), patches)):
        for g, o in zip(G, O):
            assert np.array_equal(active(g), active(o))
        assert np.array_equal(active(b.patch_ge(i).cpu().numpy()), active(ges[i]))


@pytest.mark.parametrize("left", [(1.0, 1.0), (1e-37, 1e-41), (1e39, 1e38), (1e-60, 1e-30)])
@pytest.mark.parametrize("right", [(1.0, 1.0), (1e-37, 1e-41), (1e-45, 1e-45), (1e60, 1e20)])
def test_riemann_fp64_beyond_the_range_of_fp32(left, right):
    """Newton's stopping bound is first formed in FP32: states outside FP32's
    range (density and pressure scaled per side) take the FP64 bound."""
    import torch
    rng = np.random.default_rng(21)
    rl, ul, pl, rr, ur, pr = (rng.uniform(0.5, 2.0, 512) for _ in range(6))
    rl, pl, rr, pr = rl * left[0], pl * left[1], rr * right[0], pr * right[1]
    ul = (ul - 1.25) * np.sqrt(left[1] / left[0])
    ur = (ur - 1.25) * np.sqrt(right[1] / right[0])
    kw = dict(rho_floor=1e-300, p_floor=1e-300)
    o = oracle.riemann(rl, ul, pl, rr, ur, pr, oracle.Params(**kw))
    g = ez.riemann_solve(*[torch.from_numpy(a).cuda() for a in (rl, ul, pl, rr, ur, pr)],
                         ez.Params(precision=ez.FP64, **kw))
    for k in ("pstar", "ustar", "rho", "u", "p", "iters"):
        assert np.array_equal(g[k].cpu().numpy(), o[k], equal_nan=k != "iters"), k
