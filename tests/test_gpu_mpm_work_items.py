"""Full-order step at the sizes where its work items and CTAs change: below and above one 2D block of
256 particles per SM (CTAs of 256 or 128 threads), 3D blocks in one item or split in two or more, and
large deformations that take several iterations of the rotation and of the eigen-decomposition.
Bound: as tests/test_gpu_mpm.py (1e-5, or the oracle's own FP32 sensitivity)."""
import numpy as np
import pytest

import fp32_bounds as FB
import oracle.mpm as OM
import synth.scenes as S

pytestmark = pytest.mark.gpu


def _run(sc, steps):
    from paper_2109_12390_gb300.mpm import MPM
    ctx = MPM.from_scene(sc)
    ctx.load_numpy(sc.x, sc.v, sc.F, sc.C)
    ctx.step(steps)
    assert ctx.status() == 0
    ref = sc.copy()
    OM.step(ref, steps)
    errs = FB.fom_errors(*ctx.read_numpy(), ref)
    bounds, _ = FB.fom_bounds(sc, ref, steps)
    assert all(errs[k] < bounds[k] for k in errs), (errs, bounds)


@pytest.mark.parametrize("side,material", [(7, 0), (150, 0), (196, 1), (199, 0), (230, 2)])
def test_2d_sizes(side, material):
    sc = S.batch_2d(seed=side, n_inst=1, fixed_side=side, n_grid=128, origin_y=0.03)
    sc.material = material
    sc.F = S.random_deformation(np.random.default_rng(side), sc.n_particles, 2, 0.02)
    _run(sc, 4)


@pytest.mark.parametrize("side,material,scale", [(5, 1, 0.3), (34, 2, 0.02), (34, 1, 0.3), (44, 1, 0.02)])
def test_3d_sizes(side, material, scale):
    sc = S.cube_3d(seed=side, side=side, n_grid=64, bottom=0.06)
    sc.material = material
    sc.F = S.random_deformation(np.random.default_rng(side), sc.n_particles, 3, scale)
    sc.dt = 1e-5
    _run(sc, 3)
