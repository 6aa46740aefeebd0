"""Full-order step on both sides of the sizes where the work items and CTAs change (csrc/mpm_items.cuh), for one
body and for several, on grids of odd block counts.  Bound: as tests/test_gpu_mpm.py (1e-5, or the oracle's own FP32
sensitivity)."""
import numpy as np
import pytest

import synth.scenes as S
from test_gpu_mpm_work_items import _run

pytestmark = pytest.mark.gpu


def _side(per_sm, n_inst, up):
    """Side of n_inst square bodies that hold just at most (up: just more than) per_sm particles per SM."""
    import torch
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    return int((n / n_inst) ** 0.5) + up


@pytest.mark.parametrize("n_inst,up", [(1, 0), (1, 1), (16, 0), (16, 1)])
def test_2d_cta_width(n_inst, up):
    side = _side(896, n_inst, up)
    sc = S.batch_2d(seed=side, n_inst=n_inst, fixed_side=side, n_grid=(side // 2 + 24) // 8 * 8 + 8, origin_y=0.06)
    sc.F = S.random_deformation(np.random.default_rng(side), sc.n_particles, 2, 0.02)
    _run(sc, 2)


@pytest.mark.parametrize("per_sm,n_inst,up", [(128, 1, 0), (128, 3, 1), (336, 1, 0), (336, 16, 1)])
def test_2d_item_bound(per_sm, n_inst, up):
    side = _side(per_sm, n_inst, up)
    sc = S.batch_2d(seed=side, n_inst=n_inst, fixed_side=side, n_grid=(side // 2 + 24) // 8 * 8 + 8, origin_y=0.06)
    sc.material = 1
    sc.F = S.random_deformation(np.random.default_rng(side), sc.n_particles, 2, 0.02)
    _run(sc, 2)


@pytest.mark.parametrize("material,up", [(0, 0), (1, 1)])
def test_3d_item_bound(material, up):
    import torch
    side = int((672 * torch.cuda.get_device_properties(0).multi_processor_count) ** (1 / 3)) + up
    sc = S.cube_3d(seed=side, side=side, n_grid=(side // 2 + 16) // 4 * 4 + 4, bottom=0.06)
    sc.material = material
    sc.F = S.random_deformation(np.random.default_rng(side), sc.n_particles, 3, 0.02)
    sc.dt = 1e-5
    _run(sc, 2)
