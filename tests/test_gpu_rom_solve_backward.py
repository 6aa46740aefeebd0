"""Backward error of the velocity projection's solve, which does not grow with the condition of J^T J: with fewer rows
than unknowns (the FP64 Cholesky fallback) the forward bound of tests/test_gpu_rom_solve_sizes.py allows errors of
several percent.  The residual |A x - J^T b| is held to four times 2^-40 of tr(A) |x| + ||J|^T |b||: the assembly of
A, that of J^T b and the last correction of the refinement are each within 2^-40, x comes back as a difference of
FP64 velocities.  The step raises no status."""
import numpy as np
import pytest

from test_gpu_rom import _elu_setup
from test_gpu_rom_solve_sizes import _rhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,k", [(8, 33), (16, 17), (17, 9), (31, 12), (32, 256), (32, 6)])
def test_backward_error(r, k):
    import torch
    from paper_2109_12390_gb300.decoder import PRIMAL
    from paper_2109_12390_gb300.rom import ROM
    sc, p, dec, rom, rs, xh, vh, xp = _elu_setup(seed=r + k, side=32, r=r, k=k, projection=1)
    rom.close()
    dec.set_precision(True)
    rom = ROM.from_scene(dec, sc, n_samples=k, seed=r + k, projection=1)
    rom.set_state(xh, vh, xp, 0)
    rom.step(1)
    dbg = rom.debug()
    Xs = np.ascontiguousarray(sc.x[dbg["samples"]], np.float32)
    out = dec.eval(torch.from_numpy(Xs).cuda(), torch.from_numpy(xh.astype(np.float32)[None]).cuda(),
                   [PRIMAL] + [dec.dxhat(j) for j in range(r)]).cpu().numpy()
    J32 = np.stack(out[1:], -1).reshape(-1, r)
    b = _rhs(dbg["v_trial"].reshape(-1), J32, vh)
    J = J32.astype(np.float64)
    A = J.T @ J
    tr = np.trace(A)
    A = A + 1e-10 * tr / r * np.eye(r)
    x = rom.get_state()[1] - vh
    scale = tr * np.linalg.norm(x) + np.linalg.norm(np.abs(J).T @ np.abs(b))
    assert np.linalg.norm(A @ x - J.T @ b) < 4 * 2.0 ** -40 * scale + 2.0 ** -52 * tr * np.linalg.norm(vh)
    assert rom.status() == 0
    rom.close()
    dec.close()
