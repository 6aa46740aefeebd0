"""Normal-equations solve of the velocity projection at the latent dimensions where its layout changes
(one element of the inverse per thread up to 16, four above), with row counts that leave a partial tile, and
with fewer rows than unknowns (the FP32 inverse does not converge; FP64 Cholesky).  As in
tests/test_gpu_rom.py: within 2^-40 cond(J^T J) of an FP64 solve on the GPU's own Jacobian
and FP32 right-hand side."""
import numpy as np
import pytest

from test_gpu_rom import _elu_setup, rel

pytestmark = pytest.mark.gpu
f32 = np.float32


def _rhs(v_trial, J, vh):
    """The FP32 right-hand side v_trial - J vhat as the kernel defines it: a Dot2 of J's rows with the
    hi / lo parts of vhat, subtracted in FP32."""
    sh = np.zeros(len(J), f32)
    sc = np.zeros(len(J), f32)
    for c in range(J.shape[1]):
        hi = f32(vh[c])
        for y in (hi, f32(vh[c] - float(hi))):
            exact = J[:, c].astype(np.float64) * float(y)
            p = exact.astype(f32)
            t = sh + p
            z = t - sh
            sc = sc + (((sh - (t - z)) + (p - z)) + (exact - p).astype(f32))
            sh = t
    return ((v_trial.astype(f32) - sh) - sc).astype(np.float64)


@pytest.mark.parametrize("r,k", [(1, 3), (4, 16), (8, 33), (15, 64), (16, 17), (17, 48), (31, 100), (32, 256), (32, 6)])
def test_velocity_solve(r, k):
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
    A = A + 1e-10 * np.trace(A) / r * np.eye(r)
    ref = np.linalg.solve(A, J.T @ b)
    _, vh1, _, _ = rom.get_state()
    assert rel(vh1 - vh, ref) < max(2.0 ** -40 * np.linalg.cond(A), 1e-12)
    rom.close()
    dec.close()
