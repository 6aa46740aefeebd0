"""Minibatch gradients at the edges of the training kernels' tiles (32 or 24 points in 2D and 3D, eight or six per
lane group), below and above two tiles per SM, at the largest latent dimension of the pipelined kernels (28) and
the smallest of the feature-major ones (29), and with the linear activation, against the FP64 oracle.
Bounds: 2e-2 norm-wise as tests/test_gpu_train.py; 5e-2 for the batches below 512 points, where the roundings of
the operands to BF16 (2^-9 each, six layers forward and back: 2.3e-2 if none cancel) are hardly averaged."""
import numpy as np
import pytest

import oracle.decoder as OD
import synth.scenes as S
from test_gpu_train import _oracle_batch, rel

pytestmark = pytest.mark.gpu


def _store(d, J, seed):
    import torch
    rng = np.random.default_rng(seed)
    sc = S.batch_2d(seed=seed, n_inst=1, fixed_side=8) if d == 2 else S.cube_3d(seed=seed, side=5)
    X, P = sc.x, len(sc.x)
    host = dict(X=X, P=P, J=J, x=X[None] + 0.01 * rng.normal(size=(J, P, d)), v=rng.normal(size=(J, P, d)),
                F=np.eye(d)[None, None] + 0.05 * rng.normal(size=(J, P, d, d)))
    dev = lambda a, *s: torch.from_numpy(np.ascontiguousarray(a.reshape(*s), np.float32)).cuda()
    return dict(dim=d, n_inst=1, inst_offsets=np.array([0, P], np.int64), X=dev(X, P, d), n_snap=J,
                snap_inst=np.zeros(J, np.int32), snap_next=np.array([*range(1, J), -1], np.int32),
                x=dev(host["x"], -1, d), v=dev(host["v"], -1, d), F=dev(host["F"], -1, d * d)), host


@pytest.mark.parametrize("d,r,batch,act", [(2, 8, 1, OD.ELU), (2, 16, 31, OD.ELU), (2, 5, 33, OD.ELU),
                                           (2, 28, 1000, OD.ELU), (2, 29, 1000, OD.ELU), (2, 16, 9729, OD.ELU),
                                           (2, 16, 700, OD.IDENTITY), (3, 1, 23, OD.ELU), (3, 16, 25, OD.ELU),
                                           (3, 28, 601, OD.ELU), (3, 29, 601, OD.ELU), (3, 7, 8000, OD.IDENTITY)])
def test_gradients(d, r, batch, act):
    from paper_2109_12390_gb300.decoder import Decoder
    from paper_2109_12390_gb300.train import Trainer
    tol = 2e-2 if batch >= 512 else 5e-2
    snaps, host = _store(d, 6, d + r + batch)
    X = host["X"]
    p = S.xavier_decoder(batch, d, r, 128, 5, act, X_min=X.min(0), X_range=X.max(0) - X.min(0),
                         out_shift=X.mean(0), out_scale=np.full(d, 0.1), bias_scale=0.2)
    dec = Decoder.from_params(p)
    lat = 0.5 * np.random.default_rng(3).normal(size=(6, r)).astype(np.float32)
    tr = Trainer(dec, snaps, lambda_F=3.0, lambda_v=0.05, dt_snap=0.01, batch=batch, total_steps=10, latents0=lat)
    gp, gl, bs, bp, loss = tr.gradients()
    for l in range(len(p.W)):
        p.W[l] = p.W[l].astype(np.float32).astype(np.float64)
        p.b[l] = p.b[l].astype(np.float32).astype(np.float64)
    L, gW, gb, glat = OD.batch_loss_grads(p, lat.astype(np.float64), _oracle_batch(host, snaps, bs, bp),
                                          np.float32(0.01), 3.0, 0.05)
    assert loss == pytest.approx(L, rel=tol)
    ref = np.concatenate([np.concatenate([w.reshape(-1), b]) for w, b in zip(gW, gb)])
    assert rel(gp, ref) < tol
    k = 128 * (d + r)
    assert rel(gp[:k], ref[:k]) < tol
    assert rel(gl, glat) < tol
    assert tr.status() == 0
