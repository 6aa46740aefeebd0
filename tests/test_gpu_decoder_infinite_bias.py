"""A bias of minus infinity switches a hidden unit off: its activation is -1 and its derivatives are 0, as with any
bias far below zero.  No row of a call, derivative rows included, may turn it into NaN."""
import numpy as np
import pytest

from test_gpu_decoder_fp32_tiles import _kinds, _setup
from test_gpu_train_tiles import _store

pytestmark = pytest.mark.gpu
UNITS = [(0, 3), (0, 77), (1, 40), (4, 127)]


def _params(p, value):
    b = [v.copy() for v in p.b]
    for l, f in UNITS:
        b[l][f] = value
    return np.concatenate([np.concatenate([w.reshape(-1), v]) for w, v in zip(p.W, b)]).astype(np.float32)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name,n", [("primal", 200), ("velocity", 200), ("jacobian", 40), ("secant", 90),
                                    ("velocity", 25000)])
def test_rows_are_those_of_a_unit_far_below_zero(precision, name, n):
    import torch
    p, dec, _, _, _, (Xg, latg, idxg, ug) = _setup(2, 16, n)
    dec.set_precision(precision)
    dec.set_concurrency(1000)   # FP32 secant rows on the tensor cores too
    norm = np.concatenate([p.X_min, p.X_range, p.out_shift, p.out_scale])
    out = []
    for value in (-np.inf, -1e4):
        dec.set_params(_params(p, value), norm)
        out.append(dec.eval(Xg, latg, _kinds(dec, name, 2, 16), lat_idx=idxg, dirs=ug))
        assert dec.status() == 0
    assert bool(torch.isfinite(out[1]).all())
    assert torch.equal(*out)


@pytest.mark.parametrize("d", [2, 3])
def test_training_gradients(d):
    from paper_2109_12390_gb300.train import Trainer
    p, dec, _, _, _, _ = _setup(d, 8, 10)
    snaps, _ = _store(d, 4, 5)
    norm = np.concatenate([p.X_min, p.X_range, p.out_shift, p.out_scale])
    lat = 0.5 * np.random.default_rng(3).normal(size=(4, 8)).astype(np.float32)
    got = []
    for value in (-np.inf, -1e4):
        dec.set_params(_params(p, value), norm)
        tr = Trainer(dec, snaps, dt_snap=0.01, batch=700, total_steps=10, latents0=lat)
        got.append(tr.gradients()[:2])
        assert tr.status() == 0
    for a, b in zip(*got):      # sums of the same terms in another order of the atomics
        assert np.all(np.isfinite(b))
        assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
