"""Encoder gradients at the sizes where the backward's launch changes: the shortest input, subsets whose layers leave
room for four, two and one CTA per SM, and more snapshots than CTAs.  Bound: as tests/test_gpu_encoder.py (1e-4 per
parameter block, given the GPU's own latent gradients)."""
import numpy as np
import pytest

import oracle.decoder as OD
import oracle.encoder as OE
import synth.scenes as S
from test_gpu_train import _store, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_sub,r,J,side", [(16, 1, 3, 8), (40, 13, 700, 8), (900, 8, 5, 32), (2200, 32, 3, 48),
                                            (4000, 16, 2, 64)])
def test_backward(n_sub, r, J, side):
    from paper_2109_12390_gb300.decoder import Decoder
    from paper_2109_12390_gb300.train import Trainer
    snaps, host = _store(2, n_inst=1, J=J, side=side, seed=n_sub)
    X = host["X"]
    p = S.xavier_decoder(1, 2, r, 128, 5, OD.ELU, X_min=X.min(0), X_range=X.max(0) - X.min(0), out_shift=X.mean(0),
                         out_scale=np.full(2, 0.1), bias_scale=0.2)
    dec = Decoder.from_params(p)
    tr = Trainer(dec, snaps, lambda_F=3.0, lambda_v=0.05, dt_snap=0.01, batch=1000, total_steps=5, encoder_subset=n_sub,
                 seed=7)
    vec, ss = tr.encoder_params()
    enc = OE.unflatten(OE.xavier_encoder(0, 2, r, n_sub), vec.astype(np.float64))
    enc.shift, enc.scale = ss[:2].astype(np.float64), ss[2:].astype(np.float64)
    u = OE.encoder_input(enc, host["x"][:, OE.subset_ids(len(X), n_sub)].astype(np.float32).astype(np.float64))
    _, gl, _, _, _ = tr.gradients()
    ge = tr.last_encoder_gradients
    ref = OE.vjp(enc, u, gl.astype(np.float64))
    o = 0
    for l in range(len(enc.conv_w)):
        assert rel(ge[o:o + 6], ref["conv_w"][l]) < 1e-4, ("conv w", l)
        o += 7
    for key in ("W1", "b1", "W2", "b2"):
        n = ref[key].size
        assert rel(ge[o:o + n], ref[key].ravel()) < 1e-4, key
        o += n
    assert o == len(ge)
