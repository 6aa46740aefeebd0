"""After optimisation steps every form of the weights that a kernel reads belongs to the new parameters: a decoder
that was trained gives the bits of a new one made from its parameters, in every precision and on every path."""
import numpy as np
import pytest

import synth.scenes as S
from test_gpu_train_tiles import _store

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,r,n_hidden", [(2, 16, 5), (3, 28, 2), (3, 30, 5)])
def test_every_form_follows_the_training(d, r, n_hidden):
    import torch
    from paper_2109_12390_gb300.decoder import JVP, PRIMAL, Decoder, dX, mixed
    from paper_2109_12390_gb300.train import Trainer
    snaps, host = _store(d, 4, 5)
    X = host["X"]
    p = S.xavier_decoder(3, d, r, 128, n_hidden, 0, X_min=X.min(0), X_range=X.max(0) - X.min(0), out_shift=X.mean(0),
                         out_scale=np.full(d, 0.1), bias_scale=0.2)
    dec = Decoder.from_params(p)
    tr = Trainer(dec, snaps, dt_snap=0.01, batch=500, total_steps=10, lr0=1e-2, lr1=1e-2)
    tr.step(3)
    params, norm = np.empty(dec.n_params, np.float32), np.empty(4 * d, np.float32)
    dec.get_params(params, norm)
    torch.cuda.synchronize()
    assert np.abs(params - p.flat().astype(np.float32)).max() > 1e-3
    new = Decoder(d, r, 128, n_hidden, 0)
    new.set_params(params, norm)
    g = torch.Generator(device="cuda").manual_seed(1)
    Xg = torch.rand(300, d, generator=g, device="cuda")
    lat, u = torch.randn(2, 1, r, generator=g, device="cuda")
    for precision in (0, 1, 2):
        for kinds in ([PRIMAL], [PRIMAL, dX(0), JVP], [PRIMAL, dX(0), JVP, mixed(dX(0))]):
            out = []
            for k in (dec, new):
                k.set_precision(precision)
                out.append(k.eval(Xg, lat, kinds, dirs=u))
                assert k.status() == 0
            assert torch.equal(*out), (precision, kinds)
