"""Order of the curvature sum in the training backward: a point's primal adjoint is its own term plus its
tangent rows' terms in the order of the rows, each addition rounded to FP32, in the pipelined kernel (r <= 28) as
in the feature-major one (r >= 29).  The sum is rounded to BF16 for the layers below, so another order shows in the
gradients far above FP32 rounding.

One point, and a network whose pre-activations are exact in any order of summation, so that the last hidden layer's
bias gradient is that sum: expected bit for bit.  The output adjoints come from the call's own gradients: features
whose activation is 1 on one row and 0 on the others carry them into the output layer's weight gradient."""
import numpy as np
import pytest

import synth.scenes as S

pytestmark = pytest.mark.gpu
W = 128


def _bf16(v):
    """Round to nearest even to 8 significand bits; and the distance to the nearest tie in units of the last bit."""
    m, e = np.frexp(v)
    q = m * 256
    return np.ldexp(np.rint(q) / 256, e), np.abs(np.abs(q - np.floor(q)) - 0.5)


@pytest.mark.parametrize("d,r", [(2, 2), (2, 28), (2, 29), (3, 2), (3, 28), (3, 29)])
def test_bias_gradient_is_the_ordered_sum(d, r):
    import torch
    from paper_2109_12390_gb300.decoder import Decoder
    from paper_2109_12390_gb300.train import Trainer
    rng = np.random.default_rng(10 * d + r)
    X = np.array([[0.5, 0.25, 0.75][:d]])
    lat = np.zeros((2, r))
    lat[1, 0] = 1.0                                       # JVP direction: +-1 along latent 0
    x, v, F = rng.normal(size=(2, d)), rng.normal(size=(2, d)), rng.normal(size=(2, d, d))
    dev = lambda a, *s: torch.from_numpy(np.ascontiguousarray(a.reshape(*s), np.float32)).cuda()  # noqa: E731
    snaps = dict(dim=d, n_inst=1, inst_offsets=np.array([0, 1], np.int64), X=dev(X, 1, d), n_snap=2,
                 snap_inst=np.zeros(2, np.int32), snap_next=np.array([1, 0], np.int32), x=dev(x, 2, d), v=dev(v, 2, d),
                 F=dev(F, 2, d * d))
    p = S.xavier_decoder(0, d, r, W, 2, 0)
    make = lambda: Trainer(Decoder.from_params(p), snaps, lambda_F=1.0, lambda_v=1.0, dt_snap=1.0,  # noqa: E731
                           batch=1, total_steps=10, latents0=lat.astype(np.float32))
    s = int(make().gradients()[2][0])                     # the snapshot that the first step draws
    u = lat[1 - s] - lat[s]
    # layer 0: positive pre-activations, a few bits each; feature k < d + 1 passes input k on
    W0, b0 = np.zeros((W, d + r)), np.full(W, 4.0)
    W0[:, :d + 1] = rng.integers(-2, 3, size=(W, d + 1)) * 0.5
    W0[:d + 1, :d + 1] = np.eye(d + 1)
    a0 = W0 @ np.concatenate([X[0], lat[s]]) + b0
    t0 = np.stack([W0[:, k] for k in range(d)] + [W0[:, d:] @ u])          # tangent and JVP rows
    # layer 1: chosen pre-activations, most of them negative; feature k < d + 1 is zero but for tangent row k
    W1 = rng.integers(-16, 17, size=(W, W)) / 64.0
    W1[:d + 1] = np.eye(W)[:d + 1]
    z1 = np.where(rng.random(W) < 0.1, 0.5, -rng.integers(64, 512, size=W) / 256.0)
    z1[:d + 1] = 0.0
    b1 = z1 - W1 @ a0
    zd = t0 @ W1.T                                                            # (d + 1, W)
    Wo = rng.choice([-1.0, 1.0], size=(d, W)) * 0.5 ** rng.integers(0, 4, size=(d, W))
    p.W[:], p.b[:] = [W0, W1, Wo], [b0, b1, np.zeros(d)]
    assert all(np.array_equal(a, a.astype(np.float32)) for a in p.W + p.b)
    tr = make()
    g, _, bs, _, _ = tr.gradients()
    assert bs[0] == s and tr.status() == 0
    at = np.cumsum([W * (d + r), W, W * W, W, d * W])
    gb1, gWo, gbo = g[at[2]:at[3]], g[at[3]:at[4]].reshape(d, W), g[at[4]:]
    ybar = np.stack([gbo] + [gWo[:, k] for k in range(d)] + [gWo[:, d] * u[0]])   # (row, output)
    assert np.all(ybar != 0)

    f32 = np.float32
    hb = np.stack([ybar[:, i:i + 1].astype(np.float64) * Wo[i] for i in range(d)])  # exact products
    h = hb[0].astype(f32)
    for i in range(1, d):
        h = (h.astype(np.float64) + hb[i]).astype(f32)    # (row, feature), one rounding per output
    neg = z1 < 0
    slope, m0 = _bf16(np.exp(z1))
    act, m1 = _bf16(np.exp(z1) * zd)
    want = (np.where(neg, slope, 1.0) * h[0]).astype(f32)
    for k in range(d + 1):
        want = want + (np.where(neg, act[k], 0.0) * h[1 + k]).astype(f32)
    # the GPU's exponential is within a few FP32 units: leave out what lies at a rounding to BF16
    sure = (~neg) | ((m0 > 2.0 ** -9) & np.all((m1 > 2.0 ** -9) | (zd == 0), axis=0))
    assert sure.sum() > 100
    np.testing.assert_array_equal(gb1[sure], want[sure])
