"""FP32 decoder calls on the tensor cores (three-way BF16 split) at the edges of their tiles.

Rows reach a 128-row tile in (point, kind) order, 32 or 31 per lane group; the sizes put the last row
just before, on and just after a lane group, a tile and a grid of tiles, for one to 40 rows per
point.  Oracle: FP64, 1e-5 relative (the bound of the FP32 path; the split products keep 2^-23 of each
term).  The same rows inside a call with a mixed row run on the CUDA cores (the general path): the
two agree within the sum of their bounds.
"""
import numpy as np
import pytest

import oracle.decoder as OD
import synth.scenes as S

pytestmark = pytest.mark.gpu
TOL = 1e-5


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


def _setup(d, r, n, act=OD.ELU, n_hidden=5, seed=7):
    import torch
    from paper_2109_12390_gb300.decoder import Decoder
    p = S.xavier_decoder(seed, d, r, 128, n_hidden, act, X_min=np.full(d, 0.3), X_range=np.full(d, 0.3),
                         out_shift=np.full(d, 0.5), out_scale=np.full(d, 0.1), bias_scale=0.2)
    dec = Decoder.from_params(p)
    dec.set_precision(1)
    rng = np.random.default_rng(seed + n)
    X = (0.3 + 0.3 * rng.uniform(size=(n, d))).astype(np.float32)
    lat = rng.normal(scale=0.7, size=(3, r)).astype(np.float32)
    u = (0.02 * rng.normal(size=(3, r))).astype(np.float32)
    idx = rng.integers(0, 3, size=n).astype(np.int32)
    g = [torch.from_numpy(a).cuda() for a in (X, lat, idx, u)]
    return p, dec, X.astype(np.float64), lat.astype(np.float64)[idx], u.astype(np.float64)[idx], g


def _kinds(dec, name, d, r):
    from paper_2109_12390_gb300.decoder import JVP, PRIMAL, SECANT, dX
    return {"primal": [PRIMAL], "velocity": [PRIMAL] + [dX(k) for k in range(d)] + [JVP],
            "gradient": [PRIMAL] + [dX(k) for k in range(d)],
            "jacobian": [PRIMAL] + [dec.dxhat(j) for j in range(r)],
            "secant": [PRIMAL, dX(0), SECANT]}[name]


def _reference(p, X, xh, u, name, d, r):
    g, JX, Jq = OD.jacobians(p, X, xh)
    rows = {"primal": [], "gradient": [JX[..., k] for k in range(d)],
            "velocity": [JX[..., k] for k in range(d)] + [OD.jvp_latent(p, X, xh, u)[1]],
            "jacobian": [Jq[..., j] for j in range(r)], "secant": [JX[..., 0], OD.decode(p, X, xh + u) - g]}[name]
    return [g - 0.5] + rows


@pytest.mark.parametrize("name,d,r,n", [
    ("primal", 2, 16, 1), ("primal", 3, 37, 127), ("primal", 2, 4, 128), ("primal", 3, 16, 129),
    ("gradient", 2, 8, 10), ("gradient", 2, 13, 11), ("gradient", 3, 16, 32), ("gradient", 3, 16, 33),
    ("velocity", 3, 16, 25), ("velocity", 2, 16, 31), ("jacobian", 2, 16, 8), ("jacobian", 3, 32, 5),
    ("jacobian", 2, 38, 7), ("secant", 2, 16, 42), ("secant", 3, 8, 83)])
def test_tile_edges_against_the_oracle(name, d, r, n):
    p, dec, X, xh, u, (Xg, latg, idxg, ug) = _setup(d, r, n)
    dec.set_concurrency(8)   # secant rows take the tensor cores too
    out = dec.eval(Xg, latg, _kinds(dec, name, d, r), lat_idx=idxg, dirs=ug).cpu().numpy().astype(np.float64)
    assert dec.status() == 0
    out[0] -= 0.5
    for k, (a, b) in enumerate(zip(out, _reference(p, X, xh, u, name, d, r))):
        assert rel(a, b) < TOL, (name, k)


@pytest.mark.parametrize("name,d,n", [("velocity", 2, 8192), ("velocity", 3, 15000), ("gradient", 2, 40001),
                                      ("secant", 2, 31000), ("gradient", 3, 150001)])
def test_many_tiles_against_the_general_path(name, d, n):
    """One tile per CTA, two per CTA and several passes with a partial last one, against the CUDA-core
    kernel (the same rows in a call with a mixed row)."""
    from paper_2109_12390_gb300.decoder import JVP, dX, mixed
    p, dec, X, xh, u, (Xg, latg, idxg, ug) = _setup(d, 16, n)
    kinds = _kinds(dec, name, d, 16)
    got = dec.eval(Xg, latg, kinds, lat_idx=idxg, dirs=ug)
    more = kinds + ([] if JVP in kinds else [JVP]) + [mixed(dX(0))]
    want = dec.eval(Xg, latg, more, lat_idx=idxg, dirs=ug)[:len(kinds)]
    assert dec.status() == 0
    got, want = got.double(), want.double()
    got[0] -= 0.5
    want[0] -= 0.5
    for k in range(len(kinds)):
        assert float((got[k] - want[k]).norm() / want[k].norm()) < 2 * TOL, (name, k)
    pick = np.r_[0:64, n // 2:n // 2 + 64, n - 64:n]
    for a, b in zip(got, _reference(p, X[pick], xh[pick], u[pick], name, d, 16)):
        assert rel(a[pick].cpu().numpy(), b) < TOL


@pytest.mark.parametrize("act,n_hidden", [(OD.IDENTITY, 5), (OD.ELU, 2), (OD.ELU, 4)])
def test_other_depths_and_identity(act, n_hidden):
    p, dec, X, xh, u, (Xg, latg, idxg, ug) = _setup(2, 16, 500, act, n_hidden)
    out = dec.eval(Xg, latg, _kinds(dec, "velocity", 2, 16), lat_idx=idxg, dirs=ug).cpu().numpy().astype(np.float64)
    out[0] -= 0.5
    for a, b in zip(out, _reference(p, X, xh, u, "velocity", 2, 16)):
        assert rel(a, b) < TOL
