"""Which kernel small FP32 calls with secant rows take, seen by their bits: decoder_f32 and decoder_tc3 round
differently, and each gives a row the same bits in every tiling."""
import numpy as np
import pytest

from test_gpu_decoder_fp32_tiles import TOL, _kinds, _reference, _setup, rel

pytestmark = pytest.mark.gpu


def _secants(n, concurrency, d=2, r=16, m=11):
    from paper_2109_12390_gb300.decoder import PRIMAL, secant_dir
    import torch
    p, dec, _, _, _, (Xg, latg, _, _) = _setup(d, r, n)
    dirs = 1e-3 * torch.randn(1, 1, r, generator=torch.Generator().manual_seed(1)) * 0.5 ** torch.arange(m)[None, :, None]
    dec.set_concurrency(concurrency)
    out = dec.eval(Xg, latg[:1].contiguous(), [PRIMAL] + [secant_dir(k) for k in range(m)],
                   dirs=dirs.reshape(m, r).cuda().contiguous())
    assert dec.status() == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [1, 16, 40])
def test_small_secant_calls_of_concurrent_callers_stay_on_the_cuda_cores(n):
    """12 n rows fit a small tile per SM of one of eight callers' share: as fast as a lone caller's, and its bits."""
    np.testing.assert_array_equal(_secants(n, 8), _secants(n, 1))


def test_larger_ones_take_the_tensor_cores():
    lone, shared = _secants(300, 1), _secants(300, 8)
    assert np.any(lone != shared)
    assert rel(shared, lone) < 2 * TOL


@pytest.mark.parametrize("d,r,n", [(2, 16, 42), (3, 8, 83)])
def test_secant_tile_edges_on_the_tensor_cores(d, r, n):
    p, dec, X, xh, u, (Xg, latg, idxg, ug) = _setup(d, r, n)
    dec.set_concurrency(1000)   # a share of one SM: every call of more than 31 rows
    out = dec.eval(Xg, latg, _kinds(dec, "secant", d, r), lat_idx=idxg, dirs=ug).cpu().numpy().astype(np.float64)
    assert dec.status() == 0
    out[0] -= 0.5
    for k, (a, b) in enumerate(zip(out, _reference(p, X, xh, u, "secant", d, r))):
        assert rel(a, b) < TOL, k
