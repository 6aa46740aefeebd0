"""BF16 decoder calls over many tiles: every row of decoder_bf16, over one and several passes of its two tile
slots with a partial last one, against the same rows inside a call with a mixed row, which the general kernel takes.
The two kernels' arithmetic is the same in the same order, so the rows agree bit for bit (tests/test_gpu_decoder.py
holds both against the oracle)."""
import pytest

from test_gpu_decoder_fp32_tiles import _kinds, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,d,r,n", [
    ("primal", 3, 16, 100), ("primal", 2, 13, 150001), ("gradient", 3, 28, 33), ("gradient", 3, 16, 50003),
    ("velocity", 2, 16, 10000), ("velocity", 2, 7, 40001), ("velocity", 3, 16, 30011), ("jacobian", 2, 16, 7),
    ("jacobian", 2, 16, 9001), ("jacobian", 3, 27, 5003), ("secant", 2, 16, 11), ("secant", 2, 16, 45001),
    ("secant", 3, 28, 20011)])
def test_rows_equal_the_general_kernels(name, d, r, n):
    import torch
    from paper_2109_12390_gb300.decoder import JVP, dX, mixed
    p, dec, X, xh, u, (Xg, latg, idxg, ug) = _setup(d, r, n)
    dec.set_precision(0)
    kinds = _kinds(dec, name, d, r)
    got = dec.eval(Xg, latg, kinds, lat_idx=idxg, dirs=ug)
    more = kinds + [k for k in (dX(0), JVP) if k not in kinds] + [mixed(dX(0))]
    want = dec.eval(Xg, latg, more, lat_idx=idxg, dirs=ug)[:len(kinds)]
    assert dec.status() == 0
    assert torch.equal(got, want)
