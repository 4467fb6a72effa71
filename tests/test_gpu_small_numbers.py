"""Small numbers beside large ones: a colour that reaches the result through a small
link element alone, or that is small by itself, keeps the digits of its storage."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
from tests.wd_testutil import parity_mask, parity_sites

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 8, 10)
VOL = int(np.prod(DIMS))


def _dslash(U, psi, prec, recon, dagger=False, **load):
    import paper_0911_3191_gb300 as m
    wd = m.WilsonDirac(DIMS)
    wd.load_gauge(U, recon=recon, **load)
    f, o = wd.upload(psi, prec, parity=0), wd.new_field(prec)
    wd.dslash(o, f, 1, dagger, prec)
    out = wd.download(o, prec, parity=1)
    wd.close()
    return out


@pytest.mark.parametrize("prec,unit", [(1, 2.0 ** -24), (4, 2.0 ** -8)])
@pytest.mark.parametrize("recon", [12, 18])
@pytest.mark.parametrize("small", [3e-12, 1e-20, 1e-25])
def test_small_link_elements_of_derived_links(prec, unit, recon, small):
    """FP32 and bf16 hold 1e-25 as well as 1: colour 0 of the result comes from colour 1 of the source through
    elements of that size."""
    U = np.tile(np.eye(3, dtype=np.complex128), (VOL, 4, 1, 1))
    rng = np.random.default_rng(31)
    e = small * rng.uniform(0.5, 1.0, (VOL, 4)) * np.exp(2j * np.pi * rng.random((VOL, 4)))
    U[:, :, 0, 1], U[:, :, 1, 0] = e, -e.conj()
    psi = li.gaussian_spinor(DIMS, 2600) * parity_mask(DIMS, 0)
    psi[:, :, 0] = 0
    got, want = _dslash(U, psi, prec, recon)[:, :, 0], oracle.dslash(psi, U, DIMS, out_parity=1)[:, :, 0]
    # 16 terms of at most small * max|psi|; FP32: at most 16 roundings of each, bf16: source, link and result rounded
    terms = 16 * small * np.abs(psi).max()
    bound = (16 if prec == 1 else 4) * unit * terms
    odd = parity_sites(DIMS, 1)
    assert np.abs(want[odd]).max() > 4 * bound
    assert np.abs(got - want)[odd].max() <= bound
