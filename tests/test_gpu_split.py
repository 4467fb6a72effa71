"""The dslash on both sides of the line between the two thread layouts: four warps
per 32 sites up to one block of 128 sites per SM (152 SMs: 19456 sites of a
parity), one thread per site above; neither lattice fills its last block."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
from tests.wd_testutil import TOL, parity_mask, rel_err

pytestmark = pytest.mark.gpu

_cache = {}


def _fields(dims):
    if dims not in _cache:
        _cache[dims] = (li.gauge(dims, 0.5, 1500), li.gaussian_spinor(dims, 2500))
    return _cache[dims]


@pytest.mark.parametrize("dims", [(12, 14, 10, 22), (12, 14, 10, 24)])  # 18480 and 20160 sites of a parity
@pytest.mark.parametrize("prec", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("temporal,anti,dagger,parity", [(False, True, False, 0), (True, True, True, 1)])
def test_both_sides_of_the_line(dims, prec, temporal, anti, dagger, parity):
    import paper_0911_3191_gb300 as wdp
    U, psi = _fields(dims)
    wd = wdp.WilsonDirac(dims, t_antiperiodic=anti)
    wd.load_gauge(U, recon=18, temporal_gauge=temporal)
    f, x = wd.upload(psi, prec, parity=1 - parity), wd.upload(psi, prec, parity=parity)
    o, o2 = wd.new_field(prec), wd.new_field(prec)
    wd.dslash(o, f, parity, dagger, prec)
    wd.dslash_xpay(o2, f, x, -0.37, parity, dagger, prec)
    d = oracle.dslash(psi * parity_mask(dims, 1 - parity), U, dims, dagger=dagger, out_parity=parity, tbc_anti=anti)
    tol = 2e-13 if temporal and prec == 0 else TOL[prec]  # the rotations by products of up to T links
    assert rel_err(wd.download(o, prec, parity=parity), d) <= tol
    want = psi * parity_mask(dims, parity) - 0.37 * d
    assert rel_err(wd.download(o2, prec, parity=parity), want) <= tol
    wd.close()


@pytest.mark.parametrize("dims", [(4, 16, 16, 38), (4, 16, 16, 40), (2, 6, 10, 14), (8, 8, 8, 38), (8, 8, 8, 40)])
@pytest.mark.parametrize("prec", [0, 1, 2])
def test_solvers_on_both_sides_of_the_small_shapes(dims, prec):
    """Up to 128 sites per SM (19456 with 152 SMs, the first lattice) the site kernels run
    in blocks of 128, beyond in blocks of 256; 840 sites fill neither.  The last two
    lattices lie on the two sides of 64 sites per SM (9728), up to which the FP64
    dslash with a fused reduction is the one of four warps per 32 sites."""
    import paper_0911_3191_gb300 as m
    U = li.gauge(dims, 0.4, 1030)
    b = li.gaussian_spinor(dims, 1031)
    wd = m.WilsonDirac(dims)
    wd.load_gauge(U)
    for solver in (m.BICGSTAB, m.CGNR):
        x = np.zeros_like(b)
        info = wd.solve(x, b, 0.115, tol=1e-10, solver=solver, inner_precision=prec)
        rel = oracle.true_residual(x, b, U, dims, 0.115)
        assert info.status == 0 and rel <= 1e-10, (solver, info, rel)
    wd.close()
