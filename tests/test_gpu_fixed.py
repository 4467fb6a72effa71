"""The FP64 dslash in block fixed point (integer pipe) against the oracle, at the
edges of the numbers it takes: exponents that differ from site to site, zeros,
numbers outside its range, infinities, links it does not take."""
import numpy as np
import pytest

import lattice_inputs as li
import oracle
from tests.wd_testutil import parity_mask, parity_sites, rel_err, to_internal_basis

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 8, 10)
# each output is a sum of 8 hops x 2 terms x 3 complex products: the oracle's own
# FP64 rounding is at most about sqrt(96) x 2^-53, and the fixed-point sums, kept to
# 2^-55 of the largest neighbour component, add less
TOL_REL = 1.5e-15


def _wd():
    import paper_0911_3191_gb300 as wdp
    return wdp


def _apply(U, psi, recon, dagger=False, temporal=False, anti=False, parity=1):
    wdp = _wd()
    wd = wdp.WilsonDirac(DIMS, t_antiperiodic=anti)
    wd.load_gauge(U, recon=recon, temporal_gauge=temporal)
    f = wd.upload(psi, wdp.F64, parity=1 - parity)
    o = wd.new_field(wdp.F64)
    wd.dslash(o, f, parity, dagger, wdp.F64)
    out = wd.download(o, wdp.F64, parity=parity)
    wd.close()
    return out


@pytest.mark.parametrize("recon,temporal,dagger,anti", [(18, False, False, False), (12, False, True, True),
                                                        (18, True, True, False), (12, True, False, True)])
def test_site_exponents(recon, temporal, dagger, anti):
    """Sites of very different size: every output is right to the size of its largest neighbour."""
    rng = np.random.default_rng(11)
    U = li.gauge(DIMS, 0.7, 1400)
    psi = li.gaussian_spinor(DIMS, 2400) * np.exp2(rng.integers(-70, 70, size=(li.volume(DIMS), 1, 1)))
    psi[rng.random(li.volume(DIMS)) < 0.2] = 0.0
    psi[rng.random(psi.shape) < 0.1] *= 1e-30  # small components beside large ones
    src = psi * parity_mask(DIMS, 0)
    got = _apply(U, src, recon, dagger, temporal, anti)
    want = oracle.dslash(src, U, DIMS, dagger=dagger, out_parity=1, tbc_anti=anti)
    size = np.abs(src).max(axis=(1, 2)).reshape(DIMS[::-1])
    near = np.max([np.roll(size, s, axis=a) for a in range(4) for s in (1, -1)], axis=0).reshape(-1)
    err = np.abs(got - want).max(axis=(1, 2))
    odd = parity_sites(DIMS, 1)
    # 96 products of numbers at most 1 and 2 x near, each FP64 sum rounded at 2^-53 (both sides; the temporal
    # gauge rotates by products of up to T links on the way in and out)
    bound = (96 if not temporal else 400) * 2.0 ** -53 * 2 * near[odd]
    assert (err[odd] <= bound).all(), float(np.max(err[odd] / np.maximum(near[odd], 1e-300)))
    assert (err[odd][near[odd] == 0] == 0).all()


@pytest.mark.parametrize("scale", [2.0 ** -1000, 2.0 ** -840, 2.0 ** -828, 2.0 ** 860, 2.0 ** 876, 2.0 ** 1000])
@pytest.mark.parametrize("recon", [12, 18])
def test_range(scale, recon):
    """Scales on both sides of the fixed-point range."""
    U = li.gauge(DIMS, 0.5, 1401)
    psi = li.gaussian_spinor(DIMS, 2401)
    got = _apply(U, psi * scale, recon) / scale
    want = oracle.dslash(psi * parity_mask(DIMS, 0), U, DIMS, out_parity=1)
    assert rel_err(got, want) <= TOL_REL


@pytest.mark.parametrize("recon", [12, 18])
def test_links_outside(recon):
    """A field with one link that is not SU(3) keeps FP64 links; both forms agree with the oracle and, on the
    sites away from that link, with each other."""
    U = li.gauge(DIMS, 0.5, 1402)
    psi = li.gaussian_spinor(DIMS, 2402) * parity_mask(DIMS, 0)
    V = U.copy()
    V[37, 2] *= 1.5
    if recon == 12:  # the stored rows alone say the link
        V[37, 2, 2] = np.cross(V[37, 2, 0], V[37, 2, 1]).conj()
    a, b = _apply(U, psi, recon), _apply(V, psi, recon)
    assert rel_err(a, oracle.dslash(psi, U, DIMS, out_parity=1)) <= TOL_REL
    assert rel_err(b, oracle.dslash(psi, V, DIMS, out_parity=1)) <= TOL_REL
    same = np.abs(oracle.dslash(psi, U - V, DIMS, out_parity=1)).max(axis=(1, 2)) == 0
    assert same.sum() > 900 and rel_err(a[same], b[same]) <= TOL_REL


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_not_finite(bad):
    """Infinities and NaN come out where the FP64 path has them, and nowhere else."""
    import torch
    wdp = _wd()
    U = li.gauge(DIMS, 0.5, 1403)
    psi = to_internal_basis(li.gaussian_spinor(DIMS, 2403))[parity_sites(DIMS, 0)].reshape(-1, 12)
    psi[17, 4] += bad
    psi[400, 9] += 1j * bad
    vh, st = len(psi), (len(psi) + 31) // 32 * 32
    raw = np.zeros((12, st, 2))
    raw[:, :vh, 0], raw[:, :vh, 1] = psi.real.T, psi.imag.T
    out = []
    for scale in (1.0, 1.5):  # 1.5: links above the fixed-point bound, so the FP64 path
        wd = wdp.WilsonDirac(DIMS)
        wd.load_gauge(U * scale, recon=18)
        f = torch.from_numpy(raw).cuda().view(torch.uint8).reshape(-1)
        o = wd.new_field(wdp.F64)
        wd.dslash(o, f, 1, False, wdp.F64)
        out.append(o.cpu().numpy()[: 192 * st].view(np.float64).reshape(12, st, 2)[:, :vh] / scale)
        wd.close()
    for test in (np.isnan, np.isposinf, np.isneginf):
        assert (test(out[0]) == test(out[1])).all()
    fine = np.isfinite(out[1])
    assert rel_err(out[0][fine], out[1][fine]) <= TOL_REL


@pytest.mark.parametrize("exp2", [-100, 100])
@pytest.mark.parametrize("point", [False, True])
def test_solver_products_keep_every_digit_under_scaling(exp2, point):
    """The FP64 BiCGstab takes the norm of r and its product with r_tilde from integers
    in the unit of each site's largest component; sites without an exponent (zero) and
    outside the range are told apart.  Scaled by a power of two every digit stays."""
    wdp = _wd()
    U = li.gauge(DIMS, 0.4, 1020)
    b = li.point_source(DIMS, (1, 2, 3, 4), 1, 2) if point else li.gaussian_spinor(DIMS, 1021)
    wd = wdp.WilsonDirac(DIMS)
    wd.load_gauge(U)
    xs, iters = [], []
    for k in (0, exp2):
        x = np.zeros_like(b)
        info = wd.solve(x, b * 2.0 ** k, 0.12, tol=1e-10, solver=wdp.BICGSTAB, inner_precision=wdp.F64)
        xs.append(x * 2.0 ** -k)
        iters.append(info.iters)
        rel = oracle.true_residual(xs[-1], b, U, DIMS, 0.12)
        assert info.status == 0 and rel <= 1e-10, (k, info, rel)
    assert iters[0] == iters[1] and np.array_equal(xs[0], xs[1])
    wd.close()


def test_solver_products_of_uneven_sites():
    """Sites 2^-500 of the rest are outside the integers' range and take the FP64
    products; the solve is that of the source without them to its rounding."""
    wdp = _wd()
    U = li.gauge(DIMS, 0.4, 1022)
    b = li.gaussian_spinor(DIMS, 1023)
    b[::3] *= 2.0 ** -500
    wd = wdp.WilsonDirac(DIMS)
    wd.load_gauge(U)
    x = np.zeros_like(b)
    info = wd.solve(x, b, 0.12, tol=1e-10, solver=wdp.BICGSTAB, inner_precision=wdp.F64)
    rel = oracle.true_residual(x, b, U, DIMS, 0.12)
    assert info.status == 0 and rel <= 1e-10, (info, rel)
    wd.close()


@pytest.mark.parametrize("prec", [1, 2, 3, 4])
@pytest.mark.parametrize("angle", [0.0, 1e-12, 3e-10, 1e-5])
def test_derived_links_with_small_numbers(prec, angle):
    """The FP32 and 16-bit links are derived from the limbs of the fixed-point ones: zeros,
    numbers below 2^-28 (one limb) and ordinary ones, of both signs."""
    from tests.wd_testutil import TOL
    wdp = _wd()
    U = np.zeros((int(np.prod(DIMS)), 4, 3, 3), dtype=np.complex128)
    s = angle * np.where(np.arange(U.shape[0]) % 2, 1.0, -1.0)[:, None]
    for a, f in ((0, 1.0), (1, -2.0), (2, 1.0)):
        U[:, :, a, a] = np.exp(1j * f * s)
    psi = li.gaussian_spinor(DIMS, 1024)
    wd = wdp.WilsonDirac(DIMS)
    wd.load_gauge(U)
    f, o = wd.upload(psi, prec, parity=0), wd.new_field(prec)
    wd.dslash(o, f, 1, False, prec)
    want = oracle.dslash(psi * parity_mask(DIMS, 0), U, DIMS, dagger=False, out_parity=1, tbc_anti=False)
    assert rel_err(wd.download(o, prec, parity=1), want) <= TOL[prec]
    wd.close()
