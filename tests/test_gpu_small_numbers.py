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


# --------------------------------------------- FP64: spins and colours of very different size
def _fields(dims, parity, seed, spread):
    """Device field (12, sites of the parity) of numbers 2^-k, k up to `spread`, by site, spin and colour, in the
    basis and order of device fields, and the same as (T, Z, Y, X, 4, 3) with zeros on the other parity."""
    rng = np.random.default_rng(seed)
    full = rng.normal(size=(li.volume(dims), 4, 3)) + 1j * rng.normal(size=(li.volume(dims), 4, 3))
    full *= np.exp2(-spread * rng.random((li.volume(dims), 4, 3)))
    sites = parity_sites(dims, parity)
    out = np.zeros_like(full)
    out[sites] = full[sites]
    return full[sites].reshape(-1, 12).T, out.reshape(*dims[::-1], 4, 3)


def _feeds(U, psi, dims, dagger):
    """Sum of |u| |psi| over the terms of each output: a spatial hop adds to a spin itself and its partner, a
    temporal one twice the spins that its projector keeps."""
    a, u = np.abs(psi), np.abs(U).reshape(*dims[::-1], 4, 3, 3)
    out = np.zeros_like(a)
    for mu in range(4):
        for fwd in (True, False):
            if fwd:
                h = np.einsum("...ij,...sj->...si", u[..., mu, :, :], np.roll(a, -1, 3 - mu))
            else:
                h = np.roll(np.einsum("...ji,...sj->...si", u[..., mu, :, :], a), 1, 3 - mu)
            if mu == 3:
                keep = slice(2, 4) if fwd != dagger else slice(0, 2)
                out[..., keep, :] += 2 * h[..., keep, :]
            else:
                partner = [3, 2, 1, 0] if mu < 2 else [2, 3, 0, 1]
                out += h + h[..., partner, :]
    return out.reshape(-1, 12)


def _raw_dslash(U, dims, raw, dagger, recon):
    """(sites of parity 1, 12) complex: the stored numbers of D applied to a device field."""
    import paper_0911_3191_gb300 as m
    import torch
    vh, st = raw.shape[1], (raw.shape[1] + 31) // 32 * 32
    buf = np.zeros((12, st, 2))
    buf[:, :vh, 0], buf[:, :vh, 1] = raw.real, raw.imag
    wd = m.WilsonDirac(dims)
    wd.load_gauge(U, recon=recon)
    o = wd.new_field(m.F64)
    wd.dslash(o, torch.from_numpy(buf).cuda().view(torch.uint8).reshape(-1), 1, dagger, m.F64)
    out = o.cpu().numpy()[: 192 * st].view(np.float64).reshape(12, st, 2)[:, :vh]
    wd.close()
    return (out[..., 0] + 1j * out[..., 1]).T


# one thread per site and four warps per 32 sites
@pytest.mark.parametrize("dims", [(4, 6, 8, 10), (16, 14, 12, 18)])
@pytest.mark.parametrize("recon,dagger", [(18, False), (12, True)])
@pytest.mark.parametrize("spread", [0, 6, 25, 90, "spin", "colour"])
def test_fp64_by_component(dims, recon, dagger, spread):
    """Every spin and colour is right to the sum of the |u| |psi| that feed it, however small beside the others.
    A field with a link that the integer form does not take is computed in FP64 throughout: its result is the
    reference away from that link.
    18 reals: 25 units of 2^-56 of the common exponent at most in a real part, and what feeds a component is at least
    2^-6 of it, or the site is computed in FP64: 25 sqrt(2) 2^-50, and FP64's 2^-48.  12 reals: the third row, which
    both rebuild, is right to a few 2^-53 absolute, which is 64 times as much of a component fed by 2^-6."""
    U = li.gauge(dims, 0.7, 1600)
    raw, psi = _fields(dims, 0, 2601, spread if isinstance(spread, int) else 0)
    if isinstance(spread, str):  # one spin (colour) 1e-18 of the others, links that do not mix it with them
        small = (np.arange(12) // 3 != 1) if spread == "spin" else (np.arange(12) % 3 == 1)
        raw = raw * np.where(small, 1e-18, 1.0)[:, None]
        psi = (psi.reshape(-1, 12) * np.where(small, 1e-18, 1.0)).reshape(psi.shape)
        U = U * np.eye(3)
        U /= np.abs(U).sum(-1, keepdims=True)
    if recon == 12:
        U[:, :, 2] = np.cross(U[:, :, 0], U[:, :, 1]).conj()
    V = U.copy()
    V[37, 2] *= 1.5
    got, want = _raw_dslash(U, dims, raw, dagger, recon), _raw_dslash(V, dims, raw, dagger, recon)
    feeds, feeds2 = _feeds(U, psi, dims, dagger), _feeds(V, psi, dims, dagger)
    odd = parity_sites(dims, 1)
    away = (feeds == feeds2).all(axis=1)[odd]
    assert away.sum() >= len(odd) - 2
    bound = (2.0 ** -44.6 if recon == 18 else 2.0 ** -40) * feeds[odd]
    assert (np.abs(got - want) <= bound)[away].all(), np.nanmax(np.abs(got - want)[away] / feeds[odd][away])


# 8, 840 and 22680 sites of a parity: warps with 8 and 24 lanes at work
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 10, 14), (18, 14, 10, 18)])
@pytest.mark.parametrize("temporal", [False, True])
@pytest.mark.parametrize("recon,dagger,anti", [(18, False, True), (18, True, False), (12, False, False),
                                               (12, True, True)])
@pytest.mark.parametrize("share", [0.04, 1.0])
def test_weak_sites(dims, temporal, recon, dagger, anti, share):
    """Diagonal links, and a colour 1e-18 of the others around some sites (a few of a warp, which its lanes compute
    together) or everywhere (each thread its own), in each variant of the kernel: every colour is right to the sum of
    what feeds it."""
    import paper_0911_3191_gb300 as m
    rng = np.random.default_rng(61)
    vol, odd = li.volume(dims), parity_sites(dims, 1)
    phase = rng.uniform(-np.pi, np.pi, (vol, 4, 2))
    U = np.zeros((vol, 4, 3, 3), dtype=np.complex128)
    U[:, :, 0, 0], U[:, :, 1, 1] = np.exp(1j * phase[..., 0]), np.exp(1j * phase[..., 1])
    U[:, :, 2, 2] = np.exp(-1j * phase.sum(-1))

    def around(a, f):
        grid = a.reshape(*dims[::-1], *a.shape[1:])
        return f([np.roll(grid, s, axis) for axis in range(4) for s in (1, -1)]).reshape(a.shape)

    centre = np.zeros(vol, dtype=bool)
    centre[rng.choice(odd, max(1, int(share * len(odd))), replace=False)] = True
    psi = li.gaussian_spinor(dims, 2603) * parity_mask(dims, 0)
    psi[around(centre, lambda n: np.any(n, axis=0)), :, 1] *= 1e-18
    wd = m.WilsonDirac(dims, t_antiperiodic=anti)
    wd.load_gauge(U, recon=recon, temporal_gauge=temporal)
    f, o = wd.upload(psi, m.F64, parity=0), wd.new_field(m.F64)
    wd.dslash(o, f, 1, dagger, m.F64)
    got, want = wd.download(o, m.F64, parity=1), oracle.dslash(psi, U, dims, dagger=dagger, out_parity=1, tbc_anti=anti)
    wd.close()
    # an output takes at most twice the largest spin of its colour from each neighbour; the changes of basis, the
    # temporal gauge's phases and the oracle round it a few times more, far below 2^-44 of it
    feeds = 2 * around(np.abs(psi).max(axis=1), lambda n: np.sum(n, axis=0))[odd]
    assert (np.abs(got - want)[odd].max(axis=1) <= 2.0 ** -44 * feeds).all()


@pytest.mark.parametrize("dims", [(4, 6, 8, 10), (16, 14, 12, 18)])
@pytest.mark.parametrize("recon", [12, 18])
def test_negative_zeros(dims, recon):
    """-0.0 beside -0.0 gives zeros, and beside numbers what +0.0 gives, to a unit in the last place of the largest."""
    raw, _ = _fields(dims, 0, 2602, 0)
    U = li.gauge(dims, 0.7, 1601)
    assert (_raw_dslash(U, dims, np.full_like(raw, complex(-0.0, -0.0)), False, recon) == 0).all()
    zero = np.random.default_rng(51).random(raw.shape[1]) < 0.5
    plus, minus = raw.copy(), raw.copy()
    plus[:, zero], minus[:, zero] = 0.0, complex(-0.0, -0.0)
    a, b = _raw_dslash(U, dims, plus, False, recon), _raw_dslash(U, dims, minus, False, recon)
    assert np.abs(a - b).max() <= 2.0 ** -50 * np.abs(raw).max()


@pytest.mark.parametrize("exp2", [-264, -240])
def test_solver_coefficients_of_a_small_source(exp2):
    """|b|^2 about 2^-513 (2^-465): the square in the complex divisions is below 2^-1024, which is a number but its
    reciprocal is not."""
    import paper_0911_3191_gb300 as m
    U = li.gauge(DIMS, 0.4, 1700)
    b = li.gaussian_spinor(DIMS, 2700)
    assert -514 < np.log2(np.linalg.norm(b) ** 2) - 528 < -512
    wd = m.WilsonDirac(DIMS)
    wd.load_gauge(U)
    for graph in (False, True):
        x = np.zeros_like(b)
        r = wd.solve(x, b * 2.0 ** exp2, 0.12, tol=0.05, solver=0, inner_precision=0, use_graph=graph, max_iter=50,
                     check=False)
        assert r.status == 0 and oracle.true_residual(x * 2.0 ** -exp2, b, U, DIMS, 0.12) <= 0.05, r
    wd.close()
