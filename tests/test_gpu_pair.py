"""Batched dslash with two 16-bit systems per thread, and the shapes that
wd_dslash_batch takes when no batched solve has tuned one."""
import pytest

import lattice_inputs as li
import oracle
from tests.wd_testutil import TOL, rel_err

pytestmark = pytest.mark.gpu


def fields(wd, m, dims, prec, nrhs, seed):
    fb = wd.field_bytes(prec)
    fin = wd.new_field(prec, nrhs)
    for r in range(nrhs):
        wd.field_import(fin[r * fb:(r + 1) * fb], li.gaussian_spinor(dims, seed + r), m.EVEN, prec)
    return fin, fb


@pytest.mark.parametrize("prec", [2, 3, 4])
@pytest.mark.parametrize("nrhs,grid", [(1, 4), (2, 1), (5, 16)])
@pytest.mark.parametrize("tfix", [False, True])
def test_pairs_equal_single_rows(tmp_path, monkeypatch, prec, nrhs, grid, tfix):
    """A pair of systems per thread does each system's arithmetic as one system
    per block row does: the same bytes from the dslash (an odd count leaves one
    without a partner; 768 sites, six blocks or loops over fewer).  The batched
    solve's systems converge at different iterations, so pairs break up."""
    import torch

    import paper_0911_3191_gb300 as m
    dims = (8, 6, 4, 8)
    U = li.gauge(dims, 0.5, 1014)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    srcs = [li.gaussian_spinor(dims, 5300 + r) for r in range(nrhs)]
    kappas = [0.10, 0.124, 0.115, 0.11, 0.12][:nrhs]
    outs = []
    for pack in (0, 1):
        cache = tmp_path / f"tune{pack}.txt"
        entry = f"{dims[0]}x{dims[1]}x{dims[2]}x{dims[3]} prec{prec} n{nrhs} sms{sms} links12 tfix{int(tfix)}"
        cache.write_text(f"{entry}|0 {grid} {pack}\n")
        monkeypatch.setenv("WD_TUNE_CACHE", str(cache))
        wd = m.WilsonDirac(dims, t_antiperiodic=True)
        wd.load_gauge(U, temporal_gauge=tfix)
        xs = [s * 0 for s in srcs]
        infos = wd.solve_batch(xs, srcs, kappas, tol=1e-10, inner_precision=prec)
        for x, b, k, info in zip(xs, srcs, kappas, infos):
            rel = oracle.true_residual(x, b, U, dims, k, tbc_anti=True)
            assert info.status == 0 and rel <= 1e-10, (k, info, rel)
        fin, _ = fields(wd, m, dims, prec, nrhs, 5400)
        for dagger in (False, True):
            fout = wd.new_field(prec, nrhs)
            fout.zero_()  # the padding too
            torch.cuda.synchronize()
            wd.dslash_batch(fout, fin, nrhs, m.ODD, dagger, prec)
            torch.cuda.synchronize()
            outs.append(fout.cpu())
        assert cache.read_text().count("\n") == 1  # the entry was taken
        wd.close()
    assert torch.equal(outs[0], outs[2]) and torch.equal(outs[1], outs[3])


@pytest.mark.parametrize("prec", [1, 2, 3, 4])
@pytest.mark.parametrize("nrhs", [1, 3, 4, 5])
def test_untuned_shapes(prec, nrhs):
    """Both sides of the lines between the shapes: with 152 SMs, 16^3x32 takes
    16-bit pairs from five systems and FP32 tiles of two from four."""
    import paper_0911_3191_gb300 as m
    dims = (16, 16, 16, 32)
    wd = m.WilsonDirac(dims)
    wd.load_gauge(li.gauge(dims, 0.5, 1015))
    fin, fb = fields(wd, m, dims, prec, nrhs, 5500)
    fout, single = wd.new_field(prec, nrhs), wd.new_field(prec)
    wd.dslash_batch(fout, fin, nrhs, m.ODD, False, prec)
    for r in range(nrhs):
        wd.dslash(single, fin[r * fb:(r + 1) * fb], m.ODD, False, prec)
        got, one = (wd.download(f, prec, parity=m.ODD) for f in (fout[r * fb:(r + 1) * fb], single))
        assert rel_err(got, one) <= TOL[prec] * (1 if prec <= 1 else 0.2), r
    wd.close()
