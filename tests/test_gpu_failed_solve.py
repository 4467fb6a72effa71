"""Single-system solves that fail on the device: the solver graph ends and returns
the status and the counts of the host-driven loop, which runs first in every test."""
import numpy as np
import pytest

import lattice_inputs as li

pytestmark = pytest.mark.gpu

DIMS = (4, 6, 8, 10)
KAPPA = 0.12
BREAKDOWN, NUMERIC = 5, 6


def _solver(U):
    import paper_0911_3191_gb300 as m
    wd = m.WilsonDirac(DIMS)
    wd.load_gauge(U)
    return wd


def _both_loops(wd, b, solver, prec):
    out = []
    for graph in (False, True):
        r = wd.solve(np.zeros_like(b), b, KAPPA, tol=1e-10, solver=solver, inner_precision=prec, use_graph=graph,
                     max_iter=200, check=False)
        out.append((r.status, r.iters, r.reliable_updates, r.kernel_launches))
    assert out[0] == out[1], out
    return out[0]


def _launches(iterations, updates, solver, prec):
    """Kernels of a solve without a guess: set-up 10, 7 an iteration (CG 5), 3 or 4 a reliable update (CG 5), 2 at
    the end."""
    return 12 + iterations * (7, 5)[solver] + updates * (5 if solver else 3 if prec == 0 else 4)


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2, 3, 4])
def test_every_iteration_is_ended(solver, prec):
    """The finaliser that ends an iteration counts it, so one iteration short of the iterations' own count would be
    one that left the loop's condition alone."""
    wd = _solver(li.gauge(DIMS, 0.4, 1500))
    status, iters, updates, launches = _both_loops(wd, li.gaussian_spinor(DIMS, 2500), solver, prec)
    assert status == 0 and launches == _launches(iters - updates, updates, solver, prec)
    wd.close()


# site products are FP32 numbers under an FP32 or 16-bit inner precision: 1e-30 squared is 0 in them, 1e25 infinite
@pytest.mark.parametrize("scale,want", [(1e-30, BREAKDOWN), (1e25, NUMERIC)])
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [1, 2, 4])
def test_products_outside_fp32(scale, want, solver, prec):
    wd = _solver(li.gauge(DIMS, 0.4, 1501))
    status, iters, updates, launches = _both_loops(wd, scale * li.gaussian_spinor(DIMS, 2501), solver, prec)
    assert (status, iters, updates) == (want, 0, 0)
    assert launches == _launches(1, 0, solver, prec)  # the one that failed
    wd.close()


@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("where", ["source", "link"])
def test_infinity(solver, prec, where):
    U, b = li.gauge(DIMS, 0.4, 1502), li.gaussian_spinor(DIMS, 2502)
    if where == "source":
        b[33, 1, 2] = np.inf
    else:
        U[33, 1, 0, 2] = np.inf
    wd = _solver(U)
    assert _both_loops(wd, b, solver, prec)[0] == NUMERIC
    wd.close()
