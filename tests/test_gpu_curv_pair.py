"""The FP32 curvilinear step in pairs of cells, at the sizes where its split
can go wrong: last columns without a partner, tiles one column or row past
their size, one-cell lines, every side kind on every side, both tile heights,
against the curvilinear FP64 oracle.  Tolerance as for every FP32 curvilinear
step: 1e-5 of each field's scale over three steps, 1e-6 on rho.
"""
import numpy as np
import pytest

from paper_2202_13449_gb300 import capi, inputs
from test_gpu_curv import A, D, F, P, bent, compare, cv, solver  # noqa: F401
from test_oracle_curv import o_mesh  # noqa: E402

pytestmark = pytest.mark.gpu

BASE = dict(nu=0.03, chi=0.04, beta_g=2e-3, dt=0.05, kappa=0.9, force=(1e-4, -2e-4))
BCU = ((0.0, 0.01), (0.003, 0.0), (0.0, 0.02), (0.02, -0.005))


def check(cv, p, periodic, seed):
    nj, ni = p.shape
    st = list(inputs.perturbed_state(ni, nj, seed=seed))
    ref, _, rc = cv.step(p, st, 3)
    assert rc == 0
    for rows in (8, 16):
        s = solver(p, periodic, capi.FP32, rows)
        s.set_state(*st)
        s.step(3)
        compare(s.get_state(), ref, 1e-5, capi.FP32)
        s.close()


@pytest.mark.parametrize("n", [(1, 9), (2, 1), (3, 8), (31, 16), (32, 17), (33, 7), (34, 1), (63, 9),
                               (65, 25)])
@pytest.mark.parametrize("kinds", [(D, A, A, D), (F, D, D, F), (A, F, F, A)])
def test_walls(cv, n, kinds):  # noqa: F811
    X, Y = bent(*n, 17 + n[0])
    g = np.array([0.3, 0.95]) / np.hypot(0.3, 0.95)
    check(cv, cv.ProblemC(X=X, Y=Y, gdir=tuple(g), bc_kind=kinds, bc_T=(0.9, 0.1, 0.3, 0.6), bc_u=BCU,
                          inf=(1.0, 0.01, -0.02, 0.4), **BASE), False, sum(n))


@pytest.mark.parametrize("n", [(31, 8), (32, 9), (33, 15), (64, 3), (97, 17)])
@pytest.mark.parametrize("kinds", [(P, P, D, F), (P, P, A, D)])
def test_seam(cv, n, kinds):  # noqa: F811
    X, Y = o_mesh(*n, 1.0, 3.0)
    par = dict(BASE, nu=0.003, chi=0.004, dt=0.01)
    check(cv, cv.ProblemC(X=X, Y=Y, gdir=(0.0, 1.0), bc_kind=kinds, bc_T=(0, 0, 1.0, 0.2), bc_u=BCU,
                          inf=(1.0, 0.02, 0.0, 0.1), **par), True, sum(n))
