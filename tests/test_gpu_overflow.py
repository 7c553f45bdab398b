"""FP64 runs whose |u|^2 overflows: every FP64 step kernel stops with the
oracle's outcome at the oracle's step.  A body force of 1e156 takes the fluid
from rest to 2e155 in one step: the state is finite, its square is not, so the
change of |u| is undefined and the run has diverged; a change taken as 0
against an infinite |u| would read as converged."""
import numpy as np
import pytest

from paper_2202_13449_gb300 import capi, inputs
from test_gpu3d import d3, make_pair as make_pair3  # noqa: F401
from test_gpu_curv import bent, cv, solver as solver_c  # noqa: F401
from test_gpu_parity import make_pair

pytestmark = pytest.mark.gpu

D, A = capi.WALL_DIRICHLET, capi.WALL_ADIABATIC
BIG, TOL, CAP = 1e156, 1e-3, 10


def check(got, ref):
    rc, steps, (ru, _) = got
    _, ref_steps, (ref_ru, _), ref_rc = ref
    assert ref_rc == capi.ERR_DIVERGED and rc == ref_rc and steps == ref_steps
    assert np.isnan(ref_ru) and np.isnan(ru)


@pytest.mark.parametrize("kernel,rows,scheme", [(1, 2, 0), (1, 4, 0), (1, 8, 0), (1, 16, 0), (0, 16, 0),
                                                (2, 2, 0), (2, 4, 0), (1, 16, 1)])
def test_rectilinear(orc, kernel, rows, scheme):
    xf, yf = inputs.uniform_faces(20), inputs.uniform_faces(10)
    p, s = make_pair(orc, xf, yf, 0.04, 0.05, 1e-3, 0.2, 1.0, (D, D, A, A), (1, 0, 0, 0), (0,) * 4,
                     capi.FP64, fx=BIG)
    p.scheme = scheme
    s.set_scheme(scheme)
    s.set_schedule(kernel, rows)
    st = inputs.conduction_state(xf, yf)
    s.set_state(*st)
    check(s.run_to_steady(TOL, CAP), orc.run_to_steady(p, st, TOL, CAP))
    s.close()


@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("scheme", [0, 1])
def test_3d(d3, tile, scheme):  # noqa: F811
    n = (9, 5, 4)
    faces = [inputs.uniform_faces(m) for m in n]
    p, s = make_pair3(d3, faces, (D, D, A, A, A, A), (0, 1, 0, 0, 0, 0), 2, 1.0, capi.FP64,
                      force=(0.0, BIG, 0.0))
    p.bc_u = ((0.0,) * 3,) * 6
    for side in range(6):
        s.set_bc(side, p.bc_kind[side], p.bc_T[side], (0.0,) * 3)
    p.scheme = scheme
    s.set_scheme(scheme)
    s.set_schedule(tile, 0)
    one = np.ones(n[::-1])
    st = [one, 0.0 * one, 0.0 * one, 0.0 * one, 0.5 * one]
    s.set_state(*st)
    check(s.run_to_steady(TOL, CAP), d3.run_to_steady(p, st, TOL, CAP))
    s.close()


@pytest.mark.parametrize("rows", [8, 16])
def test_curvilinear(cv, rows):  # noqa: F811
    X, Y = bent(11, 6, 5)
    p = cv.ProblemC(X=X, Y=Y, nu=0.03, chi=0.04, beta_g=2e-3, dt=0.2, kappa=0.9, gdir=(0.0, 1.0),
                    force=(BIG, 0.0), bc_kind=(D, D, A, A), bc_T=(1.0, 0.0, 0.0, 0.0))
    s = solver_c(p, False, capi.FP64, rows)
    one = np.ones(p.shape)
    st = [one, 0.0 * one, 0.0 * one, 0.5 * one]
    s.set_state(*st)
    check(s.run_to_steady(TOL, CAP), cv.run_to_steady(p, st, TOL, CAP))
    s.close()
