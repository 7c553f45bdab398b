"""The FP32 marching kernel (two columns a lane, strips of 60 columns) at the
edges of its strips and chunks, against the FP64 oracle.

Columns per line: 1 to 3 (a ghost of a ghost, no second column), around one
strip (58 to 63: the last pair whole, split and alone, ghosts in either
column of a lane) and around two (119 to 122); chunks of one row, of three
and longer than the mesh, whose prologues meet both walls.  Tolerance: the
FP32 bound of the parity tests, 1e-5 of the field's scale (a few units of
FP32 rounding, 6e-8, times the ~1e2 operations of a step).
"""
import numpy as np
import pytest

from paper_2202_13449_gb300 import capi, inputs

pytestmark = pytest.mark.gpu

D, A, P = capi.WALL_DIRICHLET, capi.WALL_ADIABATIC, capi.PERIODIC
WALLS = ((D, D, A, D), (1.0, 0.0, 0.0, 0.4), (0.01, 0.0, 0.0, 0.02))
PERIODIC_X = ((P, P, D, A), (0.0, 0.0, 1.0, 0.0), (0.0, 0.0, 0.01, 0.0))
PERIODIC_Y = ((A, D, P, P), (0.0, 0.3, 0.0, 0.0), (0.0, 0.01, 0.0, 0.0))


@pytest.mark.parametrize("sides", [WALLS, PERIODIC_X, PERIODIC_Y], ids=["walls", "per_x", "per_y"])
@pytest.mark.parametrize("nx,ny,rows", [(1, 4, 3), (2, 1, 1), (3, 5, 1), (58, 2, 3), (59, 7, 3),
                                        (60, 6, 3), (61, 9, 64), (62, 5, 1), (63, 8, 3),
                                        (119, 4, 3), (121, 11, 5), (122, 3, 64)])
def test_strip_and_chunk_edges(orc, nx, ny, rows, sides):
    kinds, bcT, bcU = sides
    xf, yf = inputs.random_faces(nx, 3 + nx), inputs.random_faces(ny, 5 + ny)
    p = orc.Problem(xf=xf, yf=yf, nu=0.04, chi=0.05, beta_g=1e-3, dt=0.2, kappa=0.9, fx=1e-4,
                    fy=-2e-4, bc_kind=kinds, bc_T=bcT, bc_u=bcU)
    s = capi.Solver(xf, yf, capi.FP32)
    s.set_params_ref(1e3, 0.71, 0.1, 0.2, 1.0, 1.0, 0.5)
    s.set_physics(0.04, 0.05, 1e-3)
    s.set_lattice(0.9)
    s.set_body_force(1e-4, -2e-4)
    for side in range(4):
        s.set_bc(side, kinds[side], bcT[side], bcU[side])
    s.set_schedule(0, rows)
    st = inputs.perturbed_state(nx, ny, seed=nx + 7 * ny)
    ref, (ru, rT), rc = orc.step(p, st, 3)
    assert rc == 0
    s.set_state(*st)
    s.step(3)
    got = s.get_state()
    (gu, gT), steps = s.residual()
    s.close()
    assert steps == 3
    d = np.max(np.abs(got[0] - ref[0])) / max(np.max(np.abs(ref[0] - 1.0)), 0.01)
    assert d < 1e-5
    for q, floor in ((1, 1e-2), (2, 1e-2), (3, 1.0)):
        assert np.max(np.abs(got[q] - ref[q])) / max(np.max(np.abs(ref[q])), floor) < 1e-5
    assert gu == pytest.approx(ru, rel=1e-3) and gT == pytest.approx(rT, rel=1e-3)
