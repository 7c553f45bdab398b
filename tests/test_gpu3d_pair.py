"""The FP32 3D step in pairs of columns, at the sizes where its split can go
wrong: last columns without a partner, tiles one column or row past their
width, one-cell lines, chunks of one plane, every tile shape and face stage,
against the 3D FP64 oracle.  Tolerance 1e-5 of each field's scale over three
steps, and 1e-6 on rho, as for every FP32 step: a step rounds increments of at
most the scale to 2^-24 and the state to 2^-30.
"""
import pytest

from paper_2202_13449_gb300 import capi, inputs
from test_gpu3d import A, D, P, compare, d3, make_pair  # noqa: F401

pytestmark = pytest.mark.gpu

WALLS = (D, A, A, D, A, D)
SIZES = [(1, 9, 5), (2, 8, 1), (3, 1, 4), (15, 4, 3), (16, 5, 2), (17, 9, 6), (31, 8, 2),
         (32, 17, 3), (33, 4, 4), (34, 9, 3), (65, 2, 3)]


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kinds", [WALLS, (P, P, A, D, D, A), (D, A, P, P, P, P), (P,) * 6])
def test_pair_steps(d3, n, kinds):  # noqa: F811
    faces = [inputs.random_faces(m, 7 + a) for a, m in enumerate(n)]
    st = inputs.perturbed_state3(*n, seed=sum(n))
    for scheme in (0, 1):
        p, s = make_pair(d3, faces, kinds, (0.9, 0, 0, 0.6, 0, 0.2), sum(n) % 3, 0.9, capi.FP32)
        p.scheme = scheme
        s.set_scheme(scheme)
        ref, _, rc = d3.step(p, st, 3)
        assert rc == 0
        for tile, kchunk in ((0, 1), (1, 0), (2, 2)):
            s.set_schedule(tile, kchunk)
            s.set_state(*st)
            s.step(3)
            compare(s.get_state(), ref, 1e-5, capi.FP32)
        s.close()
