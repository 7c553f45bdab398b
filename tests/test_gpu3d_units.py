"""3D steps of very many work units (more than 260 per SM on 152 SMs): a thin,
long mesh in chunks of one plane, against the 3D FP64 oracle, both precisions
and face stages.  Tolerances of one step as in test_gpu3d.py: 1e-12 in FP64,
1e-5 in FP32."""
import pytest

from paper_2202_13449_gb300 import capi, inputs
from test_gpu3d import A, D, compare, d3, make_pair  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [capi.FP64, capi.FP32])
def test_many_units(d3, precision):  # noqa: F811
    n = (2, 3, 39600)
    faces = [inputs.random_faces(m, 11 + a) for a, m in enumerate(n)]
    st = inputs.perturbed_state3(*n, seed=12)
    for scheme in (0, 1):
        p, s = make_pair(d3, faces, (D, A, A, D, A, D), (0.9, 0, 0, 0.6, 0, 0.2), 2, 0.9, precision)
        p.scheme = scheme
        s.set_scheme(scheme)
        s.set_schedule(1, 1)
        s.set_state(*st)
        s.step(1)
        ref, _, rc = d3.step(p, st, 1)
        assert rc == 0
        compare(s.get_state(), ref, 1e-12 if precision == capi.FP64 else 1e-5, precision)
        s.autotune(2)  # every tile in chunks of one plane
        s.close()
