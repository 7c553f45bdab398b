"""FP32 tile blocks of every width, at odd sizes, against the FP64 oracle.

A tile's block has four, two or one times the least warps when its SM gets one
tile, two or more: meshes of 17 tiles across (the last one odd and ragged) and
as many up as give about 1.5 and 2.6 tiles an SM, walled on every side and
periodic either way, at every tile height, for the kernel of one launch a step
and for the persistent one.  Then batches with more tiles than blocks on the
GPU, some cavities finishing early.  Tolerances of the parity tests: 1e-5 in
FP32 after three steps, 1e-12 in FP64 after one, ten times as much for the
batches' up to six steps, as in test_gpu_batch.py.
"""
import numpy as np
import pytest
import torch

from paper_2202_13449_gb300 import capi, inputs
from test_gpu_batch import add
from test_gpu_parity import TILE_HEIGHTS, TOL, make_pair, rel, rho_rel

pytestmark = pytest.mark.gpu

D, A, P = capi.WALL_DIRICHLET, capi.WALL_ADIABATIC, capi.PERIODIC
SIDES = {"walls": ((D, A, D, D), (0.9, 0.0, 0.2, 0.5), (0.01, 0.0, -0.01, 0.02)),
         "per_x": ((P, P, D, A), (0.0, 0.0, 1.0, 0.0), (0.0, 0.0, 0.01, 0.0)),
         "per_y": ((A, D, P, P), (0.0, 0.3, 0.0, 0.0), (0.0, 0.01, 0.0, 0.0))}


@pytest.mark.parametrize("per_sm", [1.5, 2.6])
@pytest.mark.parametrize("h,scheme", [(h, 0) for h in TILE_HEIGHTS] + [(16, 1)])
def test_block_widths(orc, h, scheme, per_sm):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nx, ty = 17 * 32 - 3, round(per_sm * sms / 17)
    ny = ty * h - (1 if h > 2 else 0)  # the persistent kernel takes no tile of one row
    assert (2 * sms < 17 * ty) == (per_sm > 2) and 17 * ty > sms
    xf, yf = inputs.random_faces(nx, h), inputs.random_faces(ny, 50 + h)
    st = inputs.perturbed_state(nx, ny, seed=nx + ny)
    for kinds, bcT, bcU in SIDES.values():
        p, s = make_pair(orc, xf, yf, 0.04, 0.05, 1e-3, 0.2, 0.9, kinds, bcT, bcU, capi.FP32,
                         fx=1e-4, fy=-2e-4)
        p.scheme = scheme
        s.set_scheme(scheme)
        ref, _, rc = orc.step(p, st, 3)
        assert rc == 0
        for kernel in (1,) if scheme else (1, 2):
            s.set_schedule(kernel, h)
            s.set_state(*st)
            try:
                s.step(3)
            except capi.RTLBFSError as e:  # more tiles than are resident at once
                assert kernel == 2 and e.rc == capi.ERR_ARG
                continue
            got = s.get_state()
            assert rho_rel(got[0], ref[0]) < TOL[capi.FP32]
            for q, floor in ((1, 1e-2), (2, 1e-2), (3, 1.0)):
                assert rel(got[q], ref[q], floor) < TOL[capi.FP32], (kernel, q)
        s.close()


@pytest.mark.parametrize("precision,h", [(capi.FP32, 16), (capi.FP32, 10), (capi.FP64, 16),
                                         (capi.FP64, 2)])
def test_batch_of_more_tiles_than_blocks(orc, precision, h):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    specs = [(61 + 7 * k, 93 + 11 * k, 0.8, 1e4, k) for k in range(20)]
    b = capi.Batch(precision, len(specs))
    b.set_schedule(1, h)
    runs = []
    for k, sp in enumerate(specs):
        st = inputs.perturbed_state(sp[0], sp[1], seed=k)
        slot, xf, yf, dt = add(b, orc, sp, st)
        n = 1 + k % 6
        b.arm(slot, 0.0, n)
        runs.append((sp, slot, xf, yf, dt, st, n))
    w = 16 if precision == capi.FP64 and h == 2 else 32
    tiles = sum(-(-sp[0] // w) * -(-sp[1] // h) for sp in specs)
    # blocks an SM at most: 227 KB over the box, gradients and faces of a tile
    cell = 16 if precision == capi.FP32 else 32
    least = cell * ((w + 4) * (h + 4) + 2 * (w + 2) * (h + 2) + 2 * w * h)
    assert tiles > sms * (227 * 1024 // least)
    b.step(6)
    _, steps, _ = b.poll()
    for sp, slot, xf, yf, dt, st, n in runs:
        nu, chi, bg = orc.params_from_ra(sp[3], 0.71, 0.1, float(sp[0]))
        ref, _, rc = orc.step(orc.Problem(xf=xf, yf=yf, nu=nu, chi=chi, beta_g=bg, dt=dt), st, n)
        assert rc == 0 and steps[slot] == n
        got = b.get_state(slot)
        for q, floor in ((1, 1e-2), (2, 1e-2), (3, 1.0)):
            assert rel(got[q], ref[q], floor) < 10 * TOL[precision], (sp, q)
    b.close()
