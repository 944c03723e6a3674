"""Ragged batches of small items: from four on they run together through the generic
per-field passes (three launches for all of them, counted here), beside the plans of
the larger items; below that each has a plan of its own."""
import ctypes

import numpy as np
import pytest
import torch

import fp32_reference
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
REL_F32, MAXABS = 1e-5, 1e-4
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16
UNIT = {F16: 2.0 ** -11, BF16: 2.0 ** -8}

SMALL = [(1, 24, 24), (3, 64, 64), (1, 65, 120), (2, 262, 50)]  # small in every type
# (items, type, launches of the generic part by one solve)
CASES = [
    (SMALL, F32, 3), (SMALL, BF16, 3),
    (SMALL[:3], F32, 0), (SMALL[:3], F16, 0),  # too few
    (SMALL + [(1, 263, 60)], F16, 3),
    (SMALL[:3] + [(1, 265, 50)], F32, 0),  # the last one's columns are too long in FP32
    (SMALL[:3] + [(1, 100, 121)], F32, 0), (SMALL[:3] + [(1, 100, 121)], F16, 3),
    (SMALL[:3] + [(1, 545, 551)], BF16, 0), (SMALL[:3] + [(1, 547, 548)], BF16, 3),  # 300 295 and 299 756 pixels
    (SMALL + [(1, 801, 700), (3, 400, 401)], F32, 3), (SMALL + [(1, 801, 700), (3, 400, 401)], BF16, 3),
]


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


def _rel(got, ref):
    return float(np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300))


def _np(t):
    return t.double().cpu().numpy()


def _assert_near(got, ref, dt, rel):
    """FP32: relative L2. 16 bits: every element within the rounding of its storage
    and 1e-4 of the largest for the FP32 arithmetic."""
    if dt == F32:
        assert _rel(got, ref) <= rel
    else:
        assert np.all(np.abs(got - ref) <= UNIT[dt] * np.abs(ref) + 2.0 ** -25 + MAXABS * np.abs(ref).max())


def _generic_launches(rp):
    pr = gfc.Profile()
    assert gfc.lib().gfc_plan_get_profile(rp._h, ctypes.byref(pr), 1) == 0
    return sum(pr.launches)


@pytest.mark.parametrize("items,dt,launches", CASES)
def test_small_items_run_together(items, dt, launches):
    pairs = [synth.ragged_item_gradients(it, item=i, seed=7) for i, it in enumerate(items)]
    ups = [synth.upstream_gradient(it, seed=9950 + i) for i, it in enumerate(items)]
    rp = gfc.RaggedPlan(items, dt, device=DEV)
    gx, gy, up = (rp.pack([torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)) for a in t])
                  for t in ([p[0] for p in pairs], [p[1] for p in pairs], ups))
    _generic_launches(rp)
    out = rp.solve_from_gradient(gx, gy)
    assert _generic_launches(rp) == launches
    lap = rp.solve_from_laplacian(up)
    bx, by = rp.backward(up)
    for (C, H, W), x, y, u, o, l, px, py in zip(items, *(rp.unpack(t) for t in (gx, gy, up, out, lap, bx, by))):
        M, N = gfc.padded_size(H, W)
        c = C - 1
        g = _np(u)[c]
        rl, (rx, ry) = O.solve_from_laplacian(g, M, N, 4), O.backward(g, M, N, 4)
        tl = tx = ty = REL_F32
        if dt == F32:  # white noise: within the bound of a plain FP32 transform
            fl = fp32_reference.torch_fp32_laplacian_solve(g, M, N, 4, DEV)
            fx, fy = fp32_reference.torch_fp32_adjoint(g, M, N, 4, DEV)
            tl, tx, ty = (max(REL_F32, 3.0 * _rel(f, r)) for f, r in ((fl, rl), (fx, rx), (fy, ry)))
        _assert_near(_np(o)[c], O.solve_from_gradient(_np(x)[c], _np(y)[c], M, N, 4), dt, REL_F32)
        _assert_near(_np(l)[c], rl, dt, tl)
        _assert_near(_np(px)[c], rx, dt, tx)
        _assert_near(_np(py)[c], ry, dt, ty)
    rp.close()
