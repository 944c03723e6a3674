"""Input and output rows of any length staged by bulk copy: rows that are not
whole 16-byte units start an item at any remainder, and the input's and the
output's last elements lie past the last whole unit.

Widths cover every remainder of a 16-byte unit, rows as wide as the staging
takes (W + 8 = N) and the narrowest of a row length, several fields and channels
(so that fields start at remainders too), one row pair, and both plans that end
and plans that do not end on a whole unit.
"""
import numpy as np
import pytest
import torch

import fp32_reference
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
REL_F32, REL_16 = 1e-5, 2e-3
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16

SHAPES = [(2, 3, 61, 333, F32), (1, 3, 40, 553, F32), (3, 1, 33, 554, F32), (1, 1, 2, 137, F32), (2, 2, 57, 499, F32),
          (1, 2, 90, 1111, F32), (1, 1, 19, 1112, F32), (1, 3, 261, 255, BF16), (2, 1, 262, 257, F16),
          (1, 2, 802, 1241, F32), (1, 1, 801, 1195, F16), (1, 1, 64, 98, F32), (3, 1, 64, 99, BF16)]


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


def _rel(got, ref):
    return float(np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300))


def _np(t):
    return t.double().cpu().numpy()


def _guarded(like):
    """A tensor of the shape of `like` between guard elements: (view, check)."""
    n = like.numel()
    buf = torch.full((n + 64,), 7.0, dtype=like.dtype, device=DEV)

    def check():
        assert bool((buf[:32] == 7.0).all()) and bool((buf[32 + n:] == 7.0).all())

    return buf[32:32 + n].view(like.shape), check


@pytest.mark.parametrize("B,C,H,W,dt", SHAPES)
def test_staged_rows_match_separate_passes(B, C, H, W, dt, monkeypatch):
    """Gradient, thresholded and Laplacian solves: staged rows give the bits of the
    packed rows stored by a pass of their own, and nothing beside the output is written."""
    gx, gy = synth.perturbed_gradient_batch(B * C, H, W, seed=9100 + W)
    tx = torch.from_numpy(gx).to(DEV).to(dt).view(B, C, H, W)
    ty = torch.from_numpy(gy).to(DEV).to(dt).view(B, C, H, W)
    p = gfc.Plan(H, W, C, B, dtype=dt, device=DEV)
    calls = [lambda o: p.solve_from_gradient(tx, ty, out=o), lambda o: p.solve_from_laplacian(tx, out=o),
             lambda o: p.solve_edited(tx, ty, edit="threshold", frac=0.1, out=o)]
    for call in calls:
        o, check = _guarded(tx)
        call(o)
        check()
        with monkeypatch.context() as m:
            m.setenv("GFC_UNFUSED_DIV", "1")
            m.setenv("GFC_UNFUSED_SMALL", "1")
            o2, _ = _guarded(tx)
            call(o2)
        assert torch.equal(o, o2)
    ref = O.solve_from_gradient(_np(tx)[-1, -1], _np(ty)[-1, -1], p.M, p.N, p.pad)
    got = _np(p.solve_from_gradient(tx, ty))[-1, -1]
    assert _rel(got, ref) <= (REL_F32 if dt == F32 else REL_16)
    p.close()


@pytest.mark.parametrize("B,C,H,W,dt", SHAPES)
def test_staged_adjoint_matches_oracle(B, C, H, W, dt):
    """The adjoint on the same shapes, held to the bound of a plain FP32 adjoint."""
    gout = synth.upstream_gradient((B, C, H, W), seed=9200 + W)
    p = gfc.Plan(H, W, C, B, dtype=dt, device=DEV)
    tg = torch.from_numpy(gout).to(DEV).to(dt)
    (ox, cx), (oy, cy) = _guarded(tg), _guarded(tg)
    p.backward(tg, ox, oy)
    cx()
    cy()
    for b, c in ((0, 0), (B - 1, C - 1)):
        g = _np(tg)[b, c]
        rx, ry = O.backward(g, p.M, p.N, p.pad)
        bx = by = REL_16
        if dt == F32:
            fx, fy = fp32_reference.torch_fp32_adjoint(g, p.M, p.N, p.pad, DEV)
            bx, by = max(REL_F32, 3.0 * _rel(fx, rx)), max(REL_F32, 3.0 * _rel(fy, ry))
        assert _rel(_np(ox)[b, c], rx) <= bx and _rel(_np(oy)[b, c], ry) <= by
    p.close()
