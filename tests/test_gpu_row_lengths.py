"""Row lengths with register-resident passes in every storage type: the short ones
(images 24 to 128 pixels wide), the 16-bit rows of the longer ones, and the row
passes of a compiled size pair at another column length."""
import numpy as np
import pytest
import torch

import fp32_reference
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc, synth

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
REL_F32, MAXABS = 1e-5, 1e-4
UNIT = {torch.float16: 2.0 ** -11, torch.bfloat16: 2.0 ** -8}  # half a unit in the last place, relative
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16

SHORT = [32, 36, 40, 42, 48, 50, 54, 56, 60, 64, 70, 72, 80, 84, 90, 96, 98, 100, 108, 112, 120, 126, 128]
HEIGHTS = [2, 5, 24, 31, 64, 65, 130, 257]
CASES = [(2, 2, HEIGHTS[i % len(HEIGHTS)], n - 8 - (i % 2), dt) for i, n in enumerate(SHORT) for dt in (F32, BF16, F16)]
CASES += [(1, 2, H, n - 8 - (i % 3), dt) for i, (n, H) in enumerate(
    [(140, 90), (160, 33), (180, 64), (200, 5), (224, 48), (252, 40), (294, 61), (320, 96), (360, 30), (400, 52),
     (448, 44), (500, 75), (560, 39), (630, 60), (700, 28), (784, 36), (882, 20), (980, 50), (1080, 23), (1120, 31),
     (1200, 40), (1372, 18), (1400, 27), (1536, 30), (1750, 16), (1960, 22), (2058, 21)]) for dt in (BF16, F16)]
CASES += [(1, 2, 50, 100, F32), (1, 2, 100, 262, F32), (1, 1, 90, 1242, F32), (1, 1, 33, 1560, F32),
          (1, 2, 100, 261, BF16), (1, 1, 60, 1200, BF16), (1, 1, 33, 1559, F16)]


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


def _rel(got, ref):
    return float(np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300))


def _np(t):
    return t.double().cpu().numpy()


def _assert_near(got, ref, dt, rel=REL_F32):
    """FP32: relative L2. 16 bits: every element within the rounding of its storage
    (also below the normal range) and 1e-4 of the largest for the FP32 arithmetic."""
    if dt == F32:
        assert _rel(got, ref) <= rel
    else:
        assert np.all(np.abs(got - ref) <= UNIT[dt] * np.abs(ref) + 2.0 ** -25 + MAXABS * np.abs(ref).max())


@pytest.mark.parametrize("B,C,H,W,dt", CASES)
def test_row_length_matches_oracle(B, C, H, W, dt):
    """Solve, Laplacian solve and adjoint of the first and the last field against the
    oracle; white-noise inputs within the bound of a plain FP32 transform."""
    rng = np.random.default_rng(9300 + W)
    img = np.add.outer(np.sin(np.arange(H) * 0.05), np.cos(np.arange(W) * 0.04))
    gx, gy = np.zeros((B, C, H, W)), np.zeros((B, C, H, W))
    gx[..., :-1] = np.diff(img, axis=1)
    gy[..., :-1, :] = np.diff(img, axis=0)
    gx += rng.uniform(-0.05, 0.05, (B, C, 1, 1))
    gy += rng.uniform(-0.05, 0.05, (B, C, 1, 1))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV).to(dt)  # noqa: E731
    tx, ty, tg = dev(gx), dev(gy), dev(synth.upstream_gradient((B, C, H, W), seed=9400 + W))
    p = gfc.Plan(H, W, C, B, dtype=dt, device=DEV)
    out, lap = _np(p.solve_from_gradient(tx, ty)), _np(p.solve_from_laplacian(tg))
    bx, by = (_np(t) for t in p.backward(tg))
    for b, c in ((0, 0), (B - 1, C - 1)):
        ref = O.solve_from_gradient(_np(tx)[b, c], _np(ty)[b, c], p.M, p.N, p.pad)
        _assert_near(out[b, c], ref, dt)
        g = _np(tg)[b, c]
        rl = O.solve_from_laplacian(g, p.M, p.N, p.pad)
        rx, ry = O.backward(g, p.M, p.N, p.pad)
        tl = tbx = tby = REL_F32
        if dt == F32:
            fl = fp32_reference.torch_fp32_laplacian_solve(g, p.M, p.N, p.pad, DEV)
            fx, fy = fp32_reference.torch_fp32_adjoint(g, p.M, p.N, p.pad, DEV)
            tl, tbx, tby = (max(REL_F32, 3.0 * _rel(f, r)) for f, r in ((fl, rl), (fx, rx), (fy, ry)))
        _assert_near(lap[b, c], rl, dt, tl)
        _assert_near(bx[b, c], rx, dt, tbx)
        _assert_near(by[b, c], ry, dt, tby)
    p.close()
