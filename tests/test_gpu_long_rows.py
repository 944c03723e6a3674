"""Row lengths above the compiled ones (images wider than 2050 pixels) against the
oracle: schedules that use every radix in every stage it can take, a length
without a schedule (generic passes), odd widths, and heights on both sides of the
carry sweep's variants (32 and 160 bands of 4 rows)."""
import numpy as np
import pytest
import torch

import fp32_reference
import oracle.gfc_oracle as O
from paper_1902_00176_gb300 import gfc

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda:0")
REL_F32, MAXABS = 1e-5, 1e-4
F32, F16, BF16 = torch.float32, torch.float16, torch.bfloat16
UNIT = {F16: 2.0 ** -11, BF16: 2.0 ** -8}

CASES = [(2, 5, 2051, 2100, F32), (1, 126, 2152, 2160, F32), (1, 127, 2441, 2450, F32), (1, 640, 2243, 2268, F32),
         (1, 641, 2421, 2430, F32), (3, 9, 2490, 2500, F32), (1, 33, 2736, 2744, F32), (1, 20, 2908, 2916, BF16),
         (2, 21, 3064, 3072, F32), (1, 64, 3191, 3200, F16), (1, 65, 3401 - 8, 3402, F32), (1, 12, 3420, 3430, F32),
         (2, 2, 3492, 3500, F32), (1, 50, 3750 - 8, 3750, F32), (1, 700, 3840, 3888, F32), (1, 3, 3912, 3920, F32),
         (1, 17, 4040, 4050, BF16), (1, 31, 4088, 4096, F32)]


@pytest.fixture(autouse=True)
def _lib(gfc_lib):
    yield


def _rel(got, ref):
    return float(np.linalg.norm(got - ref) / max(np.linalg.norm(ref), 1e-300))


def _np(t):
    return t.double().cpu().numpy()


def _assert_near(got, ref, dt, rel=REL_F32):
    """FP32: relative L2. 16 bits: every element within the rounding of its storage
    and 1e-4 of the largest for the FP32 arithmetic."""
    if dt == F32:
        assert _rel(got, ref) <= rel
    else:
        assert np.all(np.abs(got - ref) <= UNIT[dt] * np.abs(ref) + 2.0 ** -25 + MAXABS * np.abs(ref).max())


@pytest.mark.parametrize("B,H,W,N,dt", CASES)
def test_long_rows_match_oracle(B, H, W, N, dt, monkeypatch):
    rng = np.random.default_rng(9500 + W)
    img = np.add.outer(np.sin(np.arange(H) * 0.05), np.cos(np.arange(W) * 0.04))
    gx, gy = np.zeros((B, 1, H, W)), np.zeros((B, 1, H, W))
    gx[..., :-1] = np.diff(img, axis=1)
    gy[..., :-1, :] = np.diff(img, axis=0)
    gx += rng.uniform(-0.05, 0.05, (B, 1, 1, 1))
    gy += rng.uniform(-0.05, 0.05, (B, 1, 1, 1))
    lap = rng.standard_normal((B, 1, H, W))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(DEV).to(dt)  # noqa: E731
    tx, ty, tl = dev(gx), dev(gy), dev(lap)
    p = gfc.Plan(H, W, 1, B, dtype=dt, device=DEV)
    assert p.N == N
    monkeypatch.setenv("GFC_FORCE_GENERIC", "1")
    gen = gfc.Plan(H, W, 1, B, dtype=dt, device=DEV)
    # the adjoint of a long-row plan runs the generic passes: their bits
    for got, want in zip(p.backward(tl), gen.backward(tl)):
        assert torch.equal(got, want)
    to, tu = p.solve_from_gradient(tx, ty), p.solve_from_laplacian(tl)
    if H < 16:  # thin strips keep the generic passes
        assert torch.equal(to, gen.solve_from_gradient(tx, ty)) and torch.equal(tu, gen.solve_from_laplacian(tl))
        return
    out, ul = _np(to), _np(tu)
    b = B - 1
    _assert_near(out[b, 0], O.solve_from_gradient(_np(tx)[b, 0], _np(ty)[b, 0], p.M, p.N, p.pad), dt)
    g = _np(tl)[b, 0]
    rl = O.solve_from_laplacian(g, p.M, p.N, p.pad)
    ql = REL_F32
    if dt == F32:
        fl = fp32_reference.torch_fp32_laplacian_solve(g, p.M, p.N, p.pad, DEV)
        ql = max(REL_F32, 3.0 * _rel(fl, rl))
    _assert_near(ul[b, 0], rl, dt, ql)
    gen.close()
    p.close()


def test_edits_and_correction_on_long_rows():
    """Edited and corrected solves of a long-row plan: the two-step flow's bits."""
    H, W = 40, 2100
    rng = np.random.default_rng(9600)
    t = lambda: torch.from_numpy(rng.standard_normal((1, 2, H, W)).astype(np.float32)).to(DEV) * 0.05  # noqa: E731
    gx, gy, img = t(), t(), t()
    p = gfc.Plan(H, W, 2, 1, device=DEV)
    m, s = p.field_stats(img)
    one = p.solve_corrected(gx, gy, m, s, edit="threshold", frac=0.2)
    two = p.solve_edited(gx, gy, "threshold", frac=0.2)
    p.color_correct(two, m, s)
    assert torch.equal(one, two)
    p.close()


def _call(p, mode, a, b):
    return p.solve_from_gradient(a, b) if mode == "gradient" else p.solve_from_laplacian(a)


@pytest.mark.parametrize("dt", [F32, BF16])
def test_widths_and_modes_interleaved(dt):
    """Plans kept side by side: a call of one width and input form does not change what
    another may launch, whichever came first, and its bits stay the same."""
    rng = np.random.default_rng(9650)
    t = lambda W: torch.from_numpy(rng.standard_normal((1, 1, 30, W)).astype(np.float32)).to(DEV).to(dt)  # noqa: E731
    wide, narrow = gfc.Plan(30, 4088, dtype=dt, device=DEV), gfc.Plan(30, 2092, dtype=dt, device=DEV)
    ins = {p: (t(p.W), t(p.W)) for p in (wide, narrow)}
    order = [(wide, "gradient"), (narrow, "laplacian"), (wide, "gradient"), (wide, "laplacian"), (narrow, "gradient"),
             (wide, "laplacian"), (wide, "gradient")]
    first = {}
    for p, mode in order:
        out = _call(p, mode, *ins[p])
        torch.cuda.synchronize()
        assert torch.equal(out, first.setdefault((p, mode), out))
    wide.close()
    narrow.close()
